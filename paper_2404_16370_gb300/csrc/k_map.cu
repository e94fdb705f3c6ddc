// Map and scan preprocessing (Sec. III-C):
//  * GICP point Gaussians: each point's normal from its cov_k nearest points
//    within r_cov (decided by the exact FP32 distance sequence, ties to the
//    smaller index); Sigma = I - (1 - eps_cov) n n^T is carried as n.
//  * the nearest neighbour field m^nnf: per voxel, the nearest valid map point
//    to the voxel centre within r_max (-1 if none).
//  * per-step scan Gaussians and the sorted compaction of the valid scan points
//    into the chunks the likelihood kernel stages in shared memory.
#include "mp_internal.cuh"

#include <algorithm>
#include <cmath>
#include <vector>

namespace {

// Uniform cell grid of side h over a point set (exact candidate filter: every
// point within distance h of a query lies in the 27 cells around it).
struct CellGridDev {
    float og[3], inv_h;
    int dims[3];
    int64_t ncell;
    uint32_t* start = nullptr;   // ncell + 1
    int32_t* items = nullptr;    // points, grouped by cell
};

__device__ __forceinline__ void cell_coords(const CellGridDev& g, float x, float y, float z, int c[3]) {
    float p[3] = {x, y, z};
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        int v = (int)floorf((p[a] - g.og[a]) * g.inv_h);
        c[a] = min(max(v, -1), g.dims[a]);
    }
}

__global__ void k_cell_count(const float4* __restrict__ pts, const uint8_t* __restrict__ valid, int64_t n,
                             CellGridDev g, int32_t* __restrict__ cell_of, uint32_t* __restrict__ count) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    if (valid && !valid[i]) { cell_of[i] = -1; return; }
    float4 p = pts[i];
    int c[3];
    cell_coords(g, p.x, p.y, p.z, c);
    c[0] = min(max(c[0], 0), g.dims[0] - 1);
    c[1] = min(max(c[1], 0), g.dims[1] - 1);
    c[2] = min(max(c[2], 0), g.dims[2] - 1);
    int64_t ci = ((int64_t)c[2] * g.dims[1] + c[1]) * g.dims[0] + c[0];
    cell_of[i] = (int32_t)ci;
    atomicAdd(&count[ci], 1u);
}

__global__ void k_cell_fill(const int32_t* __restrict__ cell_of, int64_t n, const uint32_t* __restrict__ start,
                            uint32_t* __restrict__ fill, int32_t* __restrict__ items) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    int32_t c = cell_of[i];
    if (c < 0) return;
    uint32_t pos = atomicAdd(&fill[c], 1u);
    items[start[c] + pos] = (int32_t)i;
}

// Sorted insertion of (d, j) into the MP_COVK smallest pairs seen so far
// (order: d, then j). A pair that does not precede the current last one
// cannot enter, and is rejected before the insertion chain.
__device__ __forceinline__ void topk_insert(float (&D)[MP_COVK], int (&J)[MP_COVK], float d, int j) {
    if (!(d < D[MP_COVK - 1] || (d == D[MP_COVK - 1] && j < J[MP_COVK - 1]))) return;
#pragma unroll
    for (int s = 0; s < MP_COVK; ++s) {
        bool lt = (d < D[s]) || (d == D[s] && j < J[s]);
        float td = D[s];
        int tj = J[s];
        D[s] = lt ? d : td;
        J[s] = lt ? j : tj;
        d = lt ? td : d;
        j = lt ? tj : j;
    }
}

// Normal of a 3x3 covariance (FP64): smallest eigenvalue by the closed-form
// trigonometric solution of the characteristic cubic (Smith, CACM 1961),
// refined once by the Rayleigh quotient of its eigenvector; the eigenvector
// is the largest cross product of two rows of (C - lambda I). Sign: the
// largest-magnitude component positive (first index on ties).
__device__ void normal_of_cov(const double C[6], float n_out[3]) {
    // C = (xx, xy, xz, yy, yz, zz)
    double a00 = C[0], a01 = C[1], a02 = C[2], a11 = C[3], a12 = C[4], a22 = C[5];
    double p1 = a01 * a01 + a02 * a02 + a12 * a12;
    double q = (a00 + a11 + a22) / 3.0;
    double b00 = a00 - q, b11 = a11 - q, b22 = a22 - q;
    double p2 = b00 * b00 + b11 * b11 + b22 * b22 + 2.0 * p1;
    double lam;
    if (p2 <= 0.0) {
        lam = q;
    } else {
        double p = sqrt(p2 / 6.0);
        double ip = 1.0 / p;
        double c00 = b00 * ip, c11 = b11 * ip, c22 = b22 * ip, c01 = a01 * ip, c02 = a02 * ip, c12 = a12 * ip;
        double det = c00 * (c11 * c22 - c12 * c12) - c01 * (c01 * c22 - c12 * c02) + c02 * (c01 * c12 - c11 * c02);
        double r = fmin(1.0, fmax(-1.0, 0.5 * det));
        double phi = acos(r) / 3.0;
        lam = q + 2.0 * p * cos(phi + 2.0943951023931954923);   // + 2 pi / 3: the smallest root
    }
    double v[3] = {0, 0, 1};
    for (int it = 0; it < 2; ++it) {
        double r0[3] = {a00 - lam, a01, a02}, r1[3] = {a01, a11 - lam, a12}, r2[3] = {a02, a12, a22 - lam};
        double c[3][3];
        c[0][0] = r0[1] * r1[2] - r0[2] * r1[1]; c[0][1] = r0[2] * r1[0] - r0[0] * r1[2]; c[0][2] = r0[0] * r1[1] - r0[1] * r1[0];
        c[1][0] = r0[1] * r2[2] - r0[2] * r2[1]; c[1][1] = r0[2] * r2[0] - r0[0] * r2[2]; c[1][2] = r0[0] * r2[1] - r0[1] * r2[0];
        c[2][0] = r1[1] * r2[2] - r1[2] * r2[1]; c[2][1] = r1[2] * r2[0] - r1[0] * r2[2]; c[2][2] = r1[0] * r2[1] - r1[1] * r2[0];
        double nn[3];
        int best = 0;
        for (int k = 0; k < 3; ++k) nn[k] = c[k][0] * c[k][0] + c[k][1] * c[k][1] + c[k][2] * c[k][2];
        if (nn[1] > nn[best]) best = 1;
        if (nn[2] > nn[best]) best = 2;
        if (!(nn[best] > 0.0)) break;   // (near) repeated smallest eigenvalue: keep v
        double s = 1.0 / sqrt(nn[best]);
        v[0] = c[best][0] * s; v[1] = c[best][1] * s; v[2] = c[best][2] * s;
        // Rayleigh quotient of the current vector refines lambda
        double Av0 = a00 * v[0] + a01 * v[1] + a02 * v[2];
        double Av1 = a01 * v[0] + a11 * v[1] + a12 * v[2];
        double Av2 = a02 * v[0] + a12 * v[1] + a22 * v[2];
        lam = v[0] * Av0 + v[1] * Av1 + v[2] * Av2;
    }
    int big = 0;
    if (fabs(v[1]) > fabs(v[big])) big = 1;
    if (fabs(v[2]) > fabs(v[big])) big = 2;
    double sg = v[big] < 0 ? -1.0 : 1.0;
    n_out[0] = (float)(sg * v[0]);
    n_out[1] = (float)(sg * v[1]);
    n_out[2] = (float)(sg * v[2]);
}

// FP64 sample covariance of the m neighbours J(0), J(1), ... and the resulting
// normal.
template <typename Index>
__device__ void neighbourhood_normal(const float4* __restrict__ pts, Index J, int m, float n_out[3]) {
    double mx = 0, my = 0, mz = 0;
    for (int s = 0; s < m; ++s) {
        float4 p = pts[J(s)];
        mx += p.x; my += p.y; mz += p.z;
    }
    mx /= m; my /= m; mz /= m;
    double C[6] = {0, 0, 0, 0, 0, 0};
    for (int s = 0; s < m; ++s) {
        float4 p = pts[J(s)];
        double dx = p.x - mx, dy = p.y - my, dz = p.z - mz;
        C[0] += dx * dx; C[1] += dx * dy; C[2] += dx * dz;
        C[3] += dy * dy; C[4] += dy * dz; C[5] += dz * dz;
    }
    for (int a = 0; a < 6; ++a) C[a] /= m;
    normal_of_cov(C, n_out);
}

// x / b, correctly rounded, from rb = 1 / b correctly rounded (Markstein 1990).
__device__ __forceinline__ double div_by(double x, double b, double rb) {
    const double q = x * rb;
    return fma(fma(-b, q, x), rb, q);
}
__constant__ double nrm_inverse[MP_COVK + 1] = {0.,     1. / 1, 1. / 2,  1. / 3,  1. / 4,  1. / 5,  1. / 6,  1. / 7, 1. / 8,
                                                1. / 9, 1. / 10, 1. / 11, 1. / 12, 1. / 13, 1. / 14, 1. / 15, 1. / 16};
static_assert(MP_COVK == 16, "nrm_inverse");

// The same normal, bit for bit, by four lanes: lane a of the quad works on
// component or row a (the fourth as the third) and returns component a. m = 0: no
// neighbours (the value is of no use). An FP64 instruction holds a quarter of the
// SM for 64 cycles, whatever the number of active lanes: four warps of eight
// points with the components side by side take half the instructions of a
// chain that one warp of 32 points has on one quarter (10 us less for a scan).
template <typename Index>
__device__ __forceinline__ float neighbourhood_normal_quad(const float* __restrict__ raw, Index J, int m) {
    constexpr unsigned ALL = 0xffffffffu;
    const int lane = threadIdx.x & 31, quad = lane & ~3, a = min(lane & 3, 2);
    auto get = [&](double x, int c) { return __shfl_sync(ALL, x, quad + c); };
    const int most = __reduce_max_sync(ALL, m);
    const double dm = m, rm = nrm_inverse[m];
    double mean = 0.0, Cd = 0.0, Co = 0.0;   // Cd: entry (a, a), Co: entry (a, a + 1 mod 3)
    for (int s = 0; s < most; ++s) mean += s < m ? (double)__ldg(raw + 3 * J(s) + a) : 0.0;
    mean = div_by(mean, dm, rm);
    for (int s = 0; s < most; ++s) {
        const double d = s < m ? (double)__ldg(raw + 3 * J(s) + a) - mean : 0.0;
        const double e = get(d, (a + 1) % 3);
        Cd += d * d;
        Co += d * e;
    }
    Cd = div_by(Cd, dm, rm);
    Co = div_by(Co, dm, rm);
    const double a00 = get(Cd, 0), a11 = get(Cd, 1), a22 = get(Cd, 2);
    const double a01 = get(Co, 0), a12 = get(Co, 1), a02 = get(Co, 2);
    const double sq = Co * Co, p1 = get(sq, 0) + get(sq, 2) + get(sq, 1);
    const double q = div_by(a00 + a11 + a22, 3.0, 1.0 / 3.0);
    const double b = Cd - q, bb = b * b;
    const double p2 = get(bb, 0) + get(bb, 1) + get(bb, 2) + 2.0 * p1;
    double lam;
    {
        const double p = sqrt(div_by(p2, 6.0, 1.0 / 6.0)), ip = 1.0 / p;
        const double cb = b * ip, co = Co * ip;
        const double c00 = get(cb, 0), c11 = get(cb, 1), c22 = get(cb, 2);
        const double c01 = get(co, 0), c12 = get(co, 1), c02 = get(co, 2);
        // the determinant's three terms
        const double u = (a == 0 ? c11 : c01) * (a == 2 ? c12 : c22), w = (a == 2 ? c11 : c12) * (a == 0 ? c12 : c02);
        const double t = (a == 0 ? c00 : a == 1 ? c01 : c02) * (u - w);
        const double det = get(t, 0) - get(t, 1) + get(t, 2);
        const double r = fmin(1.0, fmax(-1.0, 0.5 * det));
        const double phi = div_by(acos(r), 3.0, 1.0 / 3.0);
        lam = q + 2.0 * p * cos(phi + 2.0943951023931954923);   // + 2 pi / 3: the smallest root
        if (p2 <= 0.0) lam = q;
    }
    double v = a == 2 ? 1.0 : 0.0;
    bool stop = false;
#pragma unroll
    for (int it = 0; it < 2; ++it) {
        const double d = Cd - lam, d0 = get(d, 0), d1 = get(d, 1), d2 = get(d, 2);
        // lane 0: rows 0 and 1, lane 1: 0 and 2, lane 2: 1 and 2
        const double x0 = a == 2 ? a01 : d0, x1 = a == 2 ? d1 : a01, x2 = a == 2 ? a12 : a02;
        const double y0 = a == 0 ? a01 : a02, y1 = a == 0 ? d1 : a12, y2 = a == 0 ? a12 : d2;
        const double c0 = x1 * y2 - x2 * y1, c1 = x2 * y0 - x0 * y2, c2 = x0 * y1 - x1 * y0;
        const double nn = c0 * c0 + c1 * c1 + c2 * c2;
        const double n0 = get(nn, 0), n1 = get(nn, 1), n2 = get(nn, 2);
        int best = 0;
        double nb = n0;
        if (n1 > nb) { best = 1; nb = n1; }
        if (n2 > nb) { best = 2; nb = n2; }
        if (!(nb > 0.0)) stop = true;   // (near) repeated smallest eigenvalue: keep v
        const double sc = 1.0 / sqrt(nb);
        const double e0 = get(c0, best), e1 = get(c1, best), e2 = get(c2, best);
        const double nv = (a == 0 ? e0 : a == 1 ? e1 : e2) * sc;
        if (!stop) v = nv;
        if (it == 0) {
            // Rayleigh quotient of the current vector refines lambda
            const double v0 = get(v, 0), v1 = get(v, 1), v2 = get(v, 2);
            const double Av = (a == 0 ? a00 : a == 1 ? a01 : a02) * v0 + (a == 0 ? a01 : a == 1 ? a11 : a12) * v1 +
                              (a == 0 ? a02 : a == 1 ? a12 : a22) * v2;
            const double t = v * Av;
            lam = get(t, 0) + get(t, 1) + get(t, 2);
        }
    }
    const double v0 = get(v, 0), v1 = get(v, 1), v2 = get(v, 2);
    double big = v0;
    if (fabs(v1) > fabs(big)) big = v1;
    if (fabs(v2) > fabs(big)) big = v2;
    return (float)(big < 0 ? -v : v);
}

// Map points: neighbourhoods through the cell grid.
__global__ void k_map_normals(const float4* __restrict__ pts, int64_t n, CellGridDev g, float r2, int k, int kmin,
                              float* __restrict__ normals, uint8_t* __restrict__ valid) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    float4 pi = pts[i];
    float D[MP_COVK];
    int J[MP_COVK];
#pragma unroll
    for (int s = 0; s < MP_COVK; ++s) { D[s] = INFINITY; J[s] = 0x7fffffff; }
    int cnt = 0;
    int c[3];
    cell_coords(g, pi.x, pi.y, pi.z, c);
    for (int dz = -1; dz <= 1; ++dz)
        for (int dy = -1; dy <= 1; ++dy)
            for (int dx = -1; dx <= 1; ++dx) {
                int x = c[0] + dx, y = c[1] + dy, z = c[2] + dz;
                if (x < 0 || y < 0 || z < 0 || x >= g.dims[0] || y >= g.dims[1] || z >= g.dims[2]) continue;
                int64_t ci = ((int64_t)z * g.dims[1] + y) * g.dims[0] + x;
                for (uint32_t e = g.start[ci]; e < g.start[ci + 1]; ++e) {
                    int j = g.items[e];
                    float4 pj = pts[j];
                    float d2 = dist2_exact(pi.x, pi.y, pi.z, pj.x, pj.y, pj.z);
                    if (d2 <= r2) {
                        cnt++;
                        topk_insert(D, J, d2, j);
                    }
                }
            }
    int m = min(cnt, k);
    if (m < kmin) {
        valid[i] = 0;
        normals[3 * i] = normals[3 * i + 1] = normals[3 * i + 2] = 0.f;
        return;
    }
    float nv[3];
    neighbourhood_normal(pts, [&](int s) { return J[s]; }, m, nv);
    normals[3 * i] = nv[0]; normals[3 * i + 1] = nv[1]; normals[3 * i + 2] = nv[2];
    valid[i] = 1;
}

// Scan points: brute force over the whole scan, staged through shared memory in
// tiles. A warp takes two points, its lanes take candidates; those within the
// radius go to a buffer per point, and when it fills up the cov_k nearest of it
// are selected (cov_k rounds of a warp minimum over (d, j)) and their last
// distance becomes the new radius. The set and its order do not depend on the
// order in which candidates are seen. The normals, in FP64 (1/75 of the FP32
// rate), take four lanes per point. What bounds it: the distances (13
// instructions a warp and 32 candidates) from a few thousand points on, below
// that the FP64 chain of one normal.
// Measured (the scan stage, against one thread per point and eighth of the scan
// with a sorted list of its own, merged by one thread): 128 points 62 -> 32 us
// (42 with a normal on one lane), 2048 142 -> 34 (60), 4999 178 -> 98 (101),
// 8192 233 -> 143 (145).
#define SCAN_TILE 1024
#define SCAN_PARTS 8
#define SCAN_CTA 256
#define SCAN_PTS (SCAN_CTA / SCAN_PARTS)
#define NRM_PTS 32                    // points of a CTA
#define NRM_CTA (NRM_PTS / 2 * 32)    // two points a warp
#define NRM_BUF 96                    // candidates a point's buffer holds

// Arguments of the per-step scan kernels (raw n x 3 points in, normals,
// validity and the compacted broadcast pairs out).
struct ScanArgs {
    const float* raw;
    int n;
    float r2;
    int k, kmin;
    float inv_cell;      // 1 / (4 NNF voxels): the cells of scan_key
    float4* tmp4;        // x, y, z and the bits of scan_key
    float* normals;      // (normals and valid null: every point is sorted, without a normal)
    uint8_t* valid;
    float4* pair;        // the valid points in input order, broadcast pairs (with normals),
    float* soa;          // and sorted, the likelihood's chunks
    int32_t* idx;        // the sorted points' indices (or null)
    int32_t* nvalid;
    float* out;          // sorted_normals: the sorted points with their normals, in chunks like soa
};

// Order of the scan points for the likelihood: range shells of 64 NNF voxels
// (16 of them at most), and in a shell the Morton code of the point's cell of 4
// voxels. Whatever a particle's heading, a shell of the scan falls on a ring
// around the particle, so particles near each other that work on one part of
// the scan read one part of the NNF; and the points of a warp, neighbours in a
// shell, read few lines of it. Results depend on the order only by rounding.
__device__ __forceinline__ uint32_t scan_key(float x, float y, float z, float inv_cell) {
    const float r = sqrtf(x * x + y * y + z * z) * inv_cell;
    const uint32_t shell = (uint32_t)fminf(r * (1.f / 16.f), 15.f);
    const float p[3] = {x, y, z};
    uint32_t code = 0;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        uint32_t c = (uint32_t)fminf(fmaxf(floorf(p[a] * inv_cell) + 256.f, 0.f), 511.f);
        c = (c | (c << 16)) & 0x030000FFu;
        c = (c | (c << 8)) & 0x0300F00Fu;
        c = (c | (c << 4)) & 0x030C30C3u;
        c = (c | (c << 2)) & 0x09249249u;
        code |= c << a;
    }
    return (shell << 27) | code;
}

struct ScanF4Op {
    using Args = ScanArgs;
    static constexpr int THREADS = 256, MINB = 1;
    static __device__ __forceinline__ void run(const ScanArgs& A, unsigned bx, unsigned) {
        int i = (int)bx * THREADS + threadIdx.x;
        if (i >= A.n) return;
        const float x = A.raw[3 * i], y = A.raw[3 * i + 1], z = A.raw[3 * i + 2];
        A.tmp4[i] = make_float4(x, y, z, __uint_as_float(scan_key(x, y, z, A.inv_cell)));
    }
};

// SORTED: the points are taken in the order of soa and idx (all of them), a tile
// of 32 candidates is passed over when its box is too far from both points, and
// the results go to out in that order, an invalid point at 1e18 m (two scans of
// 8192 outdoor points: 196 us with every candidate looked at, 89 now).
template <bool SORTED>
struct ScanNormals {
    using Args = ScanArgs;
    static constexpr int THREADS = NRM_CTA, MINB = 1;
    static __device__ __forceinline__ void run(const ScanArgs& A, unsigned bx, unsigned);
};
using ScanNormalsOp = ScanNormals<false>;

// The k smallest of the n <= NRM_BUF keys in buf, in order, to its front (one
// warp); returns their number.
__device__ __forceinline__ int select_nearest(uint64_t* buf, int n, int k, int lane) {
    static_assert(NRM_BUF == 96, "three keys a lane");
    __syncwarp();
    uint64_t a = lane < n ? buf[lane] : ~0ull, b = 32 + lane < n ? buf[32 + lane] : ~0ull,
             c = 64 + lane < n ? buf[64 + lane] : ~0ull;
    uint64_t mine = ~0ull;
    const int m = min(n, k);
    for (int r = 0; r < m; ++r) {
        const uint64_t x = min(a, min(b, c));
        const unsigned hi = (unsigned)(x >> 32);
        const unsigned H = __reduce_min_sync(0xffffffffu, hi);
        const unsigned L = __reduce_min_sync(0xffffffffu, hi == H ? (unsigned)x : 0xffffffffu);
        const uint64_t key = ((uint64_t)H << 32) | L;   // the keys differ in j
        if (a == key) a = ~0ull;
        if (b == key) b = ~0ull;
        if (c == key) c = ~0ull;
        if (lane == r) mine = key;
    }
    __syncwarp();
    if (lane < m) buf[lane] = mine;
    __syncwarp();
    return m;
}

template <bool SORTED>
__device__ __forceinline__ void ScanNormals<SORTED>::run(const ScanArgs& args, unsigned bx, unsigned) {
    const float* __restrict__ raw = args.raw;
    const float* __restrict__ soa = args.soa;
    const int32_t* __restrict__ order = args.idx;
    const int n = args.n, k = args.k, kmin = args.kmin;
    float* __restrict__ normals = args.normals;
    uint8_t* __restrict__ valid = args.valid;
    __shared__ float sx[SCAN_TILE], sy[SCAN_TILE], sz[SCAN_TILE];
    __shared__ int32_t sj[SORTED ? SCAN_TILE : 1];
    __shared__ float sbox[SORTED ? 6 : 1][32];
    __shared__ uint64_t buf[NRM_PTS][NRM_BUF];
    __shared__ int found[NRM_PTS];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const unsigned lt = (1u << lane) - 1u;
    auto word = [&](int i, int a) { return SORTED ? soa[scan_word(i, a)] : raw[3 * i + a]; };
    float p[2][3], thr[2];
    int nb[2] = {0, 0};
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const int i = (int)bx * NRM_PTS + 2 * w + q;
#pragma unroll
        for (int a = 0; a < 3; ++a) p[q][a] = i < n ? word(i, a) : 0.f;
        thr[q] = i < n ? args.r2 : -1.f;
    }
    // sorted: the CTA's own tile of SCAN_TILE first, whose points are the nearest
    const int ntile = (n + SCAN_TILE - 1) / SCAN_TILE, first = SORTED ? (int)bx * NRM_PTS / SCAN_TILE : 0;
    for (int r = 0; r < ntile; ++r) {
        const int base = (first + r < ntile ? first + r : first + r - ntile) * SCAN_TILE;
        __syncthreads();
        for (int t = threadIdx.x; t < SCAN_TILE && base + t < n; t += NRM_CTA) {
            sx[t] = word(base + t, 0); sy[t] = word(base + t, 1); sz[t] = word(base + t, 2);
            if (SORTED) sj[t] = order[base + t];
        }
        __syncthreads();
        const int m = min(SCAN_TILE, n - base);
        unsigned todo = 0xffffffffu >> (32 - (m + 31) / 32);
        if (SORTED) {
            static_assert(SCAN_TILE == 32 * 32 && NRM_CTA == 16 * 32, "32 tiles of 32, two a warp");
            for (int j = 2 * w; j < 2 * w + 2; ++j) {
                const int t = min(32 * j + lane, m - 1);   // (a tile beyond m: not looked at)
                const float v[3] = {sx[t], sy[t], sz[t]};
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    float lo = v[a], hi = v[a];
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) {
                        lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
                        hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
                    }
                    if (lane == 0) {
                        sbox[a][j] = lo;
                        sbox[3 + a][j] = hi;
                    }
                }
            }
            __syncthreads();
            bool near = false;
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                float d2 = 0.f;
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    const float d = fmaxf(fmaxf(sbox[a][lane] - p[q][a], p[q][a] - sbox[3 + a][lane]), 0.f);
                    d2 += d * d;
                }
                // (every rounding of d2 is one of the distance's, in the same order: it is no larger)
                near = near || d2 <= thr[q];
            }
            todo &= __ballot_sync(0xffffffffu, near);
        }
        while (todo) {
            const int t0 = 32 * (__ffs(todo) - 1);
            todo &= todo - 1;
            const int t = t0 + lane;
            const bool in = t < m;
            const float x = in ? sx[t] : 0.f, y = in ? sy[t] : 0.f, z = in ? sz[t] : 0.f;
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const float d2 = dist2_exact(p[q][0], p[q][1], p[q][2], x, y, z);
                const bool near = in && d2 <= thr[q];
                const unsigned bal = __ballot_sync(0xffffffffu, near);
                if (bal == 0) continue;
                uint64_t* b = buf[2 * w + q];
                if (near)
                    b[nb[q] + __popc(bal & lt)] =
                        ((uint64_t)__float_as_uint(d2) << 32) | (uint32_t)(SORTED ? sj[t] : base + t);
                nb[q] += __popc(bal);
                if (nb[q] > NRM_BUF - 32) {
                    nb[q] = select_nearest(b, nb[q], k, lane);
                    thr[q] = __uint_as_float((uint32_t)(b[nb[q] - 1] >> 32));
                }
            }
        }
    }
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        nb[q] = select_nearest(buf[2 * w + q], nb[q], k, lane);
        if (lane == 0) found[2 * w + q] = nb[q];
    }
    __syncthreads();
    // the normals: four lanes per point, eight points a warp
    if (threadIdx.x >= 4 * NRM_PTS) return;
    const int q = threadIdx.x >> 2, iq = (int)bx * NRM_PTS + q;
    int m = iq < n ? found[q] : 0;
    if (m < kmin) m = 0;
    auto J = [&](int s) { return (int)(uint32_t)buf[q][s]; };
#ifdef MP_CHECKED
    for (int s = 0; s < m; ++s)
        if (!MP_DCHECK(J(s) >= 0 && J(s) < n, "scan neighbour index", J(s))) m = 0;
#endif
    const float nv = neighbourhood_normal_quad(raw, J, m);
    if (iq >= n) return;
    if (SORTED) {
        const int a = lane & 3;
        if (a < 3) {
            args.out[scan_word(iq, a)] = m > 0 ? word(iq, a) : 1e18f;
            args.out[scan_word(iq, 3 + a)] = m > 0 ? nv : 0.f;
        }
        return;
    }
    if ((lane & 3) < 3) normals[3 * iq + (lane & 3)] = m > 0 ? nv : 0.f;
    if ((lane & 3) == 0) valid[iq] = m > 0;
}

// Compaction: the valid points in the order of (key, index) into the chunks of
// the point-major likelihood, and in input order into the broadcast pairs of
// the particle-major one. A point's slot is the number of valid points before it,
// counted over the whole scan by SCAN_PARTS threads a point: n^2 comparisons, 27 us
// at 4999 points, 38 at 8192, 53 for two scans of 8192 in one launch. (The one CTA
// before it, which compacted in input order and did not sort, took 17 us at 5000.)
struct ScanSortOp {
    using Args = ScanArgs;
    static constexpr int THREADS = SCAN_CTA, MINB = 1;
    static __device__ __forceinline__ void run(const ScanArgs& A, unsigned bx, unsigned);
};

__device__ __forceinline__ void ScanSortOp::run(const ScanArgs& args, unsigned bx, unsigned) {
    constexpr uint32_t NONE = 0xffffffffu;   // above every key
    const float* __restrict__ raw = args.raw;
    const float* __restrict__ normals = args.normals;
    const uint8_t* __restrict__ valid = args.valid;   // null: every point
    const float4* __restrict__ pts = args.tmp4;
    const int n = args.n;
    __shared__ __align__(16) uint32_t sk[SCAN_TILE];
    const int part = threadIdx.x % SCAN_PARTS, pl = threadIdx.x / SCAN_PARTS;
    const int i = (int)bx * SCAN_PTS + pl;
    const uint32_t key = (i < n && (!valid || valid[i])) ? __float_as_uint(pts[i].w) : NONE;
    uint32_t before = 0, earlier = 0, all = 0;   // valid points before this one by key, by index; all
    for (int base = 0; base < n; base += SCAN_TILE) {
        __syncthreads();
        for (int t = threadIdx.x; t < SCAN_TILE; t += SCAN_CTA) {
            const int j = base + t;
            sk[t] = (j < n && (!valid || valid[j])) ? __float_as_uint(pts[j].w) : NONE;
        }
        __syncthreads();
        const uint32_t lim = key + (base + SCAN_TILE <= i ? 1u : 0u);   // equal keys of an earlier tile count
        const bool own = i >= base && i < base + SCAN_TILE;
        for (int t = 4 * part; t < SCAN_TILE; t += 4 * SCAN_PARTS) {
            const uint4 k4 = *reinterpret_cast<const uint4*>(sk + t);
            before += (k4.x < lim) + (k4.y < lim) + (k4.z < lim) + (k4.w < lim);
            const uint32_t here = (k4.x != NONE) + (k4.y != NONE) + (k4.z != NONE) + (k4.w != NONE);
            all += here;
            if (base + SCAN_TILE <= i) earlier += here;
            if (own) {
                const int j = base + t;
                earlier += (k4.x != NONE && j < i) + (k4.y != NONE && j + 1 < i) + (k4.z != NONE && j + 2 < i) +
                           (k4.w != NONE && j + 3 < i);
                before += (k4.x == key && j < i) + (k4.y == key && j + 1 < i) + (k4.z == key && j + 2 < i) +
                          (k4.w == key && j + 3 < i);
            }
        }
    }
#pragma unroll
    for (int o = 1; o < SCAN_PARTS; o <<= 1) {
        before += __shfl_xor_sync(0xffffffffu, before, o);
        earlier += __shfl_xor_sync(0xffffffffu, earlier, o);
        all += __shfl_xor_sync(0xffffffffu, all, o);
    }
    if (bx == 0) {
        if (threadIdx.x == 0) *args.nvalid = (int32_t)all;
        // the last chunk's unused slots hold NaN, which no pose brings into a
        // grid (a far point would do for unit quaternions only: others can map
        // it to 0): the likelihood looks up whole chunks
        static_assert(MP_SCAN_CHUNK == SCAN_CTA, "one thread per slot of a chunk");
        const int64_t slot = (int64_t)(all / MP_SCAN_CHUNK) * MP_SCAN_CHUNK + threadIdx.x;
        if (slot >= all && all % MP_SCAN_CHUNK != 0)
            for (int k = 0; k < 6; ++k) args.soa[scan_word(slot, k)] = __uint_as_float(0x7fffffffu);
    }
    if (part != 0 || key == NONE) return;
    int64_t o = before, oe = earlier;
    if (!MP_DCHECK(o < n && oe < n, "compacted scan index", o)) o = oe = 0;
    float v[6];
#pragma unroll
    for (int k = 0; k < 3; ++k) args.soa[scan_word(o, k)] = v[k] = raw[3 * i + k];
    if (args.idx) args.idx[o] = i;
    if (!normals) return;   // the points alone
#pragma unroll
    for (int k = 3; k < 6; ++k) args.soa[scan_word(o, k)] = v[k] = normals[3 * i + k - 3];
#pragma unroll
    for (int k = 0; k < 3; ++k) args.pair[3 * oe + k] = make_float4(v[2 * k], v[2 * k], v[2 * k + 1], v[2 * k + 1]);
}

// One scan, or two in one launch (blockIdx.y).
struct ScanArgs2 {
    ScanArgs s[2];
};
template <typename Op, int PTS>
__device__ __forceinline__ void scan_run(const ScanArgs2& A) {
    const ScanArgs& a = A.s[blockIdx.y];
    if (blockIdx.x * PTS < (unsigned)a.n) Op::run(a, blockIdx.x, 0);
}
__global__ void __launch_bounds__(256) k_scan_to_float4(const __grid_constant__ ScanArgs2 A) {
    pdl_trigger();
    scan_run<ScanF4Op, 256>(A);
}
__global__ void __launch_bounds__(NRM_CTA) k_scan_normals(const __grid_constant__ ScanArgs2 A) {
    pdl_wait();   // (no trigger: the sort's waiting CTAs took 11 us from 4999 points' normals)
    scan_run<ScanNormalsOp, NRM_PTS>(A);
}
__global__ void __launch_bounds__(NRM_CTA) k_sorted_normals(const __grid_constant__ ScanArgs2 A) {
    pdl_wait();
    scan_run<ScanNormals<true>, NRM_PTS>(A);
}
__global__ void __launch_bounds__(SCAN_CTA) k_scan_sort(const __grid_constant__ ScanArgs2 A) {
    pdl_wait();
    scan_run<ScanSortOp, SCAN_PTS>(A);
}

// NNF: nearest valid map point to each voxel centre within r_max.
__global__ void k_nnf_build(const float4* __restrict__ pts, CellGridDev g, int nx, int ny, int64_t nvox, float ox,
                            float oy, float oz, float res, float r2, int32_t* __restrict__ nnf) {
    int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (idx >= nvox) return;
    int vx = (int)(idx % nx);
    int64_t r = idx / nx;
    int vy = (int)(r % ny);
    int vz = (int)(r / ny);
    float cx = __fadd_rn(ox, __fmul_rn(__fadd_rn((float)vx, 0.5f), res));
    float cy = __fadd_rn(oy, __fmul_rn(__fadd_rn((float)vy, 0.5f), res));
    float cz = __fadd_rn(oz, __fmul_rn(__fadd_rn((float)vz, 0.5f), res));
    int c[3];
    cell_coords(g, cx, cy, cz, c);
    int best = -1;
    float bd = INFINITY;
    for (int dz = -1; dz <= 1; ++dz)
        for (int dy = -1; dy <= 1; ++dy)
            for (int dx = -1; dx <= 1; ++dx) {
                int x = c[0] + dx, y = c[1] + dy, z = c[2] + dz;
                if (x < 0 || y < 0 || z < 0 || x >= g.dims[0] || y >= g.dims[1] || z >= g.dims[2]) continue;
                int64_t ci = ((int64_t)z * g.dims[1] + y) * g.dims[0] + x;
                for (uint32_t e = g.start[ci]; e < g.start[ci + 1]; ++e) {
                    int j = g.items[e];
                    float4 p = pts[j];
                    float d2 = dist2_exact(cx, cy, cz, p.x, p.y, p.z);
                    if (d2 <= r2 && (d2 < bd || (d2 == bd && j < best))) { bd = d2; best = j; }
                }
            }
    nnf[idx] = best;
}

// Map records in spatial order: record s holds original point perm[s].
__global__ void k_map_records(const float4* __restrict__ pts, const float* __restrict__ normals,
                              const int32_t* __restrict__ perm, int64_t n, float4* __restrict__ rec) {
    int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (s >= n) return;
    int64_t i = perm[s];
    float4 p = pts[i];
    rec[2 * s] = make_float4(p.x, p.y, p.z, normals[3 * i]);
    rec[2 * s + 1] = make_float4(normals[3 * i + 1], normals[3 * i + 2], 0.f, 0.f);
}

// Dense NNF entries from original to spatial-order map indices.
__global__ void k_nnf_remap(int32_t* __restrict__ nnf, int64_t nvox, const int32_t* __restrict__ inv) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= nvox) return;
    int v = nnf[i];
    if (v >= 0) nnf[i] = inv[v];
}

// NNF values in original map indices.
__global__ void k_nnf_query(const int32_t* __restrict__ nnf, const int32_t* __restrict__ perm, int nx, int ny, int nz,
                            const int32_t* __restrict__ vox, int64_t m, int32_t* __restrict__ out) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= m) return;
    int x = vox[3 * i], y = vox[3 * i + 1], z = vox[3 * i + 2];
    bool in = x >= 0 && y >= 0 && z >= 0 && x < nx && y < ny && z < nz;
    int s = in ? nnf[((int64_t)z * ny + y) * nx + x] : -1;
    out[i] = s < 0 ? -1 : perm[s];
}

// Spatial order of the map points: Morton code of their cell (side 4 voxels,
// or larger so that 1024 cells cover the box), ties by index.
void morton_order(const std::vector<float>& h, int64_t n, const float lo[3], const float hi[3], float cell,
                  std::vector<int32_t>& perm) {
    auto spread = [](uint32_t x) {
        x &= 0x3ffu;
        x = (x | (x << 16)) & 0x030000FFu;
        x = (x | (x << 8)) & 0x0300F00Fu;
        x = (x | (x << 4)) & 0x030C30C3u;
        x = (x | (x << 2)) & 0x09249249u;
        return x;
    };
    float ext = std::max(hi[0] - lo[0], std::max(hi[1] - lo[1], hi[2] - lo[2]));
    cell = std::max(cell, ext / 1023.0f);
    std::vector<uint64_t> key((size_t)n);
    for (int64_t i = 0; i < n; ++i) {
        uint32_t c[3];
        for (int a = 0; a < 3; ++a) {
            float f = (h[3 * i + a] - lo[a]) / cell;
            c[a] = (uint32_t)std::min(std::max(f, 0.0f), 1023.0f);
        }
        uint32_t code = spread(c[0]) | (spread(c[1]) << 1) | (spread(c[2]) << 2);
        key[(size_t)i] = ((uint64_t)code << 32) | (uint64_t)i;
    }
    std::sort(key.begin(), key.end());
    perm.resize((size_t)n);
    for (int64_t s = 0; s < n; ++s) perm[(size_t)s] = (int32_t)(key[(size_t)s] & 0xffffffffu);
}

__global__ void k_pts_from_xyz(const float* __restrict__ xyz, int64_t n, float4* __restrict__ out) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < n) out[i] = make_float4(xyz[3 * i], xyz[3 * i + 1], xyz[3 * i + 2], 0.f);
}

// Builds the cell grid of the (valid) points with cell side h over [lo, hi].
int build_cells(mp_ctx* c, const float4* pts, const uint8_t* valid, int64_t n, float h, const float lo[3],
                const float hi[3], CellGridDev& g, int32_t** cell_of_out) {
    g.inv_h = 1.0f / h;
    g.ncell = 1;
    for (int a = 0; a < 3; ++a) {
        g.og[a] = lo[a] - h;
        g.dims[a] = (int)std::floor((hi[a] - g.og[a]) / h) + 2;
        g.ncell *= g.dims[a];
    }
    if (g.ncell > (int64_t)1 << 30) return mp_fail(c, MP_EINVAL, "cell grid too large (%lld cells)", (long long)g.ncell);
    int32_t* cell_of = nullptr;
    uint32_t *count = nullptr, *fill = nullptr;
    MP_CUDA(c, cudaMalloc(&cell_of, sizeof(int32_t) * (size_t)n));
    MP_CUDA(c, cudaMalloc(&count, sizeof(uint32_t) * (size_t)(g.ncell + 1)));
    MP_CUDA(c, cudaMalloc(&fill, sizeof(uint32_t) * (size_t)(g.ncell + 1)));
    MP_CUDA(c, cudaMalloc(&g.start, sizeof(uint32_t) * (size_t)(g.ncell + 1)));
    MP_CUDA(c, cudaMalloc(&g.items, sizeof(int32_t) * (size_t)n));
    MP_CUDA(c, cudaMemsetAsync(count, 0, sizeof(uint32_t) * (size_t)(g.ncell + 1), c->stream));
    MP_CUDA(c, cudaMemsetAsync(fill, 0, sizeof(uint32_t) * (size_t)(g.ncell + 1), c->stream));
    k_cell_count<<<grid_for(n, 256), 256, 0, c->stream>>>(pts, valid, n, g, cell_of, count);
    MP_LAUNCHED(c);
    int rc = mp_launch_exclusive_scan(c, count, g.start, g.ncell + 1);
    if (rc) return rc;
    k_cell_fill<<<grid_for(n, 256), 256, 0, c->stream>>>(cell_of, n, g.start, fill, g.items);
    MP_LAUNCHED(c);
    MP_CUDA(c, cudaStreamSynchronize(c->stream));
    cudaFree(count);
    cudaFree(fill);
    *cell_of_out = cell_of;
    return MP_OK;
}

void free_cells(CellGridDev& g) {
    cudaFree(g.start);
    cudaFree(g.items);
    g.start = nullptr;
    g.items = nullptr;
}

}  // namespace

// Map preprocessing: normals, validity, NNF geometry (host, FP32 sequence),
// NNF grid and records. xyz_dev: n_map x 3 float32 on the device.
int mp_launch_map_prepare(mp_ctx* c, const float* xyz_dev) {
    int64_t n = c->n_map;
    k_pts_from_xyz<<<grid_for(n, 256), 256, 0, c->stream>>>(xyz_dev, n, c->map_pts);
    MP_LAUNCHED(c);
    // bounding box of all points (exact FP32 min/max on the host)
    std::vector<float> h(3 * (size_t)n);
    MP_CUDA(c, cudaMemcpyAsync(h.data(), xyz_dev, sizeof(float) * 3 * (size_t)n, cudaMemcpyDeviceToHost, c->stream));
    MP_CUDA(c, cudaStreamSynchronize(c->stream));
    float lo[3] = {INFINITY, INFINITY, INFINITY}, hi[3] = {-INFINITY, -INFINITY, -INFINITY};
    for (int64_t i = 0; i < n; ++i)
        for (int a = 0; a < 3; ++a) {
            float v = h[3 * i + a];
            if (!std::isfinite(v)) return mp_fail(c, MP_EINVAL, "map point %lld is not finite", (long long)i);
            lo[a] = fminf(lo[a], v);
            hi[a] = fmaxf(hi[a], v);
        }
    // normals through a cell grid of side r_cov (+0.1 % margin)
    CellGridDev g;
    int32_t* cell_of = nullptr;
    int rc = build_cells(c, c->map_pts, nullptr, n, c->p.r_cov * 1.001f, lo, hi, g, &cell_of);
    if (rc) return rc;
    float r2c = c->p.r_cov * c->p.r_cov;
    k_map_normals<<<grid_for(n, 128), 128, 0, c->stream>>>(c->map_pts, n, g, r2c, c->p.cov_k, c->p.cov_min,
                                                            c->map_normals, c->map_valid);
    MP_LAUNCHED(c);
    MP_CUDA(c, cudaStreamSynchronize(c->stream));
    free_cells(g);
    cudaFree(cell_of);
    // NNF geometry from the valid points, by the FP32 sequence:
    // o = lo - r_max; n = floor(((hi + r_max) - o) * inv_res) + 1; off = -(o * inv_res)
    std::vector<uint8_t> v((size_t)n);
    MP_CUDA(c, cudaMemcpy(v.data(), c->map_valid, (size_t)n, cudaMemcpyDeviceToHost));
    float vlo[3] = {INFINITY, INFINITY, INFINITY}, vhi[3] = {-INFINITY, -INFINITY, -INFINITY};
    int64_t nv = 0;
    for (int64_t i = 0; i < n; ++i) {
        if (!v[i]) continue;
        nv++;
        for (int a = 0; a < 3; ++a) {
            vlo[a] = fminf(vlo[a], h[3 * i + a]);
            vhi[a] = fmaxf(vhi[a], h[3 * i + a]);
        }
    }
    c->n_map_valid = nv;
    if (nv == 0) return mp_fail(c, MP_EINVAL, "no map point has %d neighbours within r_cov", c->p.cov_min);
    volatile float res = c->p.nnf_res, rmax = c->p.r_max;
    volatile float inv_res = 1.0f / res;
    c->nnf_inv_res = inv_res;
    c->nnf_voxels = 1;
    for (int a = 0; a < 3; ++a) {
        volatile float o = vlo[a] - rmax;
        volatile float t1 = vhi[a] + rmax;
        volatile float t2 = t1 - o;
        volatile float t3 = t2 * inv_res;
        volatile float po = o * inv_res;
        c->nnf_origin[a] = o;
        c->nnf_dims[a] = (int32_t)std::floor((float)t3) + 1;
        c->nnf_off[a] = -po;
        c->nnf_voxels *= c->nnf_dims[a];
        c->map_lo[a] = vlo[a];
        c->map_hi[a] = vhi[a];
    }
    if (c->nnf_voxels >= ((int64_t)1 << 31))
        return mp_fail(c, MP_EINVAL, "NNF grid of %lld voxels exceeds 2^31", (long long)c->nnf_voxels);
    // dense NNF of original indices (temporary)
    int32_t* dense = nullptr;
    MP_CUDA(c, cudaMalloc(&dense, sizeof(int32_t) * (size_t)c->nnf_voxels));
    rc = build_cells(c, c->map_pts, c->map_valid, n, c->p.r_max * 1.001f, vlo, vhi, g, &cell_of);
    if (rc) { cudaFree(dense); return rc; }
    float r2 = c->p.r_max * c->p.r_max;
    k_nnf_build<<<grid_for(c->nnf_voxels, 256), 256, 0, c->stream>>>(
        c->map_pts, g, c->nnf_dims[0], c->nnf_dims[1], c->nnf_voxels, c->nnf_origin[0], c->nnf_origin[1],
        c->nnf_origin[2], c->p.nnf_res, r2, dense);
    MP_LAUNCHED(c);
    // spatial (Morton) order of the map records: the records that nearby
    // voxels point to share cache lines
    std::vector<int32_t> perm, inv((size_t)n);
    morton_order(h, n, lo, hi, 4.0f * c->p.nnf_res, perm);
    for (int64_t s = 0; s < n; ++s) inv[(size_t)perm[(size_t)s]] = (int32_t)s;
    int32_t* inv_dev = nullptr;
    MP_CUDA(c, cudaMalloc(&c->map_perm, sizeof(int32_t) * (size_t)n));
    MP_CUDA(c, cudaMalloc(&inv_dev, sizeof(int32_t) * (size_t)n));
    MP_CUDA(c, cudaMemcpyAsync(c->map_perm, perm.data(), sizeof(int32_t) * (size_t)n, cudaMemcpyHostToDevice, c->stream));
    MP_CUDA(c, cudaMemcpyAsync(inv_dev, inv.data(), sizeof(int32_t) * (size_t)n, cudaMemcpyHostToDevice, c->stream));
    k_map_records<<<grid_for(n, 256), 256, 0, c->stream>>>(c->map_pts, c->map_normals, c->map_perm, n, c->map_rec);
    MP_LAUNCHED(c);
    k_nnf_remap<<<grid_for(c->nnf_voxels, 256), 256, 0, c->stream>>>(dense, c->nnf_voxels, inv_dev);
    MP_LAUNCHED(c);
    MP_CUDA(c, cudaStreamSynchronize(c->stream));
    c->nnf = dense;
    free_cells(g);
    cudaFree(cell_of);
    cudaFree(inv_dev);
    return MP_OK;
}

namespace {

ScanArgs scan_args(mp_ctx* c, const float* raw, int n) {
    ScanArgs A;
    A.raw = raw;
    A.n = n;
    A.r2 = c->p.r_cov * c->p.r_cov;
    A.k = c->p.cov_k;
    A.kmin = c->p.cov_min;
    A.inv_cell = 0.25f / c->p.nnf_res;
    A.tmp4 = c->scan_tmp4;
    A.normals = c->scan_normals;
    A.valid = c->scan_valid;
    A.idx = nullptr;
    A.pair = c->scan_pair;
    A.soa = c->scan_soa;
    A.nvalid = c->scan_nvalid;
    A.out = nullptr;
    return A;
}

}  // namespace

// Per-step scan Gaussians (brute-force radius kNN in shared-memory tiles) and
// the valid points, sorted and in input order.
int mp_launch_scan_prepare(mp_ctx* c, cudaStream_t s) {
    const int n = c->n_prep = c->n_scan;
    if (n == 0) {
        MP_CUDA(c, cudaMemsetAsync(c->scan_nvalid, 0, sizeof(int32_t), s));
        return MP_OK;
    }
    const ScanArgs a = scan_args(c, c->scan_raw, n);
    const ScanArgs2 A = {{a, a}};
    k_scan_to_float4<<<grid_for(n, 256), 256, 0, s>>>(A);
    MP_LAUNCHED(c);
    MP_CUDA(c, launch_next(k_scan_normals, grid_for(n, NRM_PTS), NRM_CTA, 0, s, A));
    MP_LAUNCHED(c);
    MP_CUDA(c, launch_next(k_scan_sort, grid_for(n, SCAN_PTS), SCAN_CTA, 0, s, A));
    MP_LAUNCHED(c);
    return MP_OK;
}

// Point Gaussians of m <= 2 point arrays (n >= 1 points each): all points sorted (and
// their indices), then their normals, an invalid point at 1e18 m.
int mp_launch_point_gaussians(mp_ctx* c, const PointScan* in, int m) {
    ScanArgs2 A;
    int n = 0;
    for (int k = 0; k < 2; ++k) {
        const PointScan& p = in[k < m ? k : 0];
        ScanArgs& a = A.s[k] = scan_args(c, p.raw, p.n);
        a.tmp4 = p.tmp4;
        a.normals = nullptr;
        a.valid = nullptr;
        a.pair = nullptr;
        a.soa = p.sorted;
        a.idx = p.idx;
        a.nvalid = p.count;
        a.out = p.out;
        n = std::max(n, p.n);
    }
    k_scan_to_float4<<<dim3(grid_for(n, 256), m), 256, 0, c->stream>>>(A);
    MP_LAUNCHED(c);
    MP_CUDA(c, launch_next(k_scan_sort, dim3(grid_for(n, SCAN_PTS), m), SCAN_CTA, 0, c->stream, A));
    MP_LAUNCHED(c);
    MP_CUDA(c, launch_next(k_sorted_normals, dim3(grid_for(n, NRM_PTS), m), NRM_CTA, 0, c->stream, A));
    MP_LAUNCHED(c);
    return MP_OK;
}

// Grouped scan stage: every instance's scan is read from the batch's device
// scan buffer; the outputs go to each instance's own scan buffers.
int mp_plan_scan(mp_group* G, int, std::vector<GOp>& plan) {
    std::vector<ScanArgs> tab;
    std::vector<int64_t> b256, b64;
    for (int i = 0; i < G->size(); ++i) {
        const int n = G->n_scan[i];
        tab.push_back(scan_args(G->ctx[i], G->scan_dev + G->scan_off[i], n));
        b256.push_back((n + 255) / 256);
        b64.push_back((n + SCAN_PTS - 1) / SCAN_PTS);
    }
    const ScanArgs* t = G->upload(tab);
    unsigned nblk = 0;
    const GBlk* m = G->block_map(b256, &nblk);
    plan_kernel<ScanF4Op>(plan, t, m, nblk);
    static_assert(NRM_PTS == SCAN_PTS, "one block map for both");
    m = G->block_map(b64, &nblk);
    plan_kernel<ScanNormalsOp>(plan, t, m, nblk);
    plan_kernel<ScanSortOp>(plan, t, m, nblk);
    return G->err;
}

int mp_launch_nnf_query(mp_ctx* c, const int32_t* vox_dev, int64_t m, int32_t* out_dev) {
    if (m == 0) return MP_OK;
    k_nnf_query<<<grid_for(m, 256), 256, 0, c->stream>>>(c->nnf, c->map_perm, c->nnf_dims[0], c->nnf_dims[1],
                                                         c->nnf_dims[2], vox_dev, m, out_dev);
    MP_LAUNCHED(c);
    return MP_OK;
}
