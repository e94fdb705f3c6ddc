// Scan-to-scan GICP odometry of the prediction step (Sec. III-B): DeltaT_t
// ~ T_{t-1}^-1 T_t from the current scan (source) and the previous one
// (target), and Sigma^DeltaT from the Gauss-Newton Hessian at the result.
//
// One cooperative kernel runs all iterations on the sorted points of both scans
// (those without a normal at 1e18 m: out of reach as targets, skipped as sources).
// For the current estimate T = (R, t) (FP64, in shared memory):
//  * decisions in FP32 on T's rounding to float (R from the unit quaternion,
//    q = R mu + t by the fixed sequence, squared distances un-fused); the
//    correspondence is the target point of smallest squared distance, ties to
//    the smaller index, within r_corr. Eight threads share a source point's
//    search, over the tiles of 64 target points whose bounding box is near
//    enough to one of their warp's four points: the sort makes tiles and warps
//    compact, and most tiles are skipped. Each correspondence adds J^T Omega J
//    and J^T Omega e with the GICP plane covariances (the same closed-form Omega
//    and target-frame sums as the likelihood kernel); a CTA writes one partial.
//    A search starts from the last iteration's correspondence.
//  * after a grid barrier every CTA sums the partials in FP64 and its first warp
//    rotates the target-frame sums to the source frame, solves the damped system
//    (Gauss-Jordan with partial pivoting) and sets T <- T exp(delta); once max
//    |delta| < tol all stop. The Hessian of the last iteration is kept:
//    Sigma^DeltaT = H^-1 is taken on the host.
// Bound by latency: at two scans of 8192 points 33 us an iteration, 13 of them
// the barrier and the FP64 step (28 with its instructions on one thread) and the
// rest the search (75 us without the last correspondence as a bound), before it
// 53 us for the scans' order and 88 for their normals. mp_gicp at 8192 points and
// six iterations: 3930 us with all pairs of points tested and two launches an
// iteration, 425 now.
#include "mp_internal.cuh"

#include <algorithm>
#include <cmath>
#include <cstring>

struct GicpBufs {
    int cap;
    float *src_raw, *tgt_raw;
    float *sorted, *src_soa, *tgt_soa;   // the points, sorted (scan_word): two scans' points; with their normals
    int32_t *idx, *tgt_idx, *counts;     // their original indices; points of src and tgt, error bits
    float4* tmp4;
    float* box;         // target tiles' bounding boxes
    int32_t* corr;      // correspondences
    float* partial;     // 2 x CTAs x 32
    GridBar* bar;
    int grid;           // resident CTAs of k_gicp
    double* state;      // q[4], t[3], H[21], done flag, iterations, n_corr
    float* prev;        // previous scan kept for mp_step_gicp (cap x 3)
    int n_prev;
    double last_T[16];
    int have_last;
};

namespace {

constexpr int GB = 512;        // threads per CTA (one an SM: fewer partials for every CTA to sum)
constexpr int GPARTS = 8;      // threads sharing a source point's search
constexpr int GPTS = GB / GPARTS;   // source points a CTA takes at a time (four a warp)
constexpr int GTILE = 64;      // target points per tile
constexpr int NPART = 32;      // floats per partial: 27 sums + count (+ pad)
constexpr int ST_Q = 0, ST_T = 4, ST_H = 7, ST_DONE = 28, ST_IT = 29, ST_NC = 30, ST_N = 32;

// One registration. Scans: sorted points and normals in chunks of six planes
// (scan_word), invalid points at 1e18 m, and the points' original indices.
struct GicpArgs {
    const float *src, *tgt;
    const int32_t* tgt_idx;
    int n_src, n_tgt;
    float* box;              // 6 per target tile: lower and upper corner
    int32_t* corr;           // a source point's correspondence in the last iteration
    double* state;
    float* partial;          // [2][grid][NPART]: two iterations' partials in turn
    float r2, half_a, two_eps, quarter_a;
    double lambda, eps, tol;
    int max_iters;
    GridBar* bar;
    int32_t* err;
    long long budget;
};

__device__ __forceinline__ float gicp_word(const float* s, int i, int k) { return __ldg(s + scan_word(i, k)); }

__device__ __forceinline__ bool gicp_valid(const float* s, int i) { return gicp_word(s, i, 0) < 1e17f; }

// Nearest target point (squared distance by the decision sequence, ties to the
// smaller original index) of this thread's source point, over the tiles whose
// box comes near enough to one of the warp's four points; the point's GPARTS
// threads share a tile's points. bj: a first candidate, the correspondence of
// the iteration before (-1: none), whose distance is the bound from the start;
// on return the sorted index found (-1: none within r2).
__device__ __forceinline__ void gicp_nearest(const GicpArgs& A, int nt, bool have, const float q[3], int& bj) {
    const int lane = threadIdx.x & 31, part = lane % GPARTS;
    const int ntile = (nt + GTILE - 1) / GTILE;
    float best = have ? A.r2 : -1.f;   // <= r2 counts: the index decides ties only among points found
    int bidx = 0x7fffffff, first = bj;
    bj = -1;
    auto offer = [&](int j, float d2) {
        if (d2 <= best) {
            const int idx = __ldg(A.tgt_idx + j);
            if (d2 < best || idx < bidx) {
                best = d2;
                bj = j;
                bidx = idx;
            }
        }
    };
    if (first >= 0)
        offer(first, dist2_exact(q[0], q[1], q[2], gicp_word(A.tgt, first, 0), gicp_word(A.tgt, first, 1),
                                 gicp_word(A.tgt, first, 2)));
    float px[4], py[4], pz[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        px[k] = __shfl_sync(0xffffffffu, q[0], k * GPARTS);
        py[k] = __shfl_sync(0xffffffffu, q[1], k * GPARTS);
        pz[k] = __shfl_sync(0xffffffffu, q[2], k * GPARTS);
    }
    for (int t0 = 0; t0 < ntile; t0 += 32) {
        const int t = t0 + lane;
        bool near = false;
        float lim[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) lim[k] = __shfl_sync(0xffffffffu, best, k * GPARTS);
        if (t < ntile) {
            const float* bx = A.box + 6 * t;
            const float x0 = __ldcg(bx), y0 = __ldcg(bx + 1), z0 = __ldcg(bx + 2);
            const float x1 = __ldcg(bx + 3), y1 = __ldcg(bx + 4), z1 = __ldcg(bx + 5);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const float dx = fmaxf(fmaxf(x0 - px[k], px[k] - x1), 0.f);
                const float dy = fmaxf(fmaxf(y0 - py[k], py[k] - y1), 0.f);
                const float dz = fmaxf(fmaxf(z0 - pz[k], pz[k] - z1), 0.f);
                // (the bound's own rounding: a few parts in 1e7)
                near = near || (dx * dx + dy * dy + dz * dz) * 0.99999f <= lim[k];
            }
        }
        unsigned todo = __ballot_sync(0xffffffffu, near);
        if (todo == 0) continue;
        while (todo) {
            const int j0 = (t0 + __ffs(todo) - 1) * GTILE + part;
            todo &= todo - 1;
            // a tile is part of a chunk, and whole chunks are allocated: all loads go ahead
            static_assert(MP_SCAN_CHUNK % GTILE == 0, "a tile's words are at constant distances");
            const float* w = A.tgt + scan_word(j0, 0);
            float d2[GTILE / GPARTS], least = INFINITY;
#pragma unroll
            for (int e = 0; e < GTILE / GPARTS; ++e) {
                const float* v = w + e * GPARTS;
                d2[e] = dist2_exact(q[0], q[1], q[2], __ldg(v), __ldg(v + MP_SCAN_CHUNK), __ldg(v + 2 * MP_SCAN_CHUNK));
                if (j0 + e * GPARTS >= nt) d2[e] = INFINITY;
                least = fminf(least, d2[e]);
            }
            if (least <= best)
#pragma unroll
                for (int e = 0; e < GTILE / GPARTS; ++e)
                    if (j0 + e * GPARTS < nt) offer(j0 + e * GPARTS, d2[e]);
        }
        // the parts share what they found
#pragma unroll
        for (int o = 1; o < GPARTS; o <<= 1) {
            const float b2 = __shfl_xor_sync(0xffffffffu, best, o);
            const int j2 = __shfl_xor_sync(0xffffffffu, bj, o), i2 = __shfl_xor_sync(0xffffffffu, bidx, o);
            if (b2 < best || (b2 == best && i2 < bidx)) {
                best = b2;
                bj = j2;
                bidx = i2;
            }
        }
    }
}

// The sums of a correspondence: target-frame J^T Omega J and J^T Omega e with
// J~ = [ [q~]x , -I ] and Omega in closed form, and a count of one.
__device__ __forceinline__ void gicp_terms(const GicpArgs& A, const float R[9], const float qt[3], const float q[3], int k,
                                           int j, float acc[NPART]) {
    const float qtx = qt[0], qty = qt[1], qtz = qt[2];
    const float ex = gicp_word(A.tgt, j, 0) - q[0], ey = gicp_word(A.tgt, j, 1) - q[1], ez = gicp_word(A.tgt, j, 2) - q[2];
    const float nsx = gicp_word(A.src, k, 3), nsy = gicp_word(A.src, k, 4), nsz = gicp_word(A.src, k, 5);   // source normal
    const float wx = gicp_word(A.tgt, j, 3), wy = gicp_word(A.tgt, j, 4), wz = gicp_word(A.tgt, j, 5);      // target normal
    const float ux = R[0] * nsx + R[1] * nsy + R[2] * nsz;
    const float uy = R[3] * nsx + R[4] * nsy + R[5] * nsz;
    const float uz = R[6] * nsx + R[7] * nsy + R[8] * nsz;
    const float sg = copysignf(1.f, ux * wx + uy * wy + uz * wz);
    const float sx = fmaf(sg, wx, ux), sy = fmaf(sg, wy, uy), sz = fmaf(sg, wz, uz);
    const float dx = fmaf(-sg, wx, ux), dy = fmaf(-sg, wy, uy), dz = fmaf(-sg, wz, uz);
    const float dd = dx * dx + dy * dy + dz * dz;
    const float ls = fmaf(A.half_a, dd, A.two_eps), ld = fmaf(-A.half_a, dd, 2.f);
    const float rr = A.quarter_a / (ls * ld);
    const float as = ld * rr, ad = ls * rr;
    const float Psx = as * sx, Psy = as * sy, Psz = as * sz, Qdx = ad * dx, Qdy = ad * dy, Qdz = ad * dz;
    const float Oxx = fmaf(Psx, sx, fmaf(Qdx, dx, 0.5f)), Oyy = fmaf(Psy, sy, fmaf(Qdy, dy, 0.5f));
    const float Ozz = fmaf(Psz, sz, fmaf(Qdz, dz, 0.5f));
    const float Oxy = fmaf(Psx, sy, Qdx * dy), Oxz = fmaf(Psx, sz, Qdx * dz), Oyz = fmaf(Psy, sz, Qdy * dz);
    const float gx = Oxx * ex + Oxy * ey + Oxz * ez;
    const float gy = Oxy * ex + Oyy * ey + Oyz * ez;
    const float gz = Oxz * ex + Oyz * ey + Ozz * ez;
    const float P00 = qty * Oxz - qtz * Oxy, P01 = qty * Oyz - qtz * Oyy, P02 = qty * Ozz - qtz * Oyz;
    const float P10 = qtz * Oxx - qtx * Oxz, P11 = qtz * Oxy - qtx * Oyz, P12 = qtz * Oxz - qtx * Ozz;
    const float P20 = qtx * Oxy - qty * Oxx, P21 = qtx * Oyy - qty * Oxy, P22 = qtx * Oyz - qty * Oxz;
    // Hww (6), Hwv (9), Hvv (6), bw (3), bv (3), count
    acc[0] += qty * P02 - qtz * P01;
    acc[1] += qtz * P00 - qtx * P02;
    acc[2] += qtx * P01 - qty * P00;
    acc[3] += qtz * P10 - qtx * P12;
    acc[4] += qtx * P11 - qty * P10;
    acc[5] += qtx * P21 - qty * P20;
    acc[6] += P00; acc[7] += P01; acc[8] += P02; acc[9] += P10; acc[10] += P11; acc[11] += P12;
    acc[12] += P20; acc[13] += P21; acc[14] += P22;
    acc[15] += Oxx; acc[16] += Oxy; acc[17] += Oxz; acc[18] += Oyy; acc[19] += Oyz; acc[20] += Ozz;
    acc[21] += gy * qtz - gz * qty;
    acc[22] += gz * qtx - gx * qtz;
    acc[23] += gx * qty - gy * qtx;
    acc[24] += -gx; acc[25] += -gy; acc[26] += -gz;
    acc[27] += 1.f;
}

// s(x) = sin(th/2)/th, c = cos(th/2), a = (1 - cos th)/th^2, b = (th - sin th)/th^3
// as power series in th^2 (eight terms: below 4e-20 for th <= 1/2).
__constant__ double gicp_series[4][8] = {
    {1. / 2, -1. / 48, 1. / 3840, -1. / 645120, 1. / 185794560, -1. / 81749606400., 1. / 51011754393600.,
     -1. / 42849873690624000.},
    {1., -1. / 8, 1. / 384, -1. / 46080, 1. / 10321920, -1. / 3715891200., 1. / 1961990553600., -1. / 1428329123020800.},
    {1. / 2, -1. / 24, 1. / 720, -1. / 40320, 1. / 3628800, -1. / 479001600., 1. / 87178291200., -1. / 20922789888000.},
    {1. / 6, -1. / 120, 1. / 5040, -1. / 362880, 1. / 39916800, -1. / 6227020800., 1. / 1307674368000.,
     -1. / 355687428096000.}};

// The estimate's pose as the iterations use it: unit quaternion and rotation in
// FP64, and the decisions' FP32 pose.
struct GicpPose {
    double qn[4], R[9];
    float q32[4], t32[3];
};

// One warp: the rotation and the FP32 pose of the unit quaternion P.qn and st's
// translation, an entry a lane.
__device__ __forceinline__ void gicp_pose(const double* st, GicpPose& P) {
    const int lane = threadIdx.x & 31;
    __syncwarp();
    if (lane < 9) {
        const int i = lane / 3, j = lane % 3, i1 = (i + 1) % 3, i2 = (i + 2) % 3;
        const bool diag = i == j;
        const double u = diag ? P.qn[i1] : P.qn[i], u2 = diag ? u : P.qn[j];
        const double v = diag ? P.qn[i2] : P.qn[3], v2 = diag ? v : j == i2 ? P.qn[i1] : -P.qn[i2];
        const double e = u * u2 + v * v2;
        P.R[lane] = diag ? 1.0 - 2.0 * e : 2.0 * e;
    } else if (lane < 13) {
        P.q32[lane - 9] = (float)P.qn[lane - 9];
    } else if (lane < 16) {
        P.t32[lane - 13] = (float)st[ST_T + lane - 13];
    }
    __syncwarp();
}

// The partials of an iteration, summed by the CTA in FP64: warp w takes its
// share of them in order, lane a the sum a; then the warps in order. s: a row a warp.
__device__ __forceinline__ void gicp_sum(const float* partial, int count, double (*s)[NPART], double S[NPART]) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int per = (count + GB / 32 - 1) / (GB / 32), b0 = min(w * per, count), b1 = min(b0 + per, count);
    double v = 0.0;
#pragma unroll 8
    for (int b = b0; b < b1; ++b) v += (double)__ldcg(partial + b * NPART + lane);
    s[w][lane] = v;
    __syncthreads();
    if (threadIdx.x < NPART) {
        double t = 0.0;
        for (int k = 0; k < GB / 32; ++k) t += s[k][threadIdx.x];
        S[threadIdx.x] = t;
    }
    __syncthreads();
}

// One warp: the step of an iteration. On GB300 an FP64 instruction holds its
// quarter of the SM for 64 cycles, whatever the number of active lanes, so the
// step is laid out for few instructions: an entry or a row a lane.
// Work: S (the sums), T (27 values of scratch), M (the system), P, st.
__device__ void gicp_step(const double* S, double* T, double (*M)[7], double* st, GicpPose& P, double lambda, double eps,
                          double tol) {
    constexpr unsigned ALL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    // the blocks ww, wv, vv in the source frame, B -> R^T B R, and b -> -R^T b
    const int blk = lane / 9, i = lane % 9 / 3, j = lane % 3;
    if (lane < 27) {
        double v = 0.0;
#pragma unroll
        for (int l = 0; l < 3; ++l) {
            const int lo = min(i, l), hi = max(i, l), sym = lo * 3 - lo * (lo - 1) / 2 + hi - lo;
            v += S[blk == 1 ? 6 + 3 * i + l : blk == 0 ? sym : 15 + sym] * P.R[3 * l + j];
        }
        T[lane] = v;
    }
    __syncwarp();
    if (lane < 27) {
        double v = 0.0;
#pragma unroll
        for (int k = 0; k < 3; ++k) v += P.R[3 * k + i] * T[9 * blk + 3 * k + j];
        const int r = blk == 2 ? 3 + i : i, c = blk == 0 ? j : 3 + j;
        if (r <= c) {   // the upper triangle and its mirror
            st[ST_H + r * 6 - r * (r - 1) / 2 + c - r] = v;
            M[r][c] = r == c ? v + (lambda * v + eps) : v;
            M[c][r] = M[r][c];
        }
    }
    if (lane < 6) {
        const int a = lane % 3, o = lane < 3 ? 21 : 24;
        M[lane][6] = -(P.R[a] * S[o] + P.R[3 + a] * S[o + 1] + P.R[6 + a] * S[o + 2]);
    }
    __syncwarp();
    // Gauss-Jordan elimination, a row a lane; the pivot is the largest entry of
    // the rows not yet used (magnitudes compared as integers)
    double A[7], diag = 1.0;
#pragma unroll
    for (int k = 0; k < 7; ++k) A[k] = lane < 6 ? M[lane][k] : 0.0;
    bool ok = S[27] >= 6.0;   // the same on every lane
    int col = -1;             // the column whose pivot row this is
#pragma unroll
    for (int c = 0; c < 6; ++c) {
        const long long mag = __double_as_longlong(A[c]) & 0x7fffffffffffffffll;
        long long top = lane < 6 && col < 0 ? mag : -1;
        int piv = lane;
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) {
            const long long t2 = __shfl_xor_sync(ALL, top, o);
            const int p2 = __shfl_xor_sync(ALL, piv, o);
            if (t2 > top || (t2 == top && p2 < piv)) {
                top = t2;
                piv = p2;
            }
        }
        piv = __shfl_sync(ALL, piv, 0);
        top = __shfl_sync(ALL, top, 0);
        ok = ok && top > 0 && top <= 0x7ff0000000000000ll;   // neither 0 nor NaN
        const double p = __shfl_sync(ALL, A[c], piv);
        const double f = A[c] / p;
#pragma unroll
        for (int k = c + 1; k < 7; ++k) {
            const double u = __shfl_sync(ALL, A[k], piv);
            if (lane != piv) A[k] -= f * u;
        }
        if (lane == piv) {
            col = c;
            diag = p;
        }
    }
    const double x = A[6] / diag;
    if (col >= 0) T[col] = x;
    __syncwarp();
    if (lane == 0) {
        st[ST_NC] = S[27];
        st[ST_IT] += 1.0;
        if (!ok) st[ST_DONE] = 2.0;   // too few correspondences or singular
    }
    if (!ok) return;
    // exp(delta): rotation vector w, translation part v; lane k of each three has entry k
    const int k = lane % 3, i1 = (k + 1) % 3, i2 = (k + 2) % 3;
    const double w0 = T[0], w1 = T[1], w2 = T[2], wk = T[k], wi1 = T[i1], wi2 = T[i2], vk = T[3 + k];
    const bool small = __all_sync(ALL, lane >= 6 || fabs(T[lane]) < tol);
    const double th2 = w0 * w0 + w1 * w1 + w2 * w2;
    double s, c, a, b;
    if (th2 < 0.25) {
        const double* co = gicp_series[lane & 3];
        double y = co[7];
#pragma unroll
        for (int n = 6; n >= 0; --n) y = y * th2 + co[n];
        s = __shfl_sync(ALL, y, 0);
        c = __shfl_sync(ALL, y, 1);
        a = __shfl_sync(ALL, y, 2);
        b = __shfl_sync(ALL, y, 3);
    } else {
        const double th = sqrt(th2);
        double sh;
        sincos(0.5 * th, &sh, &c);
        s = sh / th;
        a = 2.0 * s * s;   // 1 - cos th = 2 sin^2(th/2)
        b = (th - 2.0 * sh * c) / (th2 * th);
    }
    const double wv = wi1 * T[3 + i2] - wi2 * T[3 + i1];
    const double wwv = wi1 * __shfl_sync(ALL, wv, i2) - wi2 * __shfl_sync(ALL, wv, i1);
    const double t = vk + a * wv + b * wwv;
    const double tr = P.R[3 * k] * __shfl_sync(ALL, t, 0) + P.R[3 * k + 1] * __shfl_sync(ALL, t, 1) +
                      P.R[3 * k + 2] * __shfl_sync(ALL, t, 2);
    // T <- T exp(delta)
    const double qw = P.qn[3];
    const double nv = qw * (s * wk) + P.qn[k] * c + s * (P.qn[i1] * wi2 - P.qn[i2] * wi1);
    const double nw = qw * c - s * (P.qn[0] * w0 + P.qn[1] * w1 + P.qn[2] * w2);
    const double n0 = __shfl_sync(ALL, nv, 0), n1 = __shfl_sync(ALL, nv, 1), n2 = __shfl_sync(ALL, nv, 2);
    // both factors are unit to rounding: one Newton step for 1/|n|
    const double ni = 1.5 - 0.5 * (n0 * n0 + n1 * n1 + n2 * n2 + nw * nw);
    __syncwarp();
    if (lane < 4) st[ST_Q + lane] = P.qn[lane] = (lane < 3 ? nv : nw) * ni;
    if (lane < 3) st[ST_T + lane] += tr;
    if (lane == 0 && small) st[ST_DONE] = 1.0;
    gicp_pose(st, P);
}

// All iterations as one cooperative kernel. An iteration: every CTA finds its
// source points' nearest target points and writes one partial; a grid barrier;
// then every CTA sums the partials and takes the step for itself (the same
// arithmetic, so the same T), and all stop at the same iteration.
__global__ void __launch_bounds__(GB) k_gicp(const GicpArgs A) {
    __shared__ float red[GB / 32][NPART];
    __shared__ double part_s[GB / 32][NPART], S[NPART], st[ST_N], M[6][7], T[27];
    __shared__ GicpPose P;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int ns = A.n_src, nt = A.n_tgt;
    if (threadIdx.x < ST_N) st[threadIdx.x] = A.state[threadIdx.x];
    __syncthreads();
    // the target tiles' boxes
    const int ntile = (nt + GTILE - 1) / GTILE;
    for (int t = blockIdx.x * (GB / 32) + w; t < ntile; t += gridDim.x * (GB / 32)) {
        float lo[3], hi[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const int j0 = t * GTILE + lane, j1 = j0 + 32;
            const bool in0 = j0 < nt && gicp_valid(A.tgt, j0), in1 = j1 < nt && gicp_valid(A.tgt, j1);
            const float u = in0 ? gicp_word(A.tgt, j0, a) : 0.f, v = in1 ? gicp_word(A.tgt, j1, a) : 0.f;
            lo[a] = fminf(in0 ? u : INFINITY, in1 ? v : INFINITY);
            hi[a] = fmaxf(in0 ? u : -INFINITY, in1 ? v : -INFINITY);   // (none: no point is near the box)
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                lo[a] = fminf(lo[a], __shfl_xor_sync(0xffffffffu, lo[a], o));
                hi[a] = fmaxf(hi[a], __shfl_xor_sync(0xffffffffu, hi[a], o));
            }
        }
        if (lane == 0)
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                A.box[6 * t + a] = lo[a];
                A.box[6 * t + 3 + a] = hi[a];
            }
    }
    unsigned target = 0;
    auto sync = [&] {
        const bool ok = grid_sync(A.bar, target, gridDim.x, A.budget);
        if (!ok && threadIdx.x == 0) atomicOr(A.err, MP_ERR_WAIT);
        return ok;
    };
    if (w == 0) {
        const double qs = st[ST_Q + (lane & 3)];
        double n2 = qs * qs;
        n2 += __shfl_xor_sync(0xffffffffu, n2, 1);
        n2 += __shfl_xor_sync(0xffffffffu, n2, 2);
        if (lane < 4) P.qn[lane] = qs / sqrt(n2);
        gicp_pose(st, P);
    }
    if (!sync()) return;
    for (int it = 0; it < A.max_iters; ++it) {
        float R[9];
        const float t[3] = {P.t32[0], P.t32[1], P.t32[2]};
        quat_rot_exact(Quat{P.q32[0], P.q32[1], P.q32[2], P.q32[3]}, R);
        float acc[NPART];
#pragma unroll
        for (int a = 0; a < NPART; ++a) acc[a] = 0.f;
        for (int k0 = blockIdx.x * GPTS; k0 < ns; k0 += gridDim.x * GPTS) {
            const int k = k0 + threadIdx.x / GPARTS;
            const bool have = k < ns && gicp_valid(A.src, k);
            // transformed source point by the decision sequence
            const int kk = min(k, ns - 1);
            const float m[3] = {gicp_word(A.src, kk, 0), gicp_word(A.src, kk, 1), gicp_word(A.src, kk, 2)};
            float qt[3], q[3];
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                qt[a] = __fmaf_rn(R[3 * a + 2], m[2], __fmaf_rn(R[3 * a + 1], m[1], __fmul_rn(R[3 * a], m[0])));
                q[a] = __fadd_rn(qt[a], t[a]);
            }
            int j = it > 0 && have ? A.corr[k] : -1;
            gicp_nearest(A, nt, have, q, j);
            __syncwarp();
            if (have && threadIdx.x % GPARTS == 0) {
                A.corr[k] = j;
                if (j >= 0 && MP_DCHECK(j < nt, "correspondence", j)) gicp_terms(A, R, qt, q, k, j, acc);
            }
        }
#pragma unroll
        for (int a = 0; a < 28; ++a) {
            const float v = warp_sum(acc[a]);
            if (lane == 0) red[w][a] = v;
        }
        __syncthreads();
        float* partial = A.partial + (size_t)(it & 1) * gridDim.x * NPART;
        if (threadIdx.x < NPART) {
            float v = 0.f;
            if (threadIdx.x < 28)
                for (int q = 0; q < GB / 32; ++q) v += red[q][threadIdx.x];
            partial[blockIdx.x * NPART + threadIdx.x] = v;
        }
        if (!sync()) return;
        gicp_sum(partial, gridDim.x, part_s, S);
        if (w == 0) gicp_step(S, T, M, st, P, A.lambda, A.eps, A.tol);
        __syncthreads();
        if (st[ST_DONE] != 0.0) break;
    }
    if (blockIdx.x == 0 && threadIdx.x < ST_N) A.state[threadIdx.x] = st[threadIdx.x];
}

template <typename T>
cudaError_t galloc(T** p, size_t count) {
    return cudaMalloc(reinterpret_cast<void**>(p), sizeof(T) * (count > 0 ? count : 1));
}

int gicp_alloc(mp_ctx* c) {
    if (c->gicp) return MP_OK;
    GicpBufs* g = new GicpBufs();
    memset(g, 0, sizeof(*g));
    const int cap = c->p.max_scan;
    g->cap = cap;
    cudaError_t e = cudaSuccess;
    int left = c->fail_gicp_alloc;   // test knob: the allocation of this number fails (0: none)
    auto A = [&](auto** p, size_t n) {
        if (e == cudaSuccess) e = left > 0 && --left == 0 ? cudaErrorMemoryAllocation : galloc(p, n);
    };
    A(&g->src_raw, 3 * (size_t)cap); A(&g->tgt_raw, 3 * (size_t)cap); A(&g->tmp4, 2 * (size_t)cap);
    const size_t soa = scan_word((cap + MP_SCAN_CHUNK - 1) / MP_SCAN_CHUNK * MP_SCAN_CHUNK, 0);
    A(&g->sorted, 2 * soa); A(&g->src_soa, soa); A(&g->tgt_soa, soa); A(&g->idx, cap); A(&g->tgt_idx, cap); A(&g->counts, 3);
    A(&g->box, 6 * (size_t)((cap + GTILE - 1) / GTILE)); A(&g->corr, cap); A(&g->bar, 1);
    int dev = 0, sms = 0, per = 0;
    if (e == cudaSuccess) e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_gicp, GB, 0);
    g->grid = sms * std::min(per, 1);
    A(&g->partial, 2 * (size_t)NPART * std::max(g->grid, 1));
    A(&g->state, ST_N); A(&g->prev, 3 * (size_t)cap);
    c->gicp = g;
    if (e == cudaSuccess && g->grid >= 1) return MP_OK;
    mp_gicp_free(c);   // so that another call allocates again
    if (e != cudaSuccess) return mp_cuda_check(c, e, "GICP buffers");
    return mp_fail(c, MP_ECUDA, "GICP: no resident CTAs for the cooperative launch");
}

// 6x6 SPD inverse on the host (Gauss-Jordan, FP64); false if singular
bool inv6(const double H[36], double I[36]) {
    double M[6][12];
    for (int r = 0; r < 6; ++r)
        for (int c = 0; c < 12; ++c) M[r][c] = c < 6 ? H[6 * r + c] : (c - 6 == r ? 1.0 : 0.0);
    for (int c = 0; c < 6; ++c) {
        int piv = c;
        for (int r = c + 1; r < 6; ++r)
            if (std::fabs(M[r][c]) > std::fabs(M[piv][c])) piv = r;
        if (!(std::fabs(M[piv][c]) > 0.0)) return false;
        if (piv != c)
            for (int k = 0; k < 12; ++k) std::swap(M[c][k], M[piv][k]);
        const double d = M[c][c];
        for (int k = 0; k < 12; ++k) M[c][k] /= d;
        for (int r = 0; r < 6; ++r) {
            if (r == c) continue;
            const double f = M[r][c];
            for (int k = 0; k < 12; ++k) M[r][k] -= f * M[c][k];
        }
    }
    for (int r = 0; r < 6; ++r)
        for (int c = 0; c < 6; ++c) I[6 * r + c] = M[r][6 + c];
    return true;
}

}  // namespace

void mp_gicp_free(mp_ctx* c) {
    GicpBufs* g = c->gicp;
    if (!g) return;
    void* bufs[] = {g->src_raw, g->tgt_raw, g->sorted, g->src_soa, g->tgt_soa, g->idx, g->tgt_idx, g->counts, g->tmp4, g->box, g->corr, g->bar, g->partial, g->state, g->prev};
    for (void* p : bufs)
        if (p) cudaFree(p);
    delete g;
    c->gicp = nullptr;
}

extern "C" {

int mp_gicp(mp_ctx* c, const float* src, int32_t n_src, const float* tgt, int32_t n_tgt, const double init_T[16],
            int32_t max_iters, double T_out[16], double cov_out[36], int32_t* n_corr, int32_t* iters) {
    if (!c) return MP_EINVAL;
    if (n_src < 1 || n_tgt < 1 || n_src > c->p.max_scan || n_tgt > c->p.max_scan || !src || !tgt || !T_out ||
        max_iters < 1)
        return mp_fail(c, MP_EINVAL, "mp_gicp: scans of 1..max_scan points, T_out and max_iters >= 1 required");
    int rc;
    if ((rc = gicp_alloc(c))) return rc;
    GicpBufs* g = c->gicp;
    MP_CUDA(c, cudaMemcpyAsync(g->src_raw, src, sizeof(float) * 3 * (size_t)n_src, cudaMemcpyDefault, c->stream));
    MP_CUDA(c, cudaMemcpyAsync(g->tgt_raw, tgt, sizeof(float) * 3 * (size_t)n_tgt, cudaMemcpyDefault, c->stream));
    float* sorted = g->sorted + scan_word((g->cap + MP_SCAN_CHUNK - 1) / MP_SCAN_CHUNK * MP_SCAN_CHUNK, 0);
    const PointScan scans[2] = {
        {g->src_raw, n_src, g->tmp4, g->sorted, g->src_soa, g->idx, g->counts},
        {g->tgt_raw, n_tgt, g->tmp4 + g->cap, sorted, g->tgt_soa, g->tgt_idx, g->counts + 1}};
    if ((rc = mp_launch_point_gaussians(c, scans, 2))) return rc;
    // initial state from init_T (identity when NULL)
    double st[ST_N];
    memset(st, 0, sizeof(st));
    double q[4], t[3];
    odom_to_pose_host(init_T, q, t);
    for (int k = 0; k < 4; ++k) st[ST_Q + k] = q[k];
    for (int k = 0; k < 3; ++k) st[ST_T + k] = t[k];
    MP_CUDA(c, cudaMemcpyAsync(g->state, st, sizeof(st), cudaMemcpyHostToDevice, c->stream));
    const float a = 1.f - c->p.eps_cov;
    GicpArgs A = {};
    A.src = g->src_soa;
    A.tgt = g->tgt_soa;
    A.tgt_idx = g->tgt_idx;
    A.n_src = n_src;
    A.n_tgt = n_tgt;
    A.box = g->box;
    A.corr = g->corr;
    A.state = g->state;
    A.partial = g->partial;
    A.r2 = c->p.r_max * c->p.r_max;
    A.half_a = 0.5f * a;
    A.two_eps = 2.f * c->p.eps_cov;
    A.quarter_a = 0.25f * a;
    A.lambda = (double)c->p.lambda;
    A.eps = (double)c->p.eps;
    A.tol = 1e-6;
    A.max_iters = max_iters;
    A.bar = g->bar;
    A.err = g->counts + 2;
    A.budget = c->wait_budget > 0 ? c->wait_budget : MP_WAIT_BUDGET;
    MP_CUDA(c, grid_bar_reset(g->bar, c->starve_bar, c->stream));
    MP_CUDA(c, cudaMemsetAsync(A.err, 0, sizeof(int32_t), c->stream));
    MP_CUDA(c, launch_coop((const void*)k_gicp, (unsigned)std::min(g->grid, (n_src + GPTS - 1) / GPTS), GB, &A, c->stream));
    MP_LAUNCHED(c);
    int32_t err = 0;
    MP_CUDA(c, cudaMemcpyAsync(&err, A.err, sizeof(err), cudaMemcpyDeviceToHost, c->stream));
    MP_CUDA(c, cudaMemcpyAsync(st, g->state, sizeof(st), cudaMemcpyDeviceToHost, c->stream));
    MP_CUDA(c, cudaStreamSynchronize(c->stream));
    if (err) return mp_fail(c, MP_ETIMEOUT, "a bounded device-side wait gave up (error bits 0x%x)", err);
    double R[9];
    const double nq = std::sqrt(st[0] * st[0] + st[1] * st[1] + st[2] * st[2] + st[3] * st[3]);
    const double x = st[0] / nq, y = st[1] / nq, z = st[2] / nq, w = st[3] / nq;
    R[0] = 1 - 2 * (y * y + z * z); R[1] = 2 * (x * y - w * z); R[2] = 2 * (x * z + w * y);
    R[3] = 2 * (x * y + w * z); R[4] = 1 - 2 * (x * x + z * z); R[5] = 2 * (y * z - w * x);
    R[6] = 2 * (x * z - w * y); R[7] = 2 * (y * z + w * x); R[8] = 1 - 2 * (x * x + y * y);
    for (int r = 0; r < 3; ++r) {
        for (int k = 0; k < 3; ++k) T_out[4 * r + k] = R[3 * r + k];
        T_out[4 * r + 3] = st[ST_T + r];
    }
    T_out[12] = T_out[13] = T_out[14] = 0.0;
    T_out[15] = 1.0;
    if (n_corr) *n_corr = (int32_t)st[ST_NC];
    if (iters) *iters = (int32_t)st[ST_IT];
    if (st[ST_DONE] == 2.0) return mp_fail(c, MP_EINVAL, "mp_gicp: fewer than 6 correspondences or a singular system");
    if (cov_out) {
        double Hm[36];
        int o = 0;
        for (int r = 0; r < 6; ++r)
            for (int k = r; k < 6; ++k) {
                Hm[6 * r + k] = st[ST_H + o];
                Hm[6 * k + r] = st[ST_H + o];
                ++o;
            }
        if (!inv6(Hm, cov_out)) return mp_fail(c, MP_EINVAL, "mp_gicp: singular Hessian");
    }
    return MP_OK;
}

int mp_step_gicp(mp_ctx* c, const float* scan, int32_t n_scan, double cov_scale) {
    if (!c) return MP_EINVAL;
    if (c->n == 0) return mp_fail(c, MP_ENOTINIT, "particles not initialised");
    if (n_scan < 0 || n_scan > c->p.max_scan || (n_scan > 0 && !scan) || !(cov_scale >= 0.0))
        return mp_fail(c, MP_EINVAL, "mp_step_gicp: bad scan or cov_scale");
    int rc;
    if ((rc = gicp_alloc(c))) return rc;
    GicpBufs* g = c->gicp;
    if (n_scan == 0) {
        // blackout: no motion estimate; the next scan starts a new sequence
        g->n_prev = 0;
        g->have_last = 0;
        return mp_step(c, nullptr, 0, nullptr, nullptr);
    }
    double T[16], cov[36];
    if (g->n_prev > 0) {
        // constant-velocity start: the previous motion
        rc = mp_gicp(c, scan, n_scan, g->prev, g->n_prev, g->have_last ? g->last_T : nullptr, 30, T, cov, nullptr,
                     nullptr);
        if (rc) return rc;
        for (int k = 0; k < 36; ++k) cov[k] *= cov_scale;
        memcpy(g->last_T, T, sizeof(T));
        g->have_last = 1;
        if ((rc = mp_step(c, scan, n_scan, T, cov))) return rc;
    } else {
        if ((rc = mp_step(c, scan, n_scan, nullptr, nullptr))) return rc;
    }
    MP_CUDA(c, cudaMemcpyAsync(g->prev, scan, sizeof(float) * 3 * (size_t)n_scan, cudaMemcpyDefault, c->stream));
    g->n_prev = n_scan;
    return MP_OK;
}

}  // extern "C"
