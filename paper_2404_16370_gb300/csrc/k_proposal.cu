// Learned proposal: box-room sensor simulator, PointNet-style mixture network
// (forward, backward, Adam) and mixture sampling. The C ABI and the network's
// definition are in include/mp_proposal.h.
//
// Layout: activations row-major [rows][channels] in FP32, rows = batch x
// points for the shared per-point layers and = batch for the head. The FP32
// form's per-point layers are tiled products (k_gemm) and a max over points, the
// BF16 form's one tensor-core kernel (k_pn_tc.cu). The head's products are
// k_head's, and the backward pass through the per-point layers runs on the
// max-pooled rows only, in one kernel (k_pool_back).
#include "mp_internal.cuh"
#include "../../include/mp_proposal.h"

#include <cuda_bf16.h>

#include <algorithm>
#include <cstdio>

#define MP_STREAM_SIM 4u
#define MP_STREAM_PN_INIT 5u
#define MP_STREAM_PN_SAMPLE 6u

namespace {

constexpr int C1 = 64, C2 = 128, C3 = 256, C4 = 256;
constexpr int NOUT = MP_PN_OUT, NCOMP = MP_PN_COMPONENTS;
constexpr float LOGSTD_LIM = 3.f;

// offsets of the parameter blocks in the flat array
constexpr int64_t OW1 = 0, OB1 = OW1 + 3 * C1, OW2 = OB1 + C1, OB2 = OW2 + (int64_t)C1 * C2, OW3 = OB2 + C2,
                  OB3 = OW3 + (int64_t)C2 * C3, OW4 = OB3 + C3, OB4 = OW4 + (int64_t)C3 * C4, OW5 = OB4 + C4,
                  OB5 = OW5 + (int64_t)C4 * NOUT, NPARAM = OB5 + NOUT;

__device__ __forceinline__ float2 normal2(uint32_t a, uint32_t b) {
    const float rad = sqrtf(-2.f * logf(u32_to_open01(a)));
    float s, c;
    sincospif(2.f * u32_to_open01(b), &s, &c);
    return make_float2(rad * c, rad * s);
}

// ---------------------------------------------------------------------------
// sensor simulator
__global__ void k_sim_box_room(const float* __restrict__ boxes, int n_boxes, float half, float height,
                               const float* __restrict__ poses, int64_t B, const float* __restrict__ dirs, int P,
                               float noise, uint2 key, float* __restrict__ out) {
    const int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (idx >= B * P) return;
    const int64_t b = idx / P;
    const int r = (int)(idx % P);
    const float* pz = poses + b * 7;
    Quat q{pz[0], pz[1], pz[2], pz[3]};
    q = qnormalize(q);
    float R[9];
    quat_rot(q, R);
    const float dx = dirs[3 * r], dy = dirs[3 * r + 1], dz = dirs[3 * r + 2];
    const float ox = pz[4], oy = pz[5], oz = pz[6];
    const float wx = R[0] * dx + R[1] * dy + R[2] * dz;
    const float wy = R[3] * dx + R[4] * dy + R[5] * dz;
    const float wz = R[6] * dx + R[7] * dy + R[8] * dz;
    // room interior: the nearest wall ahead on each axis
    auto wall = [](float o, float d, float lo, float hi) {
        return d > 0.f ? (hi - o) / d : (d < 0.f ? (lo - o) / d : INFINITY);
    };
    float t = fminf(fminf(wall(ox, wx, -half, half), wall(oy, wy, -half, half)), wall(oz, wz, 0.f, height));
    // yawed boxes: slab test in each box's frame, hits in front of the origin
    for (int k = 0; k < n_boxes; ++k) {
        const float* bx = boxes + 7 * k;
        float sn, cs;
        sincosf(-bx[6], &sn, &cs);
        const float lx = ox - bx[0], ly = oy - bx[1];
        const float o3[3] = {cs * lx - sn * ly, sn * lx + cs * ly, oz};
        const float d3[3] = {cs * wx - sn * wy, sn * wx + cs * wy, wz};
        const float lo3[3] = {-0.5f * bx[3], -0.5f * bx[4], bx[2]};
        const float hi3[3] = {0.5f * bx[3], 0.5f * bx[4], bx[2] + bx[5]};
        float tmin = -INFINITY, tmax = INFINITY;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            if (d3[a] != 0.f) {
                const float inv = 1.f / d3[a];
                const float t1 = (lo3[a] - o3[a]) * inv, t2 = (hi3[a] - o3[a]) * inv;
                tmin = fmaxf(tmin, fminf(t1, t2));
                tmax = fminf(tmax, fmaxf(t1, t2));
            } else if (o3[a] < lo3[a] || o3[a] > hi3[a]) {
                tmin = INFINITY;   // parallel to the slab and outside it
            }
        }
        if (tmax >= tmin && tmin > 1e-6f && tmin < t) t = tmin;
    }
    const uint4 u = philox4x32_10(make_uint4((uint32_t)r, (uint32_t)b, (uint32_t)(b >> 32), MP_STREAM_SIM), key);
    const float rng = t + noise * normal2(u.x, u.y).x;
    float* o = out + 3 * idx;
    o[0] = dx * rng;
    o[1] = dy * rng;
    o[2] = dz * rng;
}

// ---------------------------------------------------------------------------
// per-point layers of the FP32 form: C[M x N] = relu(A[M x K] B[K x N] + bias)
constexpr int GT = 64, GK = 16;

__global__ void __launch_bounds__(256) k_gemm(const float* __restrict__ A, const float* __restrict__ B,
                                              float* __restrict__ C, const float* __restrict__ bias, int M, int N,
                                              int K) {
    __shared__ float As[GK][GT + 4];
    __shared__ float Bs[GK][GT + 4];
    const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
    const int m0 = blockIdx.y * GT, n0 = blockIdx.x * GT;
    float acc[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
    for (int k0 = 0; k0 < K; k0 += GK) {
        for (int e = threadIdx.x; e < GT * GK; e += 256) {
            const int m = m0 + e / GK, k = k0 + e % GK;
            As[e % GK][e / GK] = m < M && k < K ? A[(int64_t)m * K + k] : 0.f;
        }
        for (int e = threadIdx.x; e < GT * GK; e += 256) {
            const int n = n0 + e % GT, k = k0 + e / GT;
            Bs[e / GT][e % GT] = n < N && k < K ? B[(int64_t)k * N + n] : 0.f;
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < GK; ++kk) {
            float a[4], b[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) a[i] = As[kk][ty * 4 + i];
#pragma unroll
            for (int j = 0; j < 4; ++j) b[j] = Bs[kk][tx * 4 + j];
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int m = m0 + ty * 4 + i;
        if (m >= M) continue;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int n = n0 + tx * 4 + j;
            if (n < N) C[(int64_t)m * N + n] = fmaxf(acc[i][j] + bias[n], 0.f);
        }
    }
}

// The head's products, C[M x N] = op(A)[M x K] op(B)[K x N] with M, N or K the
// batch: few rows, so what counts is latency and CTAs. A CTA of 128 threads takes
// 16 x 32 outputs (4 a thread) and stages 128 of K at a time, whole slices in
// flight at once. A 64 x 64 tile with 16 of K a step left 7 CTAs waiting for 16
// loads in a row: 46 us for 4 x 416 x 256, 7 now, of which 3 pass under the kernel before
// (head); the six products and four column sums and gates of a training step at
// batch 128 320 us, 36 now.
// N and the extents along which op(A) and op(B) are contiguous are multiples of
// 4, the matrices 16-byte aligned. Each output is one chain of fmaf over k.
enum : int { HEAD_BIAS = 1, HEAD_RELU = 2, HEAD_GATE = 4, HEAD_COLSUM = 8 };
constexpr int HM = 16, HN = 32, HK = 128;

// aux: the bias [N] (HEAD_BIAS), or a matrix like C whose entries <= 0 zero the
// output's (HEAD_GATE). colsum: column sums of op(B) (HEAD_COLSUM).
struct HeadArgs {
    const float *A, *B;
    float* C;
    const float* aux;
    float* colsum;
    int M, N, K, lda, ldb, ldc;
};
struct HeadSmem {
    __align__(16) float As[HM][HK + 4];
    __align__(16) float Bs[HK][HN + 4];
};

// PDL: op(B) is a weight matrix, which the kernels just before do not write: its
// first slice is asked for before the wait for them.
template <bool TA, bool TB, int EPI, bool PDL = false>
__device__ __forceinline__ void head_tile(const HeadArgs& H, HeadSmem& S, int bx, int by) {
    const float* __restrict__ A = H.A;
    const float* __restrict__ B = H.B;
    const float* __restrict__ aux = H.aux;
    float* __restrict__ C = H.C;
    float* __restrict__ colsum = H.colsum;
    const int M = H.M, N = H.N, K = H.K, lda = H.lda, ldb = H.ldb, ldc = H.ldc;
    auto& As = S.As;
    auto& Bs = S.Bs;
    const int tid = threadIdx.x, tx = tid % 8, ty = tid / 8;
    const int m0 = by * HM, n0 = bx * HN;
    float acc[4] = {0.f, 0.f, 0.f, 0.f}, col = 0.f;
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
    float4 ra[HM * HK / 512], rb[HN * HK / 512];
    auto load_a = [&](int k0) {
#pragma unroll
        for (int e = 0; e < HM * HK / 512; ++e) {
            const int v = e * 128 + tid;
            if (TA) {   // A is [K][M]: 4 of m a thread, k along the lanes
                const int k = k0 + v % HK, m = m0 + v / HK * 4;
                ra[e] = k < K && m < M ? *reinterpret_cast<const float4*>(A + (int64_t)k * lda + m) : zero;
            } else {
                const int m = m0 + v / (HK / 4), k = k0 + v % (HK / 4) * 4;
                ra[e] = k < K && m < M ? *reinterpret_cast<const float4*>(A + (int64_t)m * lda + k) : zero;
            }
        }
    };
    auto load_b = [&](int k0) {
#pragma unroll
        for (int e = 0; e < HN * HK / 512; ++e) {
            const int v = e * 128 + tid;
            if (TB) {   // B is [N][K]: 4 of k a thread, n along the lanes
                const int n = n0 + v % HN, k = k0 + v / HN * 4;
                rb[e] = k < K && n < N ? *reinterpret_cast<const float4*>(B + (int64_t)n * ldb + k) : zero;
            } else {
                const int k = k0 + v / (HN / 4), n = n0 + v % (HN / 4) * 4;
                rb[e] = k < K && n < N ? *reinterpret_cast<const float4*>(B + (int64_t)k * ldb + n) : zero;
            }
        }
    };
    load_b(0);
    if (PDL) {
        pdl_wait();
        pdl_trigger();
    }
    load_a(0);
    for (int k0 = 0; k0 < K; k0 += HK) {
        __syncthreads();
#pragma unroll
        for (int e = 0; e < HM * HK / 512; ++e) {
            const int v = e * 128 + tid;
            if (TA) {
                const int k = v % HK, m = v / HK * 4;
                As[m][k] = ra[e].x; As[m + 1][k] = ra[e].y; As[m + 2][k] = ra[e].z; As[m + 3][k] = ra[e].w;
            } else {
                *reinterpret_cast<float4*>(&As[v / (HK / 4)][v % (HK / 4) * 4]) = ra[e];
            }
        }
#pragma unroll
        for (int e = 0; e < HN * HK / 512; ++e) {
            const int v = e * 128 + tid;
            if (TB) {
                const int n = v % HN, k = v / HN * 4;
                Bs[k][n] = rb[e].x; Bs[k + 1][n] = rb[e].y; Bs[k + 2][n] = rb[e].z; Bs[k + 3][n] = rb[e].w;
            } else {
                *reinterpret_cast<float4*>(&Bs[v / (HN / 4)][v % (HN / 4) * 4]) = rb[e];
            }
        }
        __syncthreads();
        if (k0 + HK < K) {
            load_a(k0 + HK);
            load_b(k0 + HK);
        }
        const int ke = min(HK, (K - k0 + 3) & ~3);   // beyond K both are 0
#pragma unroll 4
        for (int k = 0; k < ke; k += 4) {
            const float4 a = *reinterpret_cast<const float4*>(&As[ty][k]);
            const float av[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float4 b = *reinterpret_cast<const float4*>(&Bs[k + q][tx * 4]);
                acc[0] = fmaf(av[q], b.x, acc[0]);
                acc[1] = fmaf(av[q], b.y, acc[1]);
                acc[2] = fmaf(av[q], b.z, acc[2]);
                acc[3] = fmaf(av[q], b.w, acc[3]);
            }
        }
        if ((EPI & HEAD_COLSUM) && m0 == 0 && tid < HN) {   // (one chain over k too)
#pragma unroll 16
            for (int k = 0; k < HK; ++k) col += Bs[k][tid];
        }
    }
    if ((EPI & HEAD_COLSUM) && m0 == 0 && tid < HN && n0 + tid < N) colsum[n0 + tid] = col;
    const int m = m0 + ty, n = n0 + tx * 4;
    if (m >= M || n >= N) return;
    if (EPI & HEAD_BIAS) {
        const float4 b = *reinterpret_cast<const float4*>(aux + n);
        acc[0] += b.x; acc[1] += b.y; acc[2] += b.z; acc[3] += b.w;
    }
    if (EPI & HEAD_GATE) {
        const float4 h = *reinterpret_cast<const float4*>(aux + (int64_t)m * ldc + n);
        if (!(h.x > 0.f)) acc[0] = 0.f;
        if (!(h.y > 0.f)) acc[1] = 0.f;
        if (!(h.z > 0.f)) acc[2] = 0.f;
        if (!(h.w > 0.f)) acc[3] = 0.f;
    }
    if (EPI & HEAD_RELU)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[j] = fmaxf(acc[j], 0.f);
    *reinterpret_cast<float4*>(C + (int64_t)m * ldc + n) = make_float4(acc[0], acc[1], acc[2], acc[3]);
}

template <bool TA, bool TB, int EPI, bool PDL>
__global__ void __launch_bounds__(128) k_head(const HeadArgs H) {
    __shared__ HeadSmem S;
    head_tile<TA, TB, EPI, PDL>(H, S, blockIdx.x, blockIdx.y);
}

// A layer's two gradients in one launch: the weights' (with the bias's, column
// sums) by the first `tiles` CTAs and the input's, gated or not, by the others.
template <int EPI>
__global__ void __launch_bounds__(128) k_head_back(const HeadArgs W, const HeadArgs X, int tiles, int wx, int xx) {
    __shared__ HeadSmem S;
    const int t = blockIdx.x;
    if (t < tiles) head_tile<true, false, HEAD_COLSUM>(W, S, t % wx, t / wx);
    else head_tile<false, true, EPI>(X, S, (t - tiles) % xx, (t - tiles) / xx);
}

__global__ void k_scale_points(const float* __restrict__ x, int64_t n, float inv, float* __restrict__ y) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < n) y[i] = x[i] * inv;
}

// g[b][c] = max over points of h3[b][p][c]; index of the first maximum
__global__ void k_maxpool(const float* __restrict__ h3, int B, int P, float* __restrict__ g, int* __restrict__ gi) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    const int b = blockIdx.y;
    if (c >= C3 || b >= B) return;
    const float* base = h3 + (int64_t)b * P * C3 + c;
    float m = base[0];
    int mi = 0;
    for (int p = 1; p < P; ++p) {
        const float v = base[(int64_t)p * C3];
        if (v > m) { m = v; mi = p; }
    }
    g[b * C3 + c] = m;
    gi[b * C3 + c] = mi;
}

// Backward pass of the shared layers on the pooled rows (c, b): channel c of
// sample b reaches them through its maximum's point alone, whose x, h1 and h2 it
// reads back. Per row, with d = dg[b][c] where g > 0:
//   dW3[i][c] += d h2[i], db3[c] += d, dh2[i] = d W3[i][c] where h2[i] > 0,
//   db2 += dh2, dW2[j][i] += h1[j] dh2[i], dh1[j] = sum_i dh2[i] W2[j][i] where
//   h1[j] > 0, db1 += dh1, dW1[k][j] += x[k] dh1[j].
// Resident CTAs take tiles of 64 rows in the order of c, so that a tile of a
// large batch has one column of W3; h2, dh2 and dh1 stay on chip and dW1, dW2,
// db1 and db2 in registers until the CTA is done. Bound by the FP32 products (1.1
// GFLOP at batch 128) and their shared-memory reads. As nine kernels that passed
// the rows' h1, h2, dh1 and dh2 through memory, batch 128 took 360 us; 48 now.
struct PoolArgs {
    const float *dg, *g, *x, *W2, *W3;
    const void *h1, *h2;  // FP32 rows, or the tensor-core form's BF16 operands (its values)
    const int* gi;
    float inv;            // scale of x
    int B, P;
    float *dW1, *db1, *dW2, *db2, *dW3, *db3;
};
constexpr int PR = 64, PTH = 256;                                  // rows of a tile, threads
constexpr int LD_H2 = C2 + 4, LD_H1 = C1 + 4;                      // padded rows
constexpr int POOL_SMEM = 4 * (PR * LD_H2 + PR * LD_H1 + C2 * LD_H1 + PR * 4 + 2 * PR) + 4 * PR;

template <bool BF16>
__device__ __forceinline__ float4 pool_h1(const void* h1, int64_t row, int j) {
    if (!BF16) return *reinterpret_cast<const float4*>(static_cast<const float*>(h1) + row * C1 + j);
    const uint8_t* b = static_cast<const uint8_t*>(h1) + (row >> 7) * MP_SW_BLOCK + sw128((uint32_t)row & 127u, (uint32_t)j);
    const uint2 u = __ldg(reinterpret_cast<const uint2*>(b));
    return make_float4(__uint_as_float(u.x << 16), __uint_as_float(u.x & 0xffff0000u), __uint_as_float(u.y << 16),
                       __uint_as_float(u.y & 0xffff0000u));
}
template <bool BF16>
__device__ __forceinline__ float pool_h2(const void* h2, int64_t row, int i) {
    if (!BF16) return __ldg(static_cast<const float*>(h2) + row * C2 + i);
    const uint8_t* b = static_cast<const uint8_t*>(h2) + ((row >> 7) * 2 + (i >> 6)) * (int64_t)MP_SW_BLOCK +
                       sw128((uint32_t)row & 127u, (uint32_t)i & 63u);
    return __uint_as_float((uint32_t)__ldg(reinterpret_cast<const unsigned short*>(b)) << 16);
}

template <bool BF16>
__global__ void __launch_bounds__(PTH, 2) k_pool_back(const PoolArgs A) {
    extern __shared__ __align__(16) float pool_smem[];
    float* dh2s = pool_smem;                  // [row][i]
    float* h1s = dh2s + PR * LD_H2;           // [row][j]
    float* W2s = h1s + PR * LD_H1;            // [i][j]
    float* xs = W2s + C2 * LD_H1;             // [row][x, y, z, -]
    float* ds = xs + PR * 4;                  // [row] d
    int* cs = reinterpret_cast<int*>(ds + PR);   // [row] channel
    int* ps = cs + PR;                           // [row] the point's row
    const int tid = threadIdx.x;
    for (int e = tid; e < C1 * C2; e += PTH) W2s[e % C2 * LD_H1 + e / C2] = A.W2[e];
    const int tx = tid % 16, ty = tid / 16;
    float acc2[4][8], acc1[4][4], b2 = 0.f;   // dW2[4 tx + .][..], (dW1, db1)[4 tx + .], db2 of the thread's i
#pragma unroll
    for (int j = 0; j < 4; ++j) {
#pragma unroll
        for (int i = 0; i < 8; ++i) acc2[j][i] = 0.f;
#pragma unroll
        for (int k = 0; k < 4; ++k) acc1[j][k] = 0.f;
    }
    const int rows = A.B * C3, ntile = (rows + PR - 1) / PR;
    const int i2 = tid % C2, half = tid / C2;
    for (int t = blockIdx.x; t < ntile; t += gridDim.x) {
        __syncthreads();
        if (tid < PR) {
            const int r = t * PR + tid, c = min(r, rows - 1) / A.B, b = min(r, rows - 1) % A.B;
            const float gv = A.g[b * C3 + c];
            const int point = b * A.P + A.gi[b * C3 + c];
            ds[tid] = r < rows && gv > 0.f ? A.dg[b * C3 + c] : 0.f;
            cs[tid] = c;
            ps[tid] = point;
#pragma unroll
            for (int k = 0; k < 3; ++k) xs[tid * 4 + k] = A.x[(int64_t)point * 3 + k] * A.inv;
        }
        __syncthreads();
#pragma unroll
        for (int e = 0; e < PR * C1 / 4 / PTH; ++e) {
            const int v = e * PTH + tid, r = v / (C1 / 4), j = v % (C1 / 4) * 4;
            *reinterpret_cast<float4*>(h1s + r * LD_H1 + j) =
                pool_h1<BF16>(A.h1, ps[r], j);
        }
        // h2: a thread has one i and half of the rows
        {
            int c = cs[half * (PR / 2)];
            float w = __ldg(A.W3 + i2 * C3 + c), a3 = 0.f, a3b = 0.f;
            auto flush = [&] {
                atomicAdd(A.dW3 + i2 * C3 + c, a3);
                if (i2 == 0) atomicAdd(A.db3 + c, a3b);
            };
            for (int q0 = 0; q0 < PR / 2; q0 += 8) {
                const int r0 = half * (PR / 2) + q0;
                float h[8];
#pragma unroll
                for (int q = 0; q < 8; ++q) h[q] = pool_h2<BF16>(A.h2, ps[r0 + q], i2);
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    const int r = r0 + q;
                    if (cs[r] != c) {
                        flush();
                        c = cs[r];
                        w = __ldg(A.W3 + i2 * C3 + c);
                        a3 = a3b = 0.f;
                    }
                    const float d = ds[r];
                    a3 = fmaf(d, h[q], a3);
                    a3b += d;
                    const float dh = h[q] > 0.f ? d * w : 0.f;
                    b2 += dh;
                    dh2s[r * LD_H2 + i2] = dh;
                }
            }
            flush();
        }
        __syncthreads();
        // dh1 of rows 4 ty + ., channels 4 tx + .
        float dh1[4][4];
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int j = 0; j < 4; ++j) dh1[r][j] = 0.f;
#pragma unroll 2
        for (int i = 0; i < C2; i += 4) {
            float a[4][4], w[4][4];
#pragma unroll
            for (int r = 0; r < 4; ++r)
                *reinterpret_cast<float4*>(a[r]) = *reinterpret_cast<const float4*>(dh2s + (4 * ty + r) * LD_H2 + i);
#pragma unroll
            for (int k = 0; k < 4; ++k)
                *reinterpret_cast<float4*>(w[k]) = *reinterpret_cast<const float4*>(W2s + (i + k) * LD_H1 + 4 * tx);
#pragma unroll
            for (int k = 0; k < 4; ++k)
#pragma unroll
                for (int r = 0; r < 4; ++r)
#pragma unroll
                    for (int j = 0; j < 4; ++j) dh1[r][j] = fmaf(a[r][k], w[k][j], dh1[r][j]);
        }
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const float4 h = *reinterpret_cast<const float4*>(h1s + (4 * ty + r) * LD_H1 + 4 * tx);
            const float hv[4] = {h.x, h.y, h.z, h.w};
            const float4 x = *reinterpret_cast<const float4*>(xs + (4 * ty + r) * 4);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float v = hv[j] > 0.f ? dh1[r][j] : 0.f;
                acc1[j][0] = fmaf(x.x, v, acc1[j][0]);
                acc1[j][1] = fmaf(x.y, v, acc1[j][1]);
                acc1[j][2] = fmaf(x.z, v, acc1[j][2]);
                acc1[j][3] += v;
            }
        }
        // dW2[4 tx + .][4 ty + . and 64 + 4 ty + .]
#pragma unroll 4
        for (int r = 0; r < PR; ++r) {
            float h[4], u[8];
            *reinterpret_cast<float4*>(h) = *reinterpret_cast<const float4*>(h1s + r * LD_H1 + 4 * tx);
            *reinterpret_cast<float4*>(u) = *reinterpret_cast<const float4*>(dh2s + r * LD_H2 + 4 * ty);
            *reinterpret_cast<float4*>(u + 4) = *reinterpret_cast<const float4*>(dh2s + r * LD_H2 + 64 + 4 * ty);
#pragma unroll
            for (int j = 0; j < 4; ++j)
#pragma unroll
                for (int i = 0; i < 8; ++i) acc2[j][i] = fmaf(h[j], u[i], acc2[j][i]);
        }
    }
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int q = 0; q < 2; ++q)
            atomicAdd(reinterpret_cast<float4*>(A.dW2 + (4 * tx + j) * C2 + 64 * q + 4 * ty),
                      make_float4(acc2[j][4 * q], acc2[j][4 * q + 1], acc2[j][4 * q + 2], acc2[j][4 * q + 3]));
    atomicAdd(A.db2 + i2, b2);
    // dW1 and db1: the sums over the 16 ty, through shared memory
    __syncthreads();
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int k = 0; k < 4; ++k) dh2s[(ty * 4 + k) * C1 + 4 * tx + j] = acc1[j][k];
    __syncthreads();
    const int j = tid % C1, k = tid / C1;
    float v = 0.f;
    for (int q = 0; q < 16; ++q) v += dh2s[(q * 4 + k) * C1 + j];
    atomicAdd(k < 3 ? A.dW1 + k * C1 + j : A.db1 + j, v);
}

__device__ __forceinline__ float wrap_pi(float a) {
    // into (-pi, pi]
    a = a - 6.283185307179586f * floorf(a * 0.15915494309189535f + 0.5f);
    return a <= -3.14159265358979f ? a + 6.283185307179586f : a;
}

// Mixture negative log-likelihood of each sample and its gradient w.r.t. o,
// scaled by 1/B (mean loss). A warp takes a sample, a lane a component (one
// thread a sample, components in turn: 80 us at batch 128, 4 now).
__global__ void __launch_bounds__(64) k_mdn_loss(const float* __restrict__ o, const float* __restrict__ y, int B,
                                                 float* __restrict__ dO, float* __restrict__ loss) {
    static_assert(NCOMP == 32, "a lane per component");
    const int b = blockIdx.x * 2 + (threadIdx.x >> 5), c = threadIdx.x & 31;
    if (b >= B) return;
    const float* ob = o + (int64_t)b * NOUT;
    float* db = dO + (int64_t)b * NOUT;
    auto warp_max = [](float v) {
#pragma unroll
        for (int k = 16; k > 0; k >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, k));
        return v;
    };
    // the components' sum in their order: the same bits as one thread's, and the same
    // Adam step where a gradient is nearly zero
    auto ordered_sum = [](float v) {
        float s = 0.f;
#pragma unroll
        for (int k = 0; k < NCOMP; ++k) s += __shfl_sync(0xffffffffu, v, k);
        return s;
    };
    // log pi = a - logsumexp(a)
    const float a = ob[c];
    const float amax = warp_max(a);
    const float lse_a = amax + logf(ordered_sum(expf(a - amax)));
    const float half_log_2pi6 = 3.f * 1.8378770664093453f;
    float th[6], dl[6], s = 0.f;
#pragma unroll
    for (int d = 0; d < 6; ++d) {
        th[d] = tanhf(ob[224 + 6 * c + d] / LOGSTD_LIM);
        const float ls = LOGSTD_LIM * th[d];
        dl[d] = y[b * 6 + d] - ob[32 + 6 * c + d];
        if (d == 3) dl[d] = wrap_pi(dl[d]);
        const float z = dl[d] * expf(-ls);
        s += -0.5f * z * z - ls;
    }
    const float lj = a - lse_a + s - half_log_2pi6;
    const float jmax = warp_max(lj);
    const float L = -(jmax + logf(ordered_sum(expf(lj - jmax))));
    if (c == 0) atomicAdd(loss, L / B);
    const float invB = 1.f / B;
    const float r = expf(lj + L);               // responsibility
    db[c] = (expf(a - lse_a) - r) * invB;
#pragma unroll
    for (int d = 0; d < 6; ++d) {
        const float iv = expf(-2.f * (LOGSTD_LIM * th[d]));
        db[32 + 6 * c + d] = -r * dl[d] * iv * invB;
        db[224 + 6 * c + d] = r * (1.f - dl[d] * dl[d] * iv) * (1.f - th[d] * th[d]) * invB;
    }
}

__global__ void k_adam(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m,
                       float* __restrict__ v, int64_t n, float lr, float b1, float b2, float eps, float c1, float c2) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    p[i] -= lr * (mi * c1) / (sqrtf(vi * c2) + eps);
}

// He-normal weights (std sqrt(2 / fan_in)), zero biases, last layer N(0, 0.01^2)
__global__ void k_pn_init(float* __restrict__ p, uint2 key) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= NPARAM) return;
    float std = 0.f;
    if (i < OB1) std = sqrtf(2.f / 3.f);
    else if (i >= OW2 && i < OB2) std = sqrtf(2.f / C1);
    else if (i >= OW3 && i < OB3) std = sqrtf(2.f / C2);
    else if (i >= OW4 && i < OB4) std = sqrtf(2.f / C3);
    else if (i >= OW5 && i < OB5) std = 0.01f;
    const uint4 u = philox4x32_10(make_uint4((uint32_t)i, (uint32_t)(i >> 32), 0u, MP_STREAM_PN_INIT), key);
    p[i] = std * normal2(u.x, u.y).x;
}

__global__ void k_pn_sample(const float* __restrict__ mix, int64_t n, uint2 key, const float* __restrict__ scale,
                            const float* __restrict__ offset, float* __restrict__ out) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    float amax = -INFINITY;
    for (int c = 0; c < NCOMP; ++c) amax = fmaxf(amax, mix[c]);
    float tot = 0.f;
    for (int c = 0; c < NCOMP; ++c) tot += expf(mix[c] - amax);
    const uint4 u0 = philox4x32_10(make_uint4((uint32_t)i, (uint32_t)(i >> 32), 0u, MP_STREAM_PN_SAMPLE), key);
    const uint4 u1 = philox4x32_10(make_uint4((uint32_t)i, (uint32_t)(i >> 32), 1u, MP_STREAM_PN_SAMPLE), key);
    const float pick = u32_to_open01(u0.x) * tot;
    int comp = NCOMP - 1;
    float acc = 0.f;
    for (int c = 0; c < NCOMP; ++c) {
        acc += expf(mix[c] - amax);
        if (pick < acc) { comp = c; break; }
    }
    const float2 z0 = normal2(u0.y, u0.z), z1 = normal2(u0.w, u1.x), z2 = normal2(u1.y, u1.z);
    const float z[6] = {z0.x, z0.y, z1.x, z1.y, z2.x, z2.y};
    float v[6];
#pragma unroll
    for (int d = 0; d < 6; ++d) {
        const float ls = LOGSTD_LIM * tanhf(mix[224 + 6 * comp + d] / LOGSTD_LIM);
        v[d] = (mix[32 + 6 * comp + d] + expf(ls) * z[d]) * scale[d] + offset[d];
    }
    v[3] = wrap_pi(v[3]);
    // rotation from Z-Y-X Euler angles (yaw, pitch, roll): Rz Ry Rx
    float sy, cy, sp, cp, sr, cr;
    sincosf(0.5f * v[3], &sy, &cy);
    sincosf(0.5f * v[4], &sp, &cp);
    sincosf(0.5f * v[5], &sr, &cr);
    float* o = out + 7 * i;
    o[0] = sr * cp * cy - cr * sp * sy;
    o[1] = cr * sp * cy + sr * cp * sy;
    o[2] = cr * cp * sy - sr * sp * cy;
    o[3] = cr * cp * cy + sr * sp * sy;
    o[4] = v[0];
    o[5] = v[1];
    o[6] = v[2];
}

template <typename T>
cudaError_t dmalloc(T** p, size_t count) {
    return cudaMalloc(reinterpret_cast<void**>(p), sizeof(T) * (count > 0 ? count : 1));
}

}  // namespace

struct mp_pn {
    int P, Bmax;
    float in_scale;
    float* scale;    // device [6]
    float* offset;   // device [6]
    cudaStream_t stream;
    float *param, *grad, *am, *av;
    int64_t t;       // Adam step
    float *xs, *h1, *h2, *h3, *g, *h4, *o;   // (h1, h2: the tensor-core form's BF16 operands in that form)
    int* gi;
    float *dO, *dh4, *dg;
    int pool_grid;     // resident CTAs of k_pool_back
    uint2 key;
    int prec;          // MP_PREC_BF16: per-point layers on the tensor cores; MP_PREC_FP32: CUDA cores
    uint8_t* wimg;     // BF16 image of W2^T and W3^T for the tensor-core kernel
    int32_t* err;      // device error bits of the fused kernel
};

namespace {

int pn_fail(const char* what, cudaError_t e) {
    return mp_fail_noctx(e == cudaErrorMemoryAllocation ? MP_ENOMEM : MP_ECUDA, "mp_pn: %s: %s", what,
                         cudaGetErrorString(e));
}

#define PN_CUDA(x)                                   \
    do {                                             \
        cudaError_t e_ = (x);                        \
        if (e_ != cudaSuccess) return pn_fail(#x, e_); \
    } while (0)

void gemm(cudaStream_t s, const float* A, const float* B, float* C, const float* bias, int M, int N, int K) {
    k_gemm<<<dim3((N + GT - 1) / GT, (M + GT - 1) / GT), 256, 0, s>>>(A, B, C, bias, M, N, K);
}

static_assert(OB1 % 4 == 0 && OW4 % 4 == 0 && OB4 % 4 == 0 && OW5 % 4 == 0 && OB5 % 4 == 0 && NOUT % 4 == 0,
              "head_tile's loads of four floats");
// A forward product of the head, started while the kernel before it ends.
template <int EPI>
cudaError_t head(cudaStream_t s, const float* X, const float* W, const float* bias, float* Y, int B, int K, int N) {
    const HeadArgs H = {X, W, Y, bias, nullptr, B, N, K, K, N, N};
    return launch_next(k_head<false, false, EPI, true>, dim3((N + HN - 1) / HN, (B + HM - 1) / HM), 128, 0, s, H);
}

// Gradients of Y = X W + b from dY [B x N]: dW [K x N] = X^T dY, db, and dX = dY W^T,
// with HEAD_GATE only where X > 0.
template <int EPI>
void head_back(cudaStream_t s, const float* X, const float* W, const float* dY, float* dW, float* db, float* dX, int B,
               int K, int N) {
    const HeadArgs w = {X, dY, dW, nullptr, db, K, N, B, K, N, N};
    const HeadArgs x = {dY, W, dX, X, nullptr, B, K, N, N, N, K};
    const int wx = (N + HN - 1) / HN, wt = wx * ((K + HM - 1) / HM), xx = (K + HN - 1) / HN;
    const int64_t tiles = wt + (int64_t)xx * ((B + HM - 1) / HM);
    k_head_back<EPI><<<(unsigned)tiles, 128, 0, s>>>(w, x, wt, wx, xx);
}

// BF16 image of the per-point weights, refreshed after every parameter update
int pack_weights(mp_pn* net) {
    if (net->prec != MP_PREC_BF16) return MP_OK;
    return mp_pn_tc_pack(net->param + OW2, net->param + OW3, net->wimg, net->stream);
}

// train: keep the per-point activations h1, h2 for the backward pass
int forward(mp_pn* net, const float* scans, int B, bool train) {
    cudaStream_t s = net->stream;
    const int64_t rows = (int64_t)B * net->P;
    const float* W = net->param;
    if (net->prec == MP_PREC_BF16) {
        const int rc = mp_pn_tc_forward(scans, 1.f / net->in_scale, B, net->P, W + OW1, W + OB1, W + OB2, W + OB3,
                                        net->wimg, net->g, net->gi, train ? reinterpret_cast<uint8_t*>(net->h1) : nullptr,
                                        train ? reinterpret_cast<uint8_t*>(net->h2) : nullptr, net->err, MP_WAIT_BUDGET,
                                        s);
        if (rc) return mp_fail_noctx(rc, "mp_pn: tensor-core forward launch failed");
    } else {
        k_scale_points<<<grid_for(rows * 3, 256), 256, 0, s>>>(scans, rows * 3, 1.f / net->in_scale, net->xs);
        gemm(s, net->xs, W + OW1, net->h1, W + OB1, (int)rows, C1, 3);
        gemm(s, net->h1, W + OW2, net->h2, W + OB2, (int)rows, C2, C1);
        gemm(s, net->h2, W + OW3, net->h3, W + OB3, (int)rows, C3, C2);
        k_maxpool<<<dim3(C3 / 128, B), 128, 0, s>>>(net->h3, B, net->P, net->g, net->gi);
    }
    PN_CUDA((head<HEAD_BIAS | HEAD_RELU>(s, net->g, W + OW4, W + OB4, net->h4, B, C3, C4)));
    PN_CUDA((head<HEAD_BIAS>(s, net->h4, W + OW5, W + OB5, net->o, B, C4, NOUT)));
    PN_CUDA(cudaGetLastError());
    return MP_OK;
}

}  // namespace

extern "C" {

int mp_pn_sim_box_room(const float* boxes, int n_boxes, float half, float height, const float* poses, int64_t B,
                       const float* dirs, int P, float noise, uint64_t seed, float* out, void* cuda_stream) {
    if (n_boxes < 0 || B < 0 || P < 0 || (n_boxes > 0 && !boxes) || (B * P > 0 && (!poses || !dirs || !out)))
        return mp_fail_noctx(MP_EINVAL, "mp_pn_sim_box_room: invalid argument");
    if (B * P == 0) return MP_OK;
    cudaStream_t s = (cudaStream_t)cuda_stream;
    const uint2 key = make_uint2((uint32_t)seed, (uint32_t)(seed >> 32));
    k_sim_box_room<<<grid_for(B * P, 256), 256, 0, s>>>(boxes, n_boxes, half, height, poses, B, dirs, P, noise, key,
                                                          out);
    PN_CUDA(cudaGetLastError());
    return MP_OK;
}

int mp_pn_create(mp_pn** netp, int n_points, int max_batch, float in_scale, const float scale[6],
                 const float offset[6], uint64_t seed, void* cuda_stream) {
    if (!netp || n_points < 1 || max_batch < 1 || !(in_scale > 0.f) || !scale || !offset) return mp_fail_noctx(MP_EINVAL, "mp_pn_create: invalid argument");
    if ((int64_t)n_points * max_batch * C3 >= ((int64_t)1 << 31)) return mp_fail_noctx(MP_EINVAL, "mp_pn_create: invalid argument");
    mp_pn* net = new mp_pn();
    net->P = n_points;
    net->Bmax = max_batch;
    net->in_scale = in_scale;
    net->stream = (cudaStream_t)cuda_stream;
    net->key = make_uint2((uint32_t)seed, (uint32_t)(seed >> 32));
    const int64_t rows = (int64_t)n_points * max_batch;
    cudaError_t e = cudaSuccess;
    auto A = [&](auto** p, size_t n) {
        if (e == cudaSuccess) e = dmalloc(p, n);
    };
    A(&net->scale, 6); A(&net->offset, 6);
    A(&net->param, NPARAM); A(&net->grad, NPARAM); A(&net->am, NPARAM); A(&net->av, NPARAM);
    A(&net->xs, rows * 3); A(&net->h1, rows * C1); A(&net->h2, rows * C2); A(&net->h3, rows * C3);
    A(&net->g, (size_t)max_batch * C3); A(&net->gi, (size_t)max_batch * C3); A(&net->h4, (size_t)max_batch * C4);
    A(&net->o, (size_t)max_batch * NOUT); A(&net->dO, (size_t)max_batch * NOUT);
    A(&net->dh4, (size_t)max_batch * C4); A(&net->dg, (size_t)max_batch * C3);
    A(&net->wimg, mp_pn_tc_image_bytes()); A(&net->err, 1);
    int dev = 0, sms = 0, per = 0;
    if (e == cudaSuccess) e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    for (auto k : {k_pool_back<false>, k_pool_back<true>})
        if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, POOL_SMEM);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_pool_back<false>, PTH, POOL_SMEM);
    net->pool_grid = std::max(1, sms * per);
    if (e != cudaSuccess) {
        mp_pn_destroy(net);
        return pn_fail("allocation", e);
    }
    *netp = net;
    PN_CUDA(cudaMemcpyAsync(net->scale, scale, 6 * sizeof(float), cudaMemcpyDefault, net->stream));
    PN_CUDA(cudaMemcpyAsync(net->offset, offset, 6 * sizeof(float), cudaMemcpyDefault, net->stream));
    PN_CUDA(cudaMemsetAsync(net->am, 0, sizeof(float) * NPARAM, net->stream));
    PN_CUDA(cudaMemsetAsync(net->av, 0, sizeof(float) * NPARAM, net->stream));
    PN_CUDA(cudaMemsetAsync(net->grad, 0, sizeof(float) * NPARAM, net->stream));
    PN_CUDA(cudaMemsetAsync(net->err, 0, sizeof(int32_t), net->stream));
    k_pn_init<<<grid_for(NPARAM, 256), 256, 0, net->stream>>>(net->param, net->key);
    PN_CUDA(cudaGetLastError());
    net->prec = n_points % 128 == 0 ? MP_PREC_BF16 : MP_PREC_FP32;
    if (pack_weights(net)) return pn_fail("weight image", cudaGetLastError());
    PN_CUDA(cudaStreamSynchronize(net->stream));
    return MP_OK;
}

int mp_pn_destroy(mp_pn* net) {
    if (!net) return mp_fail_noctx(MP_EINVAL, "mp_pn_destroy: invalid argument");
    void* bufs[] = {net->scale, net->offset, net->param, net->grad, net->am, net->av, net->xs, net->h1,
                    net->h2, net->h3, net->g, net->gi, net->h4, net->o, net->dO, net->dh4, net->dg, net->wimg, net->err};
    for (void* p : bufs)
        if (p) cudaFree(p);
    delete net;
    return MP_OK;
}

int mp_pn_num_params(mp_pn* net, int64_t* n) {
    if (!net || !n) return mp_fail_noctx(MP_EINVAL, "mp_pn_num_params: invalid argument");
    *n = NPARAM;
    return MP_OK;
}

int mp_pn_get_params(mp_pn* net, float* out) {
    if (!net || !out) return mp_fail_noctx(MP_EINVAL, "mp_pn_get_params: invalid argument");
    PN_CUDA(cudaMemcpyAsync(out, net->param, sizeof(float) * NPARAM, cudaMemcpyDefault, net->stream));
    PN_CUDA(cudaStreamSynchronize(net->stream));
    return MP_OK;
}

int mp_pn_set_params(mp_pn* net, const float* in) {
    if (!net || !in) return mp_fail_noctx(MP_EINVAL, "mp_pn_set_params: invalid argument");
    PN_CUDA(cudaMemcpyAsync(net->param, in, sizeof(float) * NPARAM, cudaMemcpyDefault, net->stream));
    if (pack_weights(net)) return pn_fail("weight image", cudaGetLastError());
    PN_CUDA(cudaStreamSynchronize(net->stream));
    return MP_OK;
}

int mp_pn_forward(mp_pn* net, const float* scans, int B, float* out) {
    if (!net || !scans || !out || B < 1 || B > net->Bmax) return mp_fail_noctx(MP_EINVAL, "mp_pn_forward: invalid argument");
    int rc = forward(net, scans, B, false);
    if (rc) return rc;
    PN_CUDA(cudaMemcpyAsync(out, net->o, sizeof(float) * (size_t)B * NOUT, cudaMemcpyDefault, net->stream));
    return MP_OK;
}

int mp_pn_loss_grad(mp_pn* net, const float* scans, const float* targets, int B, float* loss_dev, float* grad_out) {
    if (!net || !scans || !targets || !loss_dev || B < 1 || B > net->Bmax) return mp_fail_noctx(MP_EINVAL, "mp_pn_loss_grad: invalid argument");
    int rc = forward(net, scans, B, true);
    if (rc) return rc;
    cudaStream_t s = net->stream;
    const float* W = net->param;
    float* G = net->grad;
    PN_CUDA(cudaMemsetAsync(G, 0, sizeof(float) * NPARAM, s));
    PN_CUDA(cudaMemsetAsync(loss_dev, 0, sizeof(float), s));
    k_mdn_loss<<<grid_for(B, 2), 64, 0, s>>>(net->o, targets, B, net->dO, loss_dev);
    // head
    head_back<HEAD_GATE>(s, net->h4, W + OW5, net->dO, G + OW5, G + OB5, net->dh4, B, C4, NOUT);
    head_back<0>(s, net->g, W + OW4, net->dh4, G + OW4, G + OB4, net->dg, B, C3, C4);
    // max-pool and the shared layers, on the pooled rows (c, b) only
    PoolArgs pa = {};
    pa.dg = net->dg; pa.g = net->g; pa.gi = net->gi;
    pa.x = scans; pa.inv = 1.f / net->in_scale;
    pa.h1 = net->h1; pa.h2 = net->h2;
    pa.W2 = W + OW2; pa.W3 = W + OW3;
    pa.B = B; pa.P = net->P;
    pa.dW1 = G + OW1; pa.db1 = G + OB1; pa.dW2 = G + OW2; pa.db2 = G + OB2; pa.dW3 = G + OW3; pa.db3 = G + OB3;
    const unsigned grid = (unsigned)std::min(net->pool_grid, (B * C3 + PR - 1) / PR);
    if (net->prec == MP_PREC_BF16) k_pool_back<true><<<grid, PTH, POOL_SMEM, s>>>(pa);
    else k_pool_back<false><<<grid, PTH, POOL_SMEM, s>>>(pa);
    PN_CUDA(cudaGetLastError());
    if (grad_out) PN_CUDA(cudaMemcpyAsync(grad_out, G, sizeof(float) * NPARAM, cudaMemcpyDefault, s));
    return MP_OK;
}

int mp_pn_adam_step(mp_pn* net, float lr, float beta1, float beta2, float eps) {
    if (!net) return mp_fail_noctx(MP_EINVAL, "mp_pn_adam_step: invalid argument");
    net->t += 1;
    const float c1 = 1.f / (1.f - powf(beta1, (float)net->t));
    const float c2 = 1.f / (1.f - powf(beta2, (float)net->t));
    k_adam<<<grid_for(NPARAM, 256), 256, 0, net->stream>>>(net->param, net->grad, net->am, net->av, NPARAM, lr, beta1,
                                                           beta2, eps, c1, c2);
    PN_CUDA(cudaGetLastError());
    if (pack_weights(net)) return pn_fail("weight image", cudaGetLastError());
    return MP_OK;
}

int mp_pn_sample(mp_pn* net, const float* mix, int64_t n, uint64_t seed, float* poses_out) {
    if (!net || !mix || n < 0 || (n > 0 && !poses_out)) return mp_fail_noctx(MP_EINVAL, "mp_pn_sample: invalid argument");
    if (n == 0) return MP_OK;
    k_pn_sample<<<grid_for(n, 256), 256, 0, net->stream>>>(mix, n, make_uint2((uint32_t)seed, (uint32_t)(seed >> 32)),
                                                          net->scale, net->offset, poses_out);
    PN_CUDA(cudaGetLastError());
    return MP_OK;
}

int mp_pn_set_precision(mp_pn* net, int precision) {
    if (!net || (precision != MP_PREC_FP32 && precision != MP_PREC_BF16))
        return mp_fail_noctx(MP_EINVAL, "mp_pn_set_precision: invalid argument");
    if (precision == MP_PREC_BF16 && net->P % 128 != 0)
        return mp_fail_noctx(MP_EINVAL, "mp_pn_set_precision: the tensor-core layers take scans of a multiple of "
                                        "128 points, not %d", net->P);
    net->prec = precision;
    if (pack_weights(net)) return pn_fail("weight image", cudaGetLastError());
    return MP_OK;
}

int mp_pn_status(mp_pn* net) {
    if (!net) return mp_fail_noctx(MP_EINVAL, "mp_pn_status: invalid argument");
    int32_t e = 0;
    PN_CUDA(cudaMemcpyAsync(&e, net->err, sizeof(e), cudaMemcpyDeviceToHost, net->stream));
    PN_CUDA(cudaStreamSynchronize(net->stream));
    if (e) {
        PN_CUDA(cudaMemsetAsync(net->err, 0, sizeof(int32_t), net->stream));
        return mp_fail_noctx(MP_ETIMEOUT, "mp_pn: a bounded wait of the tensor-core forward pass gave up");
    }
    return MP_OK;
}

}  // extern "C"
