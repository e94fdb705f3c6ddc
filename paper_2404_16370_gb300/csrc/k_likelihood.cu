// Likelihood evaluation and Gauss-Newton sums (Sec. III-C, Eq. 2-4).
//
// For particle T = (R, t) and scan point k (mu_k, normal n_k):
//   q~ = R mu_k, q = q~ + t; voxel v = floor(fma(q, 1/res, -o/res)) (FP32, the
//   fixed decision sequence); m = nnf[v] (-1 outside the grid or empty);
//   e = mu^M_m - q; Omega = (Sigma^M_m + R Sigma^S_k R^T)^-1; c = e^T Omega e;
//   inlier iff m >= 0 and c <= c_max; log p -= inlier ? c : c_max;
//   inliers add J^T Omega J and J^T Omega e with J = d e / d xi (right
//   perturbation) to H and b.
//
// GB300 formulation (algebraically equal to the definition):
//  * Both covariances are GICP planes, Sigma = I - a n n^T (a = 1 - eps_cov),
//    so R Sigma^S R^T + Sigma^M = 2I - a (u u^T + w w^T) with u = R n_k,
//    w = n_m. With s = u + sg w, d = u - sg w (sg = sign(u.w)), s is orthogonal
//    to d and Omega = I/2 + a/(4 ls) s s^T + a/(4 ld) d d^T with
//    ls = 2 eps + (a/2)|d|^2, ld = 2 - (a/2)|d|^2: one reciprocal, no 3x3
//    inverse and no cancellation.
//  * J = R [ [mu]x , -I ] = [ [q~]x , -I ] diag(R, R), so the sums are taken in
//    the map frame with J~ = [ [q~]x , -I ] and rotated once per particle:
//    H = D H~ D^T, b = D b~ with D = diag(R^T, R^T).
//
// Two forms share that arithmetic, two particle-point pairs per thread on the
// packed FP32 pipe (f32x2 fma, mul and add; each half rounds exactly as the
// scalar instruction, so the decision sequences are the same in both):
//
//  * point-major (k_likelihood): a warp takes one particle, its lanes take scan
//    points, and the sums are reduced over the warp once per particle. A few
//    hundred particles fill the GPU, and a warp's neighbouring points (the scan
//    stage sorts them) read neighbouring NNF lines.
//  * particle-major (k_likelihood_pm): a thread takes two particles and walks
//    the scan, which it reads by broadcast. Fewer instructions a pair, but it
//    needs 152 SMs x 768 particles to fill the GPU, and a full last wave. With
//    fewer on a wide map a thread takes one (k_likelihood_pm1), unpacked, to the
//    same bits.
//
// lk_particle_major() chooses. What bounds both is the same: a gather of 32
// different lines that miss L1 takes 32 cycles of its SM (one line a cycle,
// measured with a random-gather loop on L2-resident data; 11 cycles when they
// hit), and a pair makes up to two (NNF entry, map record); 64 pairs are 300
// cycles of a scheduler's FMA pipe; and the sums, the pose and the pipelined
// gathers of two pairs need 139 to 168 registers, so 12 warps an SM cover the
// latency of both (issue slots 0.47 to 0.67 used, FMA pipe 54 to 60% busy, L1 data
// pipe 53 to 72%). Measured on one GB300, likelihood stage, every size
// particle-major in one pass -> this rule: 256 x 128 points 29 -> 8.2 us, 4096 x 512
// 147 -> 26.7 us, 10000 x 2048 688 -> 178 us, 16000 x 1021 in BF16 593 -> 147 us,
// 50021 x 4999 (outdoor, one particle a thread) 3.53 -> 2.07 ms; particle-major in
// parts, 2^17 x 512 426 -> 392 us, 2^17 x 8192 10.4 -> 8.2 ms, 2^18 x 8192 around
// the sensor 17.7 -> 16.7 ms; 2^20 x 8192 takes 52.5 ms either way.
#include "mp_internal.cuh"

#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <algorithm>
#include <climits>

namespace {

constexpr int LK_WARPS = 4;                      // warps of a CTA
constexpr int LK_THREADS = 32 * LK_WARPS;
constexpr int LK_MINB = 3;                       // CTAs per SM the register budget must allow (4: spills,
                                                 // 65 against 57 ms at 2^20 x 8192; 2: 67 ms)
constexpr int LK_CHUNK = MP_SCAN_CHUNK;          // scan points per stage
constexpr int LK_SEG = 6;                        // chunks a launch stages at most (1536 points: 36 KB; 512
                                                 // points a launch 65 ms, 1024 55.6, 1536 53.8)
constexpr int LK_CHUNK_BYTES = 6 * LK_CHUNK * 4;
constexpr int LK_QCAP = LK_CHUNK + 64;           // entries of a warp's queue

constexpr int64_t LK_PM_MIN = 80 << 10;          // lk_particle_major()
constexpr int LK_WIDE = 512;                     // (voxels across a map)
constexpr int64_t LK_PM1_MAX = 112 << 10;        // of a wide map: one particle per thread

constexpr int PM_THREADS = 128;                  // particle-major form: two particles per thread
constexpr int PM_PER_CTA = 2 * PM_THREADS;
constexpr int PM_CHUNK = 128;   // points per stage: 128 x 48 B = 6 KB (smaller stages leave L1 more room
                                // for the gathers: 3% faster with converged particles than 256)
constexpr int PM_MINB = 3;      // 163 registers, over parts of the scan 166
constexpr int PM1_MINB = 3;     // one particle per thread, gathers in groups of four: 139 registers
constexpr int PMH_MINB = 4;     // its 16-bit forms: their per-pair values take half the registers, so a
                                // fourth CTA (16 warps per SM) fits in 128 registers

struct LkArgs {
    const float4* poses;
    const int32_t* order;
    int64_t n;
    const float* scan;       // chunks of LK_CHUNK points, six planes each (mu, normal)
    const float4* scan_pm;   // particle-major form: 3 float4 per valid point, every value twice
    const uint4* scan_h;     // its 16-bit forms: 2 uint4 per valid point (broadcast pairs)
    const int32_t* nvalid;
    const int32_t* nnf;      // dense voxel grid of spatial-order map indices
    int nx, ny, nz;
    const float4* rec;
    float c_max;
    float* gn;
    int64_t stride;
    int32_t* err;
    unsigned long long* pairs;
    long long budget;   // cycle limit of each barrier wait
    int starve;         // test knob: announce 16 bytes more than copied for chunk 0
    int split;          // CTAs sharing the scan of one particle block (gridDim.y); > 1 adds atomically
    int seg, seg_len;   // the launch's part of the scan, of seg_len <= LK_SEG chunks (times split)
    int wpp;            // warps sharing a particle (1 or LK_WARPS)
    int rounds;         // particles per warp (or, wpp > 1, per CTA), one after the other
    int items;          // k_likelihood_pm_parts: parts of the scan at most,
    int* ticket;        // its item counter and every block's finished parts (zeroed before each launch)
    int64_t n_rec;      // map records (checked builds test the NNF entries against it)
    int scan_cap;       // scan capacity in points (checked builds test the valid count against it)
    // constants as pairs (both halves equal)
    float2 inv2, offx2, offy2, offz2, magic2, m1, half2, half_a2, nhalf_a2, two_eps2, two2, quarter_a2;
};

// ---------------------------------------------------------------------------
// Packed pair arithmetic.

__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }

// -v by its sign bits: two integer operations in place of a multiply on the FMA
// pipe, the busiest (2^18 particles around the sensor, point-major: 11.4 -> 11.0
// ms; the same for the sign of u.w or for the inlier masks gained nothing)
__device__ __forceinline__ float2 neg2(float2 v) {
    return make_float2(__uint_as_float(__float_as_uint(v.x) ^ 0x80000000u),
                       __uint_as_float(__float_as_uint(v.y) ^ 0x80000000u));
}

// The same operations on one value: a P is a pair (float2) or one (float).
__device__ __forceinline__ float fma2(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ float mul2(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float add2(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float neg2(float v) { return __uint_as_float(__float_as_uint(v) ^ 0x80000000u); }
__device__ __forceinline__ float2 add2_rd(float2 a, float2 b) { return __fadd2_rd(a, b); }
__device__ __forceinline__ float add2_rd(float a, float b) { return __fadd_rd(a, b); }
__device__ __forceinline__ float first(float2 v) { return v.x; }
__device__ __forceinline__ float first(float v) { return v; }
__device__ __forceinline__ float second(float2 v) { return v.y; }
__device__ __forceinline__ float second(float v) { return v; }
template <typename P>
__device__ __forceinline__ P pk(float a, float b) {
    if constexpr (sizeof(P) == sizeof(float2)) return make_float2(a, b);
    else return a;
}
template <typename P>
__device__ __forceinline__ P pk(float2 both) { return pk<P>(both.x, both.y); }

template <typename P>
struct LkSums {
    P Hww[6], Hwv[9], Hvv[6], bw[3], nbv[3];   // nbv = -bv
    P lc;    // sum of the inlier costs
    P cnt;   // inlier count
};
using Lk2Acc = LkSums<float2>;

// 1 / x to one ulp in one instruction (x is the product of two positive
// information-matrix scalars, of the order of 4 eps_cov to 2)
__device__ __forceinline__ float rcp1(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// One 32-byte map record (a 32-byte-aligned pair of float4, read-only in the
// kernel) in one 256-bit load: (mu.xyz, w.x) and (w.y, w.z); the last two
// words are padding.
__device__ __forceinline__ void ld_record(const float4* p, float4& r0, float2& r1) {
    float pad0, pad1;
    asm("ld.global.nc.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
        : "=f"(r0.x), "=f"(r0.y), "=f"(r0.z), "=f"(r0.w), "=f"(r1.x), "=f"(r1.y), "=f"(pad0), "=f"(pad1)
        : "l"(p));
}

// 16-bit pairs (MP_PREC_BF16 / MP_PREC_FP16): the per-pair arithmetic on bf16x2
// / half2. R mu, the normal rotation R n, the information matrix, the cost, g =
// Omega e and [q~]x Omega run in 16 bits; the decision path (q = float(R mu) +
// t, the voxel floor, the NNF), the residual mu^M - q and the lever arm q - t
// stay FP32, and the per-pair products enter the FP32 sums after conversion.
// Masking multiplies only finite values (the information-matrix scalars are
// at most a / (8 eps)); the cost of a point without a map point may overflow
// to +inf in half precision and is only compared, never multiplied.
template <typename H2> struct Half2;
template <> struct Half2<__nv_bfloat162> {
    static __device__ __forceinline__ __nv_bfloat162 from(float2 v) { return __float22bfloat162_rn(v); }
    static __device__ __forceinline__ float2 to(__nv_bfloat162 v) { return __bfloat1622float2(v); }
};
template <> struct Half2<__half2> {
    static __device__ __forceinline__ __half2 from(float2 v) { return __float22half2_rn(v); }
    static __device__ __forceinline__ float2 to(__half2 v) { return __half22float2(v); }
};
template <typename H2>
__device__ __forceinline__ H2 h2_bits(uint32_t u) {
    H2 h;
    memcpy(&h, &u, 4);
    return h;
}
template <typename H2>
__device__ __forceinline__ uint32_t h2_word(H2 h) {
    uint32_t u;
    memcpy(&u, &h, 4);
    return u;
}

// ---------------------------------------------------------------------------
// Point-major form. A CTA stages up to 1536 scan points (1-D bulk copies, TMA)
// and takes 64 particles on them, a warp one at a time; a launch covers that
// part of the scan for all particles, and the next adds to its sums. Per 256
// points a warp looks up its lanes' voxels (the loads for the next 256 are in
// flight meanwhile); the points that have a map point join a queue in shared
// memory, in scan order, so that the arithmetic runs on full warps (outdoors a
// third of a spread particle's points have none). Groups of 64 entries, two a
// lane, are accumulated; a group's records are loaded when the group before has
// read its own, and the rest of that group's arithmetic covers them.

// q~ = R mu and q = q~ + t of a pair of points, by the decision sequence (q~ =
// fma(R_a2, mz, fma(R_a1, my, R_a0 mx)), q = q~ + t).
__device__ __forceinline__ void lk_transform(const float2 R[9], const float2 t[3], const float2 m[3], float2 qt[3],
                                             float2 q[3]) {
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        qt[a] = fma2(R[3 * a + 2], m[2], fma2(R[3 * a + 1], m[1], mul2(R[3 * a], m[0])));
        q[a] = add2(qt[a], t[a]);
    }
}

// The same in 16-bit pairs: R mu (and R n, the information matrix, the cost and
// the Jacobian products) on bf16x2 / half2; q = float(R mu) + t, the residual
// and the lever arm q - t in FP32, and the products enter the FP32 sums.
template <typename H2>
__device__ __forceinline__ void lk_transform(const H2 R[9], const float2 t[3], const float2 m[3], float2 qt[3],
                                             float2 q[3]) {
    using T = Half2<H2>;
    const H2 mx = T::from(m[0]), my = T::from(m[1]), mz = T::from(m[2]);
#pragma unroll
    for (int a = 0; a < 3; ++a)
        q[a] = add2(T::to(__hfma2(R[3 * a + 2], mz, __hfma2(R[3 * a + 1], my, __hmul2(R[3 * a], mx)))), t[a]);
}

// The map index of a point's voxel (-1: none, or outside the grid).
__device__ __forceinline__ int lk_lookup(const LkArgs& A, float fx, float fy, float fz) {
    // unsigned arithmetic: an out-of-range voxel wraps to a large value
    const unsigned vx = __float_as_uint(fx) - 0x4B400000u;
    const unsigned vy = __float_as_uint(fy) - 0x4B400000u;
    const unsigned vz = __float_as_uint(fz) - 0x4B400000u;
    int m = -1;
    if (vx < (unsigned)A.nx && vy < (unsigned)A.ny && vz < (unsigned)A.nz)
        m = __ldg(A.nnf + (((int)vz * A.ny + (int)vy) * A.nx + (int)vx));
    return m;
}

// A pair of queue entries of a lane: the staged scan slot of each, and their
// map records.
struct LkEntry {
    unsigned ka, kb;
};
struct LkRec {
    float4 a0, b0;
    float2 a1, b1;
};
// What a pair keeps of its records: lever arm, residual, u + w' and u - w'.
template <typename V, typename Q = float2>
struct LkPair {
    Q qt[3];
    V e[3], s[3], d[3];
};

__device__ __forceinline__ void lk_record(const LkArgs& A, int mm, float4& r0, float2& r1) {
    if (!MP_DCHECK(mm >= 0 && mm < A.n_rec, "NNF entry beyond the map records", mm)) mm = 0;
    ld_record(A.rec + 2 * (int64_t)mm, r0, r1);
}


// The pair's residuals and normals from q, the scan normals nn and the records.
template <typename P>
__device__ __forceinline__ void lk_geometry_f(const LkArgs& A, const P R[9], const P q[3], const P nn[3], const LkRec& r,
                                              LkPair<P, P>& o) {
    const P m1 = pk<P>(A.m1);
    // residual e = mu^M - q
    o.e[0] = pk<P>(r.a0.x - first(q[0]), r.b0.x - second(q[0]));
    o.e[1] = pk<P>(r.a0.y - first(q[1]), r.b0.y - second(q[1]));
    o.e[2] = pk<P>(r.a0.z - first(q[2]), r.b0.z - second(q[2]));
    // u = R n (scan normal in the map frame), w = map normal
    const P ux = fma2(R[2], nn[2], fma2(R[1], nn[1], mul2(R[0], nn[0])));
    const P uy = fma2(R[5], nn[2], fma2(R[4], nn[1], mul2(R[3], nn[0])));
    const P uz = fma2(R[8], nn[2], fma2(R[7], nn[1], mul2(R[6], nn[0])));
    // sign of u.w as an explicit fma chain (every instantiation rounds it the
    // same way)
    const float sga = copysignf(1.f, fmaf(first(uz), r.a1.y, fmaf(first(uy), r.a1.x, first(ux) * r.a0.w)));
    const float sgb = copysignf(1.f, fmaf(second(uz), r.b1.y, fmaf(second(uy), r.b1.x, second(ux) * r.b0.w)));
    const P swx = pk<P>(sga * r.a0.w, sgb * r.b0.w);
    const P swy = pk<P>(sga * r.a1.x, sgb * r.b1.x);
    const P swz = pk<P>(sga * r.a1.y, sgb * r.b1.y);
    o.s[0] = add2(ux, swx); o.s[1] = add2(uy, swy); o.s[2] = add2(uz, swz);
    o.d[0] = fma2(m1, swx, ux); o.d[1] = fma2(m1, swy, uy); o.d[2] = fma2(m1, swz, uz);
}

__device__ __forceinline__ void lk_geometry(const LkArgs& A, const float2 R[9], const float2 q[3], const float2 nn[3],
                                            const LkRec& r, LkPair<float2>& o) {
    lk_geometry_f<float2>(A, R, q, nn, r, o);
}
__device__ __forceinline__ void lk_geometry(const LkArgs& A, const float R[9], const float q[3], const float nn[3],
                                            const LkRec& r, LkPair<float, float>& o) {
    lk_geometry_f<float>(A, R, q, nn, r, o);
}

__device__ __forceinline__ void lk_pair(const LkArgs& A, const float2 R[9], const float2 t[3], const float* scan,
                                        const LkEntry& E, const LkRec& r, LkPair<float2>& o) {
    float2 m[3], nn[3], q[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        m[k] = make_float2(scan[E.ka + k * LK_CHUNK], scan[E.kb + k * LK_CHUNK]);
        nn[k] = make_float2(scan[E.ka + (3 + k) * LK_CHUNK], scan[E.kb + (3 + k) * LK_CHUNK]);
    }
    lk_transform(R, t, m, o.qt, q);   // q~ = R mu (the lever arm) and q = q~ + t, as in the lookup
    lk_geometry(A, R, q, nn, r, o);
}

// va, vb: whether the pair's points count at all.
template <typename P>
__device__ __forceinline__ void lk_accumulate_f(const LkArgs& A, LkSums<P>& S, const LkPair<P, P>& o, bool va, bool vb) {
    const P half2 = pk<P>(A.half2), half_a2 = pk<P>(A.half_a2), nhalf_a2 = pk<P>(A.nhalf_a2), two_eps2 = pk<P>(A.two_eps2);
    const P two2 = pk<P>(A.two2), quarter_a2 = pk<P>(A.quarter_a2);
    const P qtx = o.qt[0], qty = o.qt[1], qtz = o.qt[2];
    const P ex = o.e[0], ey = o.e[1], ez = o.e[2];
    const P sx = o.s[0], sy = o.s[1], sz = o.s[2], dx = o.d[0], dy = o.d[1], dz = o.d[2];
    const P nqx = neg2(qtx), nqy = neg2(qty), nqz = neg2(qtz);
    // closed-form Omega = I/2 + as s s^T + ad d d^T
    const P dd = fma2(dz, dz, fma2(dy, dy, mul2(dx, dx)));
    const P ls = fma2(half_a2, dd, two_eps2);
    const P ld = fma2(nhalf_a2, dd, two2);
    const P pr = mul2(ls, ld);
    const P rr = mul2(quarter_a2, pk<P>(rcp1(first(pr)), rcp1(second(pr))));
    const P as = mul2(ld, rr), ad = mul2(ls, rr);
    const P se = fma2(sz, ez, fma2(sy, ey, mul2(sx, ex)));
    const P de = fma2(dz, ez, fma2(dy, ey, mul2(dx, ex)));
    const P ee = fma2(ez, ez, fma2(ey, ey, mul2(ex, ex)));
    const P cost = fma2(half2, ee, fma2(mul2(as, se), se, mul2(mul2(ad, de), de)));
    const bool ia = va && (first(cost) <= A.c_max);
    const bool ib = vb && (second(cost) <= A.c_max);
    const P inl = pk<P>(ia ? 1.f : 0.f, ib ? 1.f : 0.f);
    S.lc = fma2(inl, cost, S.lc);
    S.cnt = add2(S.cnt, inl);
    const P h = mul2(half2, inl), Pw = mul2(as, inl), Qw = mul2(ad, inl);
    const P Psx = mul2(Pw, sx), Psy = mul2(Pw, sy), Psz = mul2(Pw, sz);
    const P Qdx = mul2(Qw, dx), Qdy = mul2(Qw, dy), Qdz = mul2(Qw, dz);
    const P Oxx = fma2(Psx, sx, fma2(Qdx, dx, h));
    const P Oyy = fma2(Psy, sy, fma2(Qdy, dy, h));
    const P Ozz = fma2(Psz, sz, fma2(Qdz, dz, h));
    const P Oxy = fma2(Psx, sy, mul2(Qdx, dy));
    const P Oxz = fma2(Psx, sz, mul2(Qdx, dz));
    const P Oyz = fma2(Psy, sz, mul2(Qdy, dz));
    const P gx = fma2(Oxz, ez, fma2(Oxy, ey, mul2(Oxx, ex)));
    const P gy = fma2(Oyz, ez, fma2(Oyy, ey, mul2(Oxy, ex)));
    const P gz = fma2(Ozz, ez, fma2(Oyz, ey, mul2(Oxz, ex)));
    // Pm = [q~]x Omega (nq = -q~ carries the minus signs)
    const P P00 = fma2(qty, Oxz, mul2(nqz, Oxy)), P01 = fma2(qty, Oyz, mul2(nqz, Oyy)),
                 P02 = fma2(qty, Ozz, mul2(nqz, Oyz));
    const P P10 = fma2(qtz, Oxx, mul2(nqx, Oxz)), P11 = fma2(qtz, Oxy, mul2(nqx, Oyz)),
                 P12 = fma2(qtz, Oxz, mul2(nqx, Ozz));
    const P P20 = fma2(qtx, Oxy, mul2(nqy, Oxx)), P21 = fma2(qtx, Oyy, mul2(nqy, Oxy)),
                 P22 = fma2(qtx, Oyz, mul2(nqy, Oxz));
    // H~_ww += Pm [q~]x^T ; H~_wv += Pm ; H~_vv += Omega
    S.Hww[0] = fma2(qty, P02, fma2(nqz, P01, S.Hww[0]));
    S.Hww[1] = fma2(qtz, P00, fma2(nqx, P02, S.Hww[1]));
    S.Hww[2] = fma2(qtx, P01, fma2(nqy, P00, S.Hww[2]));
    S.Hww[3] = fma2(qtz, P10, fma2(nqx, P12, S.Hww[3]));
    S.Hww[4] = fma2(qtx, P11, fma2(nqy, P10, S.Hww[4]));
    S.Hww[5] = fma2(qtx, P21, fma2(nqy, P20, S.Hww[5]));
    S.Hwv[0] = add2(S.Hwv[0], P00); S.Hwv[1] = add2(S.Hwv[1], P01); S.Hwv[2] = add2(S.Hwv[2], P02);
    S.Hwv[3] = add2(S.Hwv[3], P10); S.Hwv[4] = add2(S.Hwv[4], P11); S.Hwv[5] = add2(S.Hwv[5], P12);
    S.Hwv[6] = add2(S.Hwv[6], P20); S.Hwv[7] = add2(S.Hwv[7], P21); S.Hwv[8] = add2(S.Hwv[8], P22);
    S.Hvv[0] = add2(S.Hvv[0], Oxx); S.Hvv[1] = add2(S.Hvv[1], Oxy); S.Hvv[2] = add2(S.Hvv[2], Oxz);
    S.Hvv[3] = add2(S.Hvv[3], Oyy); S.Hvv[4] = add2(S.Hvv[4], Oyz); S.Hvv[5] = add2(S.Hvv[5], Ozz);
    // b~ = [ g x q~ ; -g ]
    S.bw[0] = fma2(gy, qtz, fma2(gz, nqy, S.bw[0]));
    S.bw[1] = fma2(gz, qtx, fma2(gx, nqz, S.bw[1]));
    S.bw[2] = fma2(gx, qty, fma2(gy, nqx, S.bw[2]));
    S.nbv[0] = add2(S.nbv[0], gx); S.nbv[1] = add2(S.nbv[1], gy); S.nbv[2] = add2(S.nbv[2], gz);
}

__device__ __forceinline__ void lk_accumulate(const LkArgs& A, Lk2Acc& S, const LkPair<float2>& o, bool va, bool vb) {
    lk_accumulate_f<float2>(A, S, o, va, vb);
}
__device__ __forceinline__ void lk_accumulate(const LkArgs& A, LkSums<float>& S, const LkPair<float, float>& o, bool va,
                                              bool vb) {
    lk_accumulate_f<float>(A, S, o, va, vb);
}

template <typename H2>
__device__ __forceinline__ void lk_geometry(const LkArgs& A, const H2 R[9], const float2 q[3], const H2 nn[3],
                                            const LkRec& r, LkPair<H2>& o) {
    using T = Half2<H2>;
    o.e[0] = T::from(make_float2(r.a0.x - q[0].x, r.b0.x - q[0].y));
    o.e[1] = T::from(make_float2(r.a0.y - q[1].x, r.b0.y - q[1].y));
    o.e[2] = T::from(make_float2(r.a0.z - q[2].x, r.b0.z - q[2].y));
    const H2 nx = nn[0], ny = nn[1], nz = nn[2];
    // u = R n, w = map normal
    const H2 ux = __hfma2(R[2], nz, __hfma2(R[1], ny, __hmul2(R[0], nx)));
    const H2 uy = __hfma2(R[5], nz, __hfma2(R[4], ny, __hmul2(R[3], nx)));
    const H2 uz = __hfma2(R[8], nz, __hfma2(R[7], ny, __hmul2(R[6], nx)));
    const H2 wx = T::from(make_float2(r.a0.w, r.b0.w)), wy = T::from(make_float2(r.a1.x, r.b1.x));
    const H2 wz = T::from(make_float2(r.a1.y, r.b1.y));
    const float2 uw = T::to(__hfma2(uz, wz, __hfma2(uy, wy, __hmul2(ux, wx))));
    const H2 sg = T::from(make_float2(copysignf(1.f, uw.x), copysignf(1.f, uw.y)));
    const H2 swx = __hmul2(sg, wx), swy = __hmul2(sg, wy), swz = __hmul2(sg, wz);
    o.s[0] = __hadd2(ux, swx); o.s[1] = __hadd2(uy, swy); o.s[2] = __hadd2(uz, swz);
    o.d[0] = __hsub2(ux, swx); o.d[1] = __hsub2(uy, swy); o.d[2] = __hsub2(uz, swz);
}

template <typename H2>
__device__ __forceinline__ void lk_pair(const LkArgs& A, const H2 R[9], const float2 t[3], const float* scan,
                                        const LkEntry& E, const LkRec& r, LkPair<H2>& o) {
    using T = Half2<H2>;
    float2 m[3], q[3];
    H2 nn[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        m[k] = make_float2(scan[E.ka + k * LK_CHUNK], scan[E.kb + k * LK_CHUNK]);
        nn[k] = T::from(make_float2(scan[E.ka + (3 + k) * LK_CHUNK], scan[E.kb + (3 + k) * LK_CHUNK]));
    }
    lk_transform(R, t, m, o.qt, q);
#pragma unroll
    for (int k = 0; k < 3; ++k) o.qt[k] = fma2(A.m1, t[k], q[k]);
    lk_geometry(A, R, q, nn, r, o);
}

template <typename H2>
__device__ __forceinline__ void lk_accumulate(const LkArgs& A, Lk2Acc& S, const LkPair<H2>& o, bool va, bool vb) {
    using T = Half2<H2>;
    const H2 half = T::from(make_float2(0.5f, 0.5f));
    const H2 half_a = T::from(A.half_a2), nhalf_a = T::from(A.nhalf_a2), two_eps = T::from(A.two_eps2);
    const H2 two = T::from(A.two2), quarter_a = T::from(A.quarter_a2);
    const float2 qtx = o.qt[0], qty = o.qt[1], qtz = o.qt[2];
    const float2 nqx = mul2(A.m1, qtx), nqy = mul2(A.m1, qty), nqz = mul2(A.m1, qtz);
    const H2 hqx = T::from(qtx), hqy = T::from(qty), hqz = T::from(qtz);
    const H2 hnx = __hneg2(hqx), hny = __hneg2(hqy), hnz = __hneg2(hqz);
    const H2 ex = o.e[0], ey = o.e[1], ez = o.e[2];
    const H2 sx = o.s[0], sy = o.s[1], sz = o.s[2], dx = o.d[0], dy = o.d[1], dz = o.d[2];
    const H2 dd = __hfma2(dz, dz, __hfma2(dy, dy, __hmul2(dx, dx)));
    const H2 ls = __hfma2(half_a, dd, two_eps);
    const H2 ld = __hfma2(nhalf_a, dd, two);
    const H2 rr = __hmul2(quarter_a, h2rcp(__hmul2(ls, ld)));
    const H2 as = __hmul2(ld, rr), ad = __hmul2(ls, rr);
    const H2 se = __hfma2(sz, ez, __hfma2(sy, ey, __hmul2(sx, ex)));
    const H2 de = __hfma2(dz, ez, __hfma2(dy, ey, __hmul2(dx, ex)));
    const H2 ee = __hfma2(ez, ez, __hfma2(ey, ey, __hmul2(ex, ex)));
    const float2 cost = T::to(__hfma2(half, ee, __hfma2(__hmul2(as, se), se, __hmul2(__hmul2(ad, de), de))));
    const bool ia = va && (cost.x <= A.c_max);
    const bool ib = vb && (cost.y <= A.c_max);
    S.lc.x += ia ? cost.x : 0.f;
    S.lc.y += ib ? cost.y : 0.f;
    S.cnt = add2(S.cnt, make_float2(ia ? 1.f : 0.f, ib ? 1.f : 0.f));
    const H2 inl = T::from(make_float2(ia ? 1.f : 0.f, ib ? 1.f : 0.f));
    const H2 h = __hmul2(half, inl), Pw = __hmul2(as, inl), Qw = __hmul2(ad, inl);
    const H2 Psx = __hmul2(Pw, sx), Psy = __hmul2(Pw, sy), Psz = __hmul2(Pw, sz);
    const H2 Qdx = __hmul2(Qw, dx), Qdy = __hmul2(Qw, dy), Qdz = __hmul2(Qw, dz);
    const H2 Oxx = __hfma2(Psx, sx, __hfma2(Qdx, dx, h));
    const H2 Oyy = __hfma2(Psy, sy, __hfma2(Qdy, dy, h));
    const H2 Ozz = __hfma2(Psz, sz, __hfma2(Qdz, dz, h));
    const H2 Oxy = __hfma2(Psx, sy, __hmul2(Qdx, dy));
    const H2 Oxz = __hfma2(Psx, sz, __hmul2(Qdx, dz));
    const H2 Oyz = __hfma2(Psy, sz, __hmul2(Qdy, dz));
    const float2 gx = T::to(__hfma2(Oxz, ez, __hfma2(Oxy, ey, __hmul2(Oxx, ex))));
    const float2 gy = T::to(__hfma2(Oyz, ez, __hfma2(Oyy, ey, __hmul2(Oxy, ex))));
    const float2 gz = T::to(__hfma2(Ozz, ez, __hfma2(Oyz, ey, __hmul2(Oxz, ex))));
    // Pm = [q~]x Omega
    const float2 P00 = T::to(__hfma2(hqy, Oxz, __hmul2(hnz, Oxy))), P01 = T::to(__hfma2(hqy, Oyz, __hmul2(hnz, Oyy))),
                 P02 = T::to(__hfma2(hqy, Ozz, __hmul2(hnz, Oyz)));
    const float2 P10 = T::to(__hfma2(hqz, Oxx, __hmul2(hnx, Oxz))), P11 = T::to(__hfma2(hqz, Oxy, __hmul2(hnx, Oyz))),
                 P12 = T::to(__hfma2(hqz, Oxz, __hmul2(hnx, Ozz)));
    const float2 P20 = T::to(__hfma2(hqx, Oxy, __hmul2(hny, Oxx))), P21 = T::to(__hfma2(hqx, Oyy, __hmul2(hny, Oxy))),
                 P22 = T::to(__hfma2(hqx, Oyz, __hmul2(hny, Oxz)));
    // FP32 sums
    S.Hww[0] = fma2(qty, P02, fma2(nqz, P01, S.Hww[0]));
    S.Hww[1] = fma2(qtz, P00, fma2(nqx, P02, S.Hww[1]));
    S.Hww[2] = fma2(qtx, P01, fma2(nqy, P00, S.Hww[2]));
    S.Hww[3] = fma2(qtz, P10, fma2(nqx, P12, S.Hww[3]));
    S.Hww[4] = fma2(qtx, P11, fma2(nqy, P10, S.Hww[4]));
    S.Hww[5] = fma2(qtx, P21, fma2(nqy, P20, S.Hww[5]));
    S.Hwv[0] = add2(S.Hwv[0], P00); S.Hwv[1] = add2(S.Hwv[1], P01); S.Hwv[2] = add2(S.Hwv[2], P02);
    S.Hwv[3] = add2(S.Hwv[3], P10); S.Hwv[4] = add2(S.Hwv[4], P11); S.Hwv[5] = add2(S.Hwv[5], P12);
    S.Hwv[6] = add2(S.Hwv[6], P20); S.Hwv[7] = add2(S.Hwv[7], P21); S.Hwv[8] = add2(S.Hwv[8], P22);
    S.Hvv[0] = add2(S.Hvv[0], T::to(Oxx)); S.Hvv[1] = add2(S.Hvv[1], T::to(Oxy)); S.Hvv[2] = add2(S.Hvv[2], T::to(Oxz));
    S.Hvv[3] = add2(S.Hvv[3], T::to(Oyy)); S.Hvv[4] = add2(S.Hvv[4], T::to(Oyz)); S.Hvv[5] = add2(S.Hvv[5], T::to(Ozz));
    S.bw[0] = fma2(gy, qtz, fma2(gz, nqy, S.bw[0]));
    S.bw[1] = fma2(gz, qtx, fma2(gx, nqz, S.bw[1]));
    S.bw[2] = fma2(gx, qty, fma2(gy, nqx, S.bw[2]));
    S.nbv[0] = add2(S.nbv[0], gx); S.nbv[1] = add2(S.nbv[1], gy); S.nbv[2] = add2(S.nbv[2], gz);
}

// Sums of a warp's lanes: lane l of the result holds the sum over the warp of
// v[l] (a transposing tree: 16 + 8 + 4 + 2 + 1 exchanges).
__device__ __forceinline__ float lk_warp_transpose_sum(float (&v)[32], int lane) {
#pragma unroll
    for (int w = 16; w >= 1; w >>= 1) {
        const bool up = (lane & w) != 0;
#pragma unroll
        for (int i = 0; i < w; ++i) {
            const float keep = up ? v[i + w] : v[i], send = up ? v[i] : v[i + w];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, w);
        }
    }
    return v[0];
}

// index of the (r, c) entry in the upper rows of a symmetric 3x3 block
__device__ __forceinline__ int sym3(int r, int c) {
    const int a = min(r, c), b = max(r, c);
    return a * 3 - (a * (a - 1)) / 2 + (b - a);
}

// v in both halves of a pair, in the pair's type.
template <typename V>
__device__ __forceinline__ V lk_pair_of(float v) { return Half2<V>::from(make_float2(v, v)); }
template <>
__device__ __forceinline__ float2 lk_pair_of<float2>(float v) { return make_float2(v, v); }

// WPP warps share a particle: 1 (every warp its own particle) or LK_WARPS
// (every fourth 64 points of the scan each). V: the type of the pairs.
template <int WPP, typename V>
struct LkOp {
    using Args = LkArgs;
    static constexpr int THREADS = LK_THREADS, MINB = LK_MINB;
    static __device__ __forceinline__ void run(const LkArgs& A, unsigned bxi, unsigned byi);
};

template <int WPP, typename V>
__device__ __forceinline__ void LkOp<WPP, V>::run(const LkArgs& A, unsigned bxi, unsigned byi) {
    constexpr int SUB = WPP == 1 ? LK_CHUNK : 64;   // points looked up at a time
    constexpr int IT = SUB / 64;
    __shared__ __align__(128) float stage[LK_SEG * 6 * LK_CHUNK];
    __shared__ __align__(8) uint2 queue[LK_WARPS][LK_QCAP];
    __shared__ float sums[LK_WARPS][32];
    __shared__ float rots[LK_WARPS][12];
    __shared__ __align__(8) uint64_t full[LK_SEG];
    __shared__ int failed_s;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const unsigned lt = (1u << lane) - 1u;

    int nv = *A.nvalid;
    if (!MP_DCHECK(nv >= 0 && nv <= A.scan_cap, "valid scan points", nv)) nv = 0;
    const int nchunks = (nv + LK_CHUNK - 1) / LK_CHUNK;
    // this CTA's chunks: cc(0), cc(1), ... (at most LK_SEG of them)
    const int split = A.split, first = A.seg * A.seg_len * split + (int)byi;
    const int nmine = first < nchunks ? min(A.seg_len, (nchunks - first + split - 1) / split) : 0;
    const int npts = nmine > 0 ? (nmine - 1) * LK_CHUNK + min(LK_CHUNK, nv - (first + (nmine - 1) * split) * LK_CHUNK) : 0;
    const int nsub = (npts + SUB - 1) / SUB;
    if (nmine == 0 && (A.seg > 0 || split > 1)) return;   // (the first segment writes its zeros)
    const int64_t p0 = (int64_t)bxi * A.rounds * (LK_WARPS / WPP);
    const int rounds = (int)min((int64_t)A.rounds, (A.n - p0 + LK_WARPS / WPP - 1) / (LK_WARPS / WPP));
    if (A.seg == 0 && bxi == 0 && byi == 0 && threadIdx.x == 0)
        atomicAdd(A.pairs, (unsigned long long)A.n * (unsigned long long)nv);
    if (threadIdx.x == 0) {
        for (int k = 0; k < LK_SEG; ++k) mbar_init(&full[k], 1);
        failed_s = 0;
        mbar_fence_init();
        for (int k = 0; k < nmine; ++k) {
            const int cc = first + k * split;
            if (!MP_DCHECK(cc >= 0 && cc < nchunks && ((reinterpret_cast<uintptr_t>(A.scan) & 15) == 0), "scan chunk", cc))
                break;
            mbar_expect_tx(&full[k], LK_CHUNK_BYTES + ((A.starve && cc == 0) ? 16u : 0u));
            bulk_g2s(stage + k * 6 * LK_CHUNK, A.scan + (int64_t)cc * 6 * LK_CHUNK, LK_CHUNK_BYTES, &full[k]);
        }
    }
    __syncthreads();

    bool failed = false;
    uint2* const Q = queue[w];
    for (int r = 0; r < rounds; ++r) {
        const int64_t p = p0 + (int64_t)r * (LK_WARPS / WPP) + (WPP == 1 ? w : 0);
        if (WPP == 1 && p >= A.n) break;
        V R[9];
        float2 t[3];
        {
            int64_t i = A.order[p];
            if (!MP_DCHECK(i >= 0 && i < A.n, "particle order entry", i)) i = 0;
            Quat q;
            float tt[3], Rs[9];
            load_pose(A.poses, i, q, tt);
            quat_rot_exact(q, Rs);
#pragma unroll
            for (int k = 0; k < 9; ++k) R[k] = lk_pair_of<V>(Rs[k]);
#pragma unroll
            for (int k = 0; k < 3; ++k) t[k] = make_float2(tt[k], tt[k]);
            __syncwarp();
            if (lane == 0) {
#pragma unroll
                for (int k = 0; k < 9; ++k) rots[w][k] = Rs[k];
            }
        }
        Lk2Acc S;
        const float2 z2 = make_float2(0.f, 0.f);
#pragma unroll
        for (int k = 0; k < 6; ++k) { S.Hww[k] = z2; S.Hvv[k] = z2; }
#pragma unroll
        for (int k = 0; k < 9; ++k) S.Hwv[k] = z2;
#pragma unroll
        for (int k = 0; k < 3; ++k) { S.bw[k] = z2; S.nbv[k] = z2; }
        S.lc = z2;
        S.cnt = z2;

        int cnt = 0;                  // queued entries
        bool pend = false;            // a group whose records are in flight
        LkEntry pe;
        LkRec pr;
        // the 64 entries at h, h + 1, ... become the pending group
        auto form = [&](int h) {
            const uint2 a = Q[h + lane], b = Q[h + 32 + lane];
            pe.ka = a.y;
            pe.kb = b.y;
            lk_record(A, (int)a.x, pr.a0, pr.a1);
            lk_record(A, (int)b.x, pr.b0, pr.b1);
            pend = true;
        };
        // the pending group's sums; `next` may form the next one once the
        // records are read, which the rest of the arithmetic then covers
        auto take = [&](auto next) {
            LkPair<V> o;
            lk_pair(A, R, t, stage, pe, pr, o);
            next();
            lk_accumulate(A, S, o, true, true);
        };
        // voxel lookups of points s * SUB + ... (their map indices, -1: none;
        // the scan's last chunk is filled with points outside every grid)
        auto lookup = [&](int s, int (&idx)[2 * IT]) {
            const int c = s * SUB / LK_CHUNK;
            if (r == 0) {   // the chunks stay staged for the later rounds
                const bool got = !failed && mbar_wait_bounded(&full[c], 0, A.budget);
                if (!__all_sync(0xffffffffu, got)) failed = true;
                if (failed) return;
            }
            const float* base = stage + c * 6 * LK_CHUNK + s * SUB % LK_CHUNK + lane;
#pragma unroll
            for (int k = 0; k < IT; ++k) {
                const float* b = base + 64 * k;
                const float2 mu[3] = {make_float2(b[0], b[32]), make_float2(b[LK_CHUNK], b[LK_CHUNK + 32]),
                                      make_float2(b[2 * LK_CHUNK], b[2 * LK_CHUNK + 32])};
                float2 qt[3], q[3];
                lk_transform(R, t, mu, qt, q);
                // voxel = floor(fma(q, 1/res, off)): round-down add of 1.5 * 2^23
                const float2 fx = __fadd2_rd(fma2(q[0], A.inv2, A.offx2), A.magic2);
                const float2 fy = __fadd2_rd(fma2(q[1], A.inv2, A.offy2), A.magic2);
                const float2 fz = __fadd2_rd(fma2(q[2], A.inv2, A.offz2), A.magic2);
                idx[2 * k] = lk_lookup(A, fx.x, fy.x, fz.x);
                idx[2 * k + 1] = lk_lookup(A, fx.y, fy.y, fz.y);
            }
        };
        int cur[2 * IT];
        const int s0 = WPP > 1 ? w : 0;
        if (s0 < nsub) lookup(s0, cur);
        for (int s = s0; s < nsub; s += WPP) {
            // the next lookups are in flight while this part is accumulated
            int nxt[2 * IT];
            if (s + WPP < nsub) lookup(s + WPP, nxt);
            if (failed) break;
            // the points that have a map point join the queue, in scan order
            const unsigned k0 = (unsigned)(s * SUB / LK_CHUNK * 6 * LK_CHUNK + s * SUB % LK_CHUNK + lane);
#pragma unroll
            for (int k = 0; k < 2 * IT; ++k) {
                const unsigned bal = __ballot_sync(0xffffffffu, cur[k] >= 0);
                if (cur[k] >= 0) Q[cnt + __popc(bal & lt)] = make_uint2((unsigned)cur[k], k0 + 32 * k);
                cnt += __popc(bal);
            }
            __syncwarp();
            int h = 0;
            while (cnt - h >= 64) {
                if (pend) take([&] { form(h); });
                else form(h);
                h += 64;
            }
            __syncwarp();
            if (h > 0) {   // the rest to the front
                const int rest = cnt - h;
                uint2 a[2];
#pragma unroll
                for (int k = 0; k < 2; ++k)
                    if (32 * k + lane < rest) a[k] = Q[h + 32 * k + lane];
                __syncwarp();
#pragma unroll
                for (int k = 0; k < 2; ++k)
                    if (32 * k + lane < rest) Q[32 * k + lane] = a[k];
                cnt = rest;
                __syncwarp();
            }
#pragma unroll
            for (int k = 0; k < 2 * IT; ++k) cur[k] = nxt[k];   // (here: the copy waits for the loads)
        }
        if (pend) take([] {});
        if (cnt > 0) {   // the last, partial group: lanes beyond it take its last entry, masked
            const uint2 a = Q[min(lane, cnt - 1)], b = Q[min(32 + lane, cnt - 1)];
            pe.ka = a.y;
            pe.kb = b.y;
            lk_record(A, (int)a.x, pr.a0, pr.a1);
            lk_record(A, (int)b.x, pr.b0, pr.b1);
            LkPair<V> o;
            lk_pair(A, R, t, stage, pe, pr, o);
            lk_accumulate(A, S, o, lane < cnt, 32 + lane < cnt);
        }
        // the 29 sums over the warp's lanes, value l in lane l
        float v[32];
#pragma unroll
        for (int k = 0; k < 6; ++k) { v[k] = S.Hww[k].x + S.Hww[k].y; v[15 + k] = S.Hvv[k].x + S.Hvv[k].y; }
#pragma unroll
        for (int k = 0; k < 9; ++k) v[6 + k] = S.Hwv[k].x + S.Hwv[k].y;
#pragma unroll
        for (int k = 0; k < 3; ++k) { v[21 + k] = S.bw[k].x + S.bw[k].y; v[24 + k] = S.nbv[k].x + S.nbv[k].y; }
        v[27] = S.lc.x + S.lc.y;
        v[28] = S.cnt.x + S.cnt.y;
        v[29] = 0.f;
        v[30] = 0.f;
        v[31] = 0.f;
        const float mine = lk_warp_transpose_sum(v, lane);
        sums[w][lane] = mine;
        if (WPP > 1) {
            __syncthreads();
            if (w == 0) {
                float tot = 0.f;
#pragma unroll
                for (int k = 0; k < WPP; ++k) tot += sums[k][lane];
                __syncwarp();
                sums[0][lane] = tot;
            }
        }
        __syncwarp();
        // rotate the map-frame sums to the sensor frame: output f in lane f
        if ((WPP == 1 || w == 0) && !failed && lane < MP_GN) {
            const float* M = sums[WPP == 1 ? w : 0];
            const float* Rr = rots[w];
            float out;
            if (lane < 21) {
                const int row = (lane >= 6) + (lane >= 11) + (lane >= 15) + (lane >= 18) + (lane >= 20);
                const int col = row + lane - (row * 6 - row * (row - 1) / 2);
                const int a = row < 3 ? row : row - 3, b = col < 3 ? col : col - 3;
                out = 0.f;
#pragma unroll
                for (int k = 0; k < 3; ++k)
#pragma unroll
                    for (int l = 0; l < 3; ++l) {
                        const int e = col < 3 ? sym3(k, l) : row < 3 ? 6 + 3 * k + l : 15 + sym3(k, l);
                        out = fmaf(Rr[3 * k + a] * Rr[3 * l + b], M[e], out);
                    }
            } else if (lane < 27) {
                const int a = lane < 24 ? lane - 21 : lane - 24, o = lane < 24 ? 21 : 24;
                const float x = fmaf(Rr[6 + a], M[o + 2], fmaf(Rr[3 + a], M[o + 1], Rr[a] * M[o]));
                out = lane < 24 ? x : -x;
            } else if (lane == 27) {
                // log p = -(sum of inlier costs) - c_max * (points that are not inliers)
                out = fmaf(-A.c_max, (float)(npts - (int)M[28]), -M[27]);
            } else {
                out = M[28];
            }
            float* dst = A.gn + (int64_t)lane * A.stride + p;
            if (split > 1) atomicAdd(dst, out);
            else *dst = A.seg > 0 ? *dst + out : out;
        }
        if (WPP > 1) __syncthreads();
    }
    if (failed) failed_s = 1;
    __syncthreads();
    if (failed_s && threadIdx.x == 0) {
        atomicOr(A.err, MP_ERR_WAIT);
        // copies still in flight end before the CTA does (bounded)
        for (int k = 0; k < nmine; ++k) mbar_wait_bounded(&full[k], 0, A.budget);
    }
}

template <int WPP, typename V>
__global__ void __launch_bounds__(LK_THREADS, LK_MINB) k_likelihood(const LkArgs A) {
    pdl_wait();
    pdl_trigger();
    LkOp<WPP, V>::run(A, blockIdx.x, blockIdx.y);
}

// ---------------------------------------------------------------------------
// Particle-major form. Every per-pair value is a float2 holding particle a in
// .x and particle b in .y. Particles are visited in the order the sort stage
// leaves for this kernel: by the cell of their position (a coarse Morton
// order), in LSH order within a cell, so that the CTAs resident at one time
// hold particles of one part of the map. A thread takes slots p and p + 128 of
// that order. The scan streams through shared memory in chunks of 128 points
// stored as broadcast pairs (48 bytes a point), double-buffered with 1-D bulk
// copies (TMA, cp.async.bulk) completing on mbarriers, and every thread of a
// warp reads the same point. The two dependent gathers of a point (NNF entry,
// then map record) are software-pipelined: the NNF entries of point k+2 and the
// records of point k+1 are in flight while point k is accumulated.
// Sums of one particle over the scan (map frame, see the file comment).
struct LkAcc {
    float Hww[6];    // (00 01 02 11 12 22)
    float Hwv[9];    // row-major
    float Hvv[6];    // (00 01 02 11 12 22)
    float bw[3], bv[3];
    float ll;
    int cnt;
};

// Rotates the map-frame sums of one particle back to the sensor frame
// (blocks M -> R^T M R, b -> R^T b) and stores the 29 outputs at sorted slot p.
__device__ __forceinline__ void lk_store(const LkArgs& A, const float R[9], const LkAcc& S, int64_t p) {
    float Hw[3][3] = {{S.Hww[0], S.Hww[1], S.Hww[2]}, {S.Hww[1], S.Hww[3], S.Hww[4]}, {S.Hww[2], S.Hww[4], S.Hww[5]}};
    float Hc[3][3] = {{S.Hwv[0], S.Hwv[1], S.Hwv[2]}, {S.Hwv[3], S.Hwv[4], S.Hwv[5]}, {S.Hwv[6], S.Hwv[7], S.Hwv[8]}};
    float Hv[3][3] = {{S.Hvv[0], S.Hvv[1], S.Hvv[2]}, {S.Hvv[1], S.Hvv[3], S.Hvv[4]}, {S.Hvv[2], S.Hvv[4], S.Hvv[5]}};
    float Ow[3][3], Oc[3][3], Ov[3][3];
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int bb = 0; bb < 3; ++bb) {
            float sw = 0.f, sc = 0.f, sv = 0.f;
#pragma unroll
            for (int k = 0; k < 3; ++k)
#pragma unroll
                for (int l = 0; l < 3; ++l) {
                    float rr = R[3 * k + a] * R[3 * l + bb];
                    sw += rr * Hw[k][l];
                    sc += rr * Hc[k][l];
                    sv += rr * Hv[k][l];
                }
            Ow[a][bb] = sw; Oc[a][bb] = sc; Ov[a][bb] = sv;
        }
    float bwr[3], bvr[3];
    rot_apply_T(R, S.bw, bwr);
    rot_apply_T(R, S.bv, bvr);
    float out[MP_GN];
    // upper rows of the 6x6 [ [Hww, Hwv], [Hwv^T, Hvv] ]
    int o = 0;
#pragma unroll
    for (int r = 0; r < 6; ++r)
#pragma unroll
        for (int cc = r; cc < 6; ++cc) {
            float v;
            if (r < 3 && cc < 3) v = Ow[r][cc];
            else if (r < 3) v = Oc[r][cc - 3];
            else v = Ov[r - 3][cc - 3];
            out[o++] = v;
        }
    out[21] = bwr[0]; out[22] = bwr[1]; out[23] = bwr[2];
    out[24] = bvr[0]; out[25] = bvr[1]; out[26] = bvr[2];
    out[27] = S.ll;
    out[28] = (float)S.cnt;
#pragma unroll
    for (int f = 0; f < MP_GN; ++f) A.gn[(int64_t)f * A.stride + p] = out[f];
}

// (P = float: particle a alone, and mb = -1)
template <typename P>
struct LkLook {
    int ma, mb;
    P qx, qy, qz;
};
using Lk2Look = LkLook<float2>;

// A staged point of the particle (pair): q alone.
template <typename P>
__device__ __forceinline__ LkLook<P> lk2_point(const P R[9], P tx, P ty, P tz, const float4* Pp) {
    const float4 p0 = Pp[0], p1 = Pp[1];
    const P mx = pk<P>(p0.x, p0.y), my = pk<P>(p0.z, p0.w), mz = pk<P>(p1.x, p1.y);
    LkLook<P> L;
    // decision sequence: q~ = fma(R_a2, mz, fma(R_a1, my, R_a0 mx)), q = q~ + t
    L.qx = add2(fma2(R[2], mz, fma2(R[1], my, mul2(R[0], mx))), tx);
    L.qy = add2(fma2(R[5], mz, fma2(R[4], my, mul2(R[3], mx))), ty);
    L.qz = add2(fma2(R[8], mz, fma2(R[7], my, mul2(R[6], mx))), tz);
    return L;
}

// And its map indices.
template <typename P>
__device__ __forceinline__ LkLook<P> lk2_lookup(const LkArgs& A, const P R[9], P tx, P ty, P tz, const float4* Pp) {
    constexpr bool PAIR = sizeof(P) == sizeof(float2);
    LkLook<P> L = lk2_point<P>(R, tx, ty, tz, Pp);
    // voxel = floor(fma(q, 1/res, off)): round-down add of 1.5 * 2^23
    const P fx = add2_rd(fma2(L.qx, pk<P>(A.inv2), pk<P>(A.offx2)), pk<P>(A.magic2));
    const P fy = add2_rd(fma2(L.qy, pk<P>(A.inv2), pk<P>(A.offy2)), pk<P>(A.magic2));
    const P fz = add2_rd(fma2(L.qz, pk<P>(A.inv2), pk<P>(A.offz2)), pk<P>(A.magic2));
    // unsigned arithmetic: an out-of-range voxel wraps to a large value
    const unsigned vxa = __float_as_uint(first(fx)) - 0x4B400000u, vxb = __float_as_uint(second(fx)) - 0x4B400000u;
    const unsigned vya = __float_as_uint(first(fy)) - 0x4B400000u, vyb = __float_as_uint(second(fy)) - 0x4B400000u;
    const unsigned vza = __float_as_uint(first(fz)) - 0x4B400000u, vzb = __float_as_uint(second(fz)) - 0x4B400000u;
    const bool ina = vxa < (unsigned)A.nx && vya < (unsigned)A.ny && vza < (unsigned)A.nz;
    const bool inb = vxb < (unsigned)A.nx && vyb < (unsigned)A.ny && vzb < (unsigned)A.nz;
    L.ma = -1;
    L.mb = -1;
    if (ina) L.ma = __ldg(A.nnf + (((int)vza * A.ny + (int)vya) * A.nx + (int)vxa));
    if (PAIR && inb) L.mb = __ldg(A.nnf + (((int)vzb * A.ny + (int)vyb) * A.nx + (int)vxb));
    return L;
}

template <typename P>
__device__ __forceinline__ LkLook<P> lk2_none() {
    LkLook<P> L;
    L.ma = L.mb = -1;
    L.qx = L.qy = L.qz = pk<P>(0.f, 0.f);
    return L;
}

// Map record of index mm: (mu.xyz, w.x) and (w.y, w.z).
__device__ __forceinline__ void lk2_record(const LkArgs& A, int mm, float4& r0, float2& r1) {
    r0 = make_float4(0.f, 0.f, 0.f, 0.f);
    r1 = make_float2(0.f, 0.f);
    if (mm >= 0 && MP_DCHECK(mm < A.n_rec, "NNF entry beyond the map records", mm)) ld_record(A.rec + 2 * mm, r0, r1);
}

// The pair's sums: its lever arm q~ = q - t, its geometry, and the shared
// accumulation.
template <typename V, typename P>
__device__ __forceinline__ void lk2_accumulate(const LkArgs& A, LkSums<P>& S, const V R[9], P tx, P ty, P tz,
                                               const V nn[3], const LkLook<P>& L, const float4& ra0, const float2& ra1,
                                               const float4& rb0, const float2& rb1) {
    const P q[3] = {L.qx, L.qy, L.qz}, m1 = pk<P>(A.m1);
    LkPair<V, P> o;
    o.qt[0] = fma2(m1, tx, L.qx);
    o.qt[1] = fma2(m1, ty, L.qy);
    o.qt[2] = fma2(m1, tz, L.qz);
    lk_geometry(A, R, q, nn, LkRec{ra0, rb0, ra1, rb1}, o);
    lk_accumulate(A, S, o, L.ma >= 0, L.mb >= 0);
}

// The scan normal of a staged point (broadcast pairs).
template <typename P>
__device__ __forceinline__ void lk2_normal(const float4* p, P nn[3]) {
    nn[0] = pk<P>(p[1].z, p[1].w);
    nn[1] = pk<P>(p[2].x, p[2].y);
    nn[2] = pk<P>(p[2].z, p[2].w);
}

// One half (particle a: h = 0, b: h = 1) of the packed sums as scalar sums.
template <typename P>
__device__ __forceinline__ LkAcc lk2_half(const LkArgs& A, const LkSums<P>& S, int h, int nv) {
    LkAcc o;
#pragma unroll
    for (int k = 0; k < 6; ++k) { o.Hww[k] = h ? second(S.Hww[k]) : first(S.Hww[k]); o.Hvv[k] = h ? second(S.Hvv[k]) : first(S.Hvv[k]); }
#pragma unroll
    for (int k = 0; k < 9; ++k) o.Hwv[k] = h ? second(S.Hwv[k]) : first(S.Hwv[k]);
#pragma unroll
    for (int k = 0; k < 3; ++k) { o.bw[k] = h ? second(S.bw[k]) : first(S.bw[k]); o.bv[k] = -(h ? second(S.nbv[k]) : first(S.nbv[k])); }
    const float lc = h ? second(S.lc) : first(S.lc);
    const float cnt = h ? second(S.cnt) : first(S.cnt);
    // log p = -(sum of inlier costs) - c_max * (points that are not inliers)
    o.ll = fmaf(-A.c_max, (float)(nv - (int)cnt), -lc);
    o.cnt = (int)cnt;
    return o;
}

// Staging of the scan: two buffers, filled in turn; chunk q of a CTA's sequence
// is in buffer q & 1.
struct LkPmStage {
    float4 buf[2][3 * PM_CHUNK];
    uint64_t bar[2];
};

// One particle's sums over the m points of a staged chunk. With few warps a
// scheduler nothing hides a gather but the thread's own work, so the gathers run
// in groups of four points: while a group is accumulated, the records of the next
// and the NNF entries of the one after are in flight.
__device__ __forceinline__ void lk_pm1_chunk(const LkArgs& A, LkSums<float>& S, const float R[9], float tx, float ty, float tz,
                                             const float4* pts, int m) {
    constexpr int G = 4;   // (8: 198 registers, 2218 against 1926 us at 1024 particles x 8192 points)
    struct Group {
        float4 r0[G];
        float2 r1[G];
        bool hit[G];
    } u, v;
    int mm[G];
    auto look = [&](int k0) {
#pragma unroll
        for (int g = 0; g < G; ++g) mm[g] = k0 + g < m ? lk2_lookup<float>(A, R, tx, ty, tz, pts + 3 * (k0 + g)).ma : -1;
    };
    auto records = [&](Group& r) {
#pragma unroll
        for (int g = 0; g < G; ++g) {
            r.hit[g] = mm[g] >= 0;
            lk2_record(A, mm[g], r.r0[g], r.r1[g]);
        }
    };
    auto accumulate = [&](const Group& r, int k0) {
#pragma unroll
        for (int g = 0; g < G; ++g) {
            if (k0 + g >= m) break;
            LkLook<float> L = lk2_point<float>(R, tx, ty, tz, pts + 3 * (k0 + g));
            L.ma = r.hit[g] ? 0 : -1;
            float nn[3];
            lk2_normal<float>(pts + 3 * (k0 + g), nn);
            lk2_accumulate(A, S, R, tx, ty, tz, nn, L, r.r0[g], r.r1[g], r.r0[g], r.r1[g]);
        }
    };
    look(0);
    records(u);
    look(G);
    for (int k0 = 0; k0 < m; k0 += 2 * G) {
        records(v);
        look(k0 + 2 * G);
        accumulate(u, k0);
        records(u);
        look(k0 + 3 * G);
        accumulate(v, k0 + G);
    }
}

// The sums of particle block bxi over chunks [c0, c1) of the scan, whose
// sequence numbers start at q; returns false when a wait gave up. PART: the
// block's sums so far are read from (c0 > 0) and left in (c1 < all) its columns
// of the Gauss-Newton sums, in FP32 as they are.
template <bool PART, typename P>
__device__ __forceinline__ bool lk_pm_block(const LkArgs& A, LkPmStage& st, int64_t bxi, int nv, int c0, int c1, int q) {
    // particles a and b of this thread sit PM_THREADS apart in sorted order,
    // so each half of a warp covers 32 consecutive sorted particles
    constexpr bool PAIR = sizeof(P) == sizeof(float2);
    const int64_t pa = (int64_t)bxi * (PAIR ? PM_PER_CTA : PM_THREADS) + threadIdx.x;
    const int64_t pb = pa + PM_THREADS;
    const bool acta = pa < A.n, actb = PAIR && pb < A.n;
    int64_t ia = acta ? A.order[pa] : 0, ib = actb ? A.order[pb] : 0;
    if (!MP_DCHECK(ia >= 0 && ia < A.n, "particle order entry", ia)) ia = 0;
    if (!MP_DCHECK(ib >= 0 && ib < A.n, "particle order entry", ib)) ib = 0;
    P R[9];
    P tx, ty, tz;
    {
        Quat qa, qb;
        float ta[3], tb[3], Ra[9], Rb[9];
        load_pose(A.poses, ia, qa, ta);
        load_pose(A.poses, ib, qb, tb);
        quat_rot_exact(qa, Ra);
        quat_rot_exact(qb, Rb);
#pragma unroll
        for (int k = 0; k < 9; ++k) R[k] = pk<P>(Ra[k], Rb[k]);
        tx = pk<P>(ta[0], tb[0]);
        ty = pk<P>(ta[1], tb[1]);
        tz = pk<P>(ta[2], tb[2]);
    }

    const int nchunks = (nv + PM_CHUNK - 1) / PM_CHUNK;
    auto issue = [&](int cc) {
        float4* dst = st.buf[(q + cc - c0) & 1];
        uint64_t* b = &st.bar[(q + cc - c0) & 1];
        int m = min(PM_CHUNK, nv - cc * PM_CHUNK);
        if (!MP_DCHECK(cc >= 0 && m > 0 && ((reinterpret_cast<uintptr_t>(A.scan_pm) & 15) == 0), "scan chunk", cc))
            return;
        uint32_t bytes = (uint32_t)m * 48u;
        fence_proxy_async_smem();   // the block's reads of dst (a reused buffer) before the copy's writes
        mbar_expect_tx(b, bytes + ((A.starve && cc == 0) ? 16u : 0u));
        bulk_g2s(dst, A.scan_pm + 3 * (int64_t)cc * PM_CHUNK, bytes, b);
    };
    if (threadIdx.x == 0) {
        if (c0 < c1) issue(c0);
        if (c0 + 1 < c1) issue(c0 + 1);
    }

    LkSums<P> S;
    P* const sum = reinterpret_cast<P*>(&S);   // LK_SUMS of them
    constexpr int LK_SUMS = sizeof(S) / sizeof(P);
    static_assert(LK_SUMS == MP_GN, "one column of the Gauss-Newton sums each");
#pragma unroll
    for (int k = 0; k < LK_SUMS; ++k) {
        sum[k] = pk<P>(0.f, 0.f);
        if (PART && c0 > 0)   // (through L2: another SM may have stored them in this launch)
            sum[k] = pk<P>(acta ? __ldcg(A.gn + (int64_t)k * A.stride + pa) : 0.f,
                           actb ? __ldcg(A.gn + (int64_t)k * A.stride + pb) : 0.f);
    }

    const bool active = acta;   // acta is false only if actb is false too
    bool failed = false;
    int c = c0;
    for (; c < c1; ++c) {
        const int b = (q + c - c0) & 1;
        const uint32_t parity = (uint32_t)(((q + c - c0) >> 1) & 1);
        bool got = mbar_wait_bounded(&st.bar[b], parity, A.budget);
        if (__syncthreads_or(!got)) { failed = true; break; }
        const int m = min(PM_CHUNK, nv - c * PM_CHUNK);
        if constexpr (!PAIR) {
            if (active) lk_pm1_chunk(A, S, R, tx, ty, tz, st.buf[b], m);
        } else if (active) {
            const float4* pts = st.buf[b];
            // software pipeline over the two dependent gathers: every
            // iteration issues the NNF loads of point k+2 and the record loads
            // of point k+1 before the arithmetic of point k. Invariant at the
            // loop head: sc = point k (records loaded), sb = point k+1 (map
            // indices loaded).
            LkLook<P> sb = lk2_none<P>(), sc = lk2_lookup<P>(A, R, tx, ty, tz, pts);
            float4 ra0, rb0;
            float2 ra1, rb1;
            lk2_record(A, sc.ma, ra0, ra1);
            lk2_record(A, sc.mb, rb0, rb1);
            if (m > 1) sb = lk2_lookup<P>(A, R, tx, ty, tz, pts + 3);
            for (int k = 0; k < m; ++k) {
                const LkLook<P> nb = (k + 2 < m) ? lk2_lookup<P>(A, R, tx, ty, tz, pts + 3 * (k + 2)) : lk2_none<P>();
                float4 na0, nb0;
                float2 na1, nb1;
                lk2_record(A, sb.ma, na0, na1);
                lk2_record(A, sb.mb, nb0, nb1);
                P nn[3];
                lk2_normal<P>(pts + 3 * k, nn);
                lk2_accumulate(A, S, R, tx, ty, tz, nn, sc, ra0, ra1, rb0, rb1);
                sc = sb;
                sb = nb;
                ra0 = na0; ra1 = na1; rb0 = nb0; rb1 = nb1;
            }
        }
        __syncthreads();
        if (threadIdx.x == 0 && c + 2 < c1) issue(c + 2);
    }
    if (failed) {
        if (threadIdx.x == 0) {
            atomicOr(A.err, MP_ERR_WAIT);
            for (int k = c; k < min(c + 2, c1); ++k)
                mbar_wait_bounded(&st.bar[(q + k - c0) & 1], (uint32_t)(((q + k - c0) >> 1) & 1), A.budget);
        }
        return false;
    }
    if (PART && c1 < nchunks) {
#pragma unroll
        for (int k = 0; k < LK_SUMS; ++k) {
            if (acta) A.gn[(int64_t)k * A.stride + pa] = first(sum[k]);
            if (actb) A.gn[(int64_t)k * A.stride + pb] = second(sum[k]);
        }
        return true;
    }
    float Rs[9];
    if (acta) {
#pragma unroll
        for (int k = 0; k < 9; ++k) Rs[k] = first(R[k]);
        lk_store(A, Rs, lk2_half(A, S, 0, nv), pa);
    }
    if (actb) {
#pragma unroll
        for (int k = 0; k < 9; ++k) Rs[k] = second(R[k]);
        lk_store(A, Rs, lk2_half(A, S, 1, nv), pb);
    }
    return true;
}

__device__ __forceinline__ int lk_pm_begin(const LkArgs& A, LkPmStage& st, unsigned bxi) {
    int nv = *A.nvalid;
    if (!MP_DCHECK(nv >= 0 && nv <= A.scan_cap, "valid scan points", nv)) nv = 0;
    if (bxi == 0 && threadIdx.x == 0)
        atomicAdd(A.pairs, (unsigned long long)A.n * (unsigned long long)nv);
    if (threadIdx.x == 0) {
        mbar_init(&st.bar[0], 1);
        mbar_init(&st.bar[1], 1);
        mbar_fence_init();
    }
    __syncthreads();
    return nv;
}

struct LkPmOp {
    using Args = LkArgs;
    static constexpr int THREADS = PM_THREADS, MINB = PM_MINB;
    static __device__ __forceinline__ void run(const LkArgs& A, unsigned bxi, unsigned) {
        __shared__ __align__(128) LkPmStage st;
        const int nv = lk_pm_begin(A, st, bxi);
        lk_pm_block<false, float2>(A, st, bxi, nv, 0, (nv + PM_CHUNK - 1) / PM_CHUNK, 0);
    }
};

__global__ void __launch_bounds__(PM_THREADS, PM_MINB) k_likelihood_pm(const LkArgs A) {
    LkPmOp::run(A, blockIdx.x, 0);
}

// One particle a thread, for fewer particles than pairs of them would keep the
// SMs' schedulers busy with: twice the warps, and gathers four points deep where
// a lone warp waited 1200 cycles a point (outdoors, likelihood stage, packed ->
// now: 1024 particles x 8192 points 6.2 -> 1.9 ms, 8192 5.7 -> 1.9, 32768 5.5 ->
// 2.6, 65536 6.2 -> 5.0, 98304 7.2 -> 6.7; 131072 8.15 and 8.19; 50021 x 4999 3.59
// -> 2.07). The sums are the packed form's, bit for bit.
struct LkPm1Op {
    using Args = LkArgs;
    static constexpr int THREADS = PM_THREADS, MINB = PM1_MINB;
    static __device__ __forceinline__ void run(const LkArgs& A, unsigned bxi, unsigned) {
        __shared__ __align__(128) LkPmStage st;
        const int nv = lk_pm_begin(A, st, bxi);
        lk_pm_block<false, float>(A, st, bxi, nv, 0, (nv + PM_CHUNK - 1) / PM_CHUNK, 0);
    }
};

__global__ void __launch_bounds__(PM_THREADS, PM1_MINB) k_likelihood_pm1(const LkArgs A) {
    LkPm1Op::run(A, blockIdx.x, 0);
}

// The same over parts of the scan: item t of A.items x blocks is part t /
// blocks of particle block t mod blocks, taken from a counter by the resident
// CTAs. A block's parts follow one another (the sums and their rounding are
// those of one pass), each waiting, boundedly, until the part before is
// stored; that part was taken earlier, by a running CTA. With whole blocks the
// last wave of CTAs is as long as the others however few they are: 2^17
// particles are 1.1 waves of 152 x 3 CTAs and took 2 (box room x 1024 points 919
// -> 818 us, outdoors 10.4 -> 8.2 ms; 4 or 16 parts instead of 8: 847, 816 us).
__global__ void __launch_bounds__(PM_THREADS, PM_MINB) k_likelihood_pm_parts(const LkArgs A) {
    __shared__ __align__(128) LkPmStage st;
    __shared__ int take;
    const int nv = lk_pm_begin(A, st, blockIdx.x);
    const int nchunks = (nv + PM_CHUNK - 1) / PM_CHUNK;
    const int blocks = (int)((A.n + PM_PER_CTA - 1) / PM_PER_CTA);
    const int len = max(1, (nchunks + A.items - 1) / A.items);   // chunks of a part
    const int parts = max(1, (nchunks + len - 1) / len);
    int* const next = A.ticket;
    int* const done = A.ticket + 1;
    int q = 0;
    for (;;) {
        if (threadIdx.x == 0) {
            int t = atomicAdd(next, 1);
            if (t < parts * blocks) {
                const int part = t / blocks, blk = t - part * blocks;
                const long long t0 = clock64();
                while ((int)ld_acquire_u32(reinterpret_cast<unsigned*>(done + blk)) < part) {
                    if (clock64() - t0 > A.budget) {
                        atomicOr(A.err, MP_ERR_WAIT);
                        t = INT_MAX;
                        break;
                    }
                    __nanosleep(200);
                }
            }
            take = t;
        }
        __syncthreads();
        const int t = take;
        if (t >= parts * blocks) return;
        const int part = t / blocks, blk = t - part * blocks;
        const int c0 = part * len, c1 = min(nchunks, c0 + len);
        if (!lk_pm_block<true, float2>(A, st, blk, nv, c0, c1, q)) return;
        q += c1 - c0;
        __threadfence();      // the stored sums before the count
        __syncthreads();
        if (threadIdx.x == 0) atomicExch(done + blk, part + 1);
    }
}

// the valid scan as 16-bit broadcast pairs: (mx,mx) (my,my) (mz,mz) (nx,nx) | (ny,ny) (nz,nz) 0 0
template <typename H2>
__global__ void k_scan_to_h2(const float4* __restrict__ pair, const int32_t* __restrict__ nvalid, int n,
                             uint4* __restrict__ out) {
    using T = Half2<H2>;
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n || i >= *nvalid) return;
    const float4 a = pair[3 * i], b = pair[3 * i + 1], c = pair[3 * i + 2];
    out[2 * i] = make_uint4(h2_word(T::from(make_float2(a.x, a.y))), h2_word(T::from(make_float2(a.z, a.w))),
                            h2_word(T::from(make_float2(b.x, b.y))), h2_word(T::from(make_float2(b.z, b.w))));
    out[2 * i + 1] = make_uint4(h2_word(T::from(make_float2(c.x, c.y))), h2_word(T::from(make_float2(c.z, c.w))), 0u, 0u);
}

template <typename H2>
__device__ __forceinline__ Lk2Look lkh_lookup(const LkArgs& A, const H2 R[9], float2 tx, float2 ty, float2 tz,
                                              const uint4* Pp) {
    using T = Half2<H2>;
    const uint4 p0 = Pp[0];
    const H2 mx = h2_bits<H2>(p0.x), my = h2_bits<H2>(p0.y), mz = h2_bits<H2>(p0.z);
    Lk2Look L;
    L.qx = add2(T::to(__hfma2(R[2], mz, __hfma2(R[1], my, __hmul2(R[0], mx)))), tx);
    L.qy = add2(T::to(__hfma2(R[5], mz, __hfma2(R[4], my, __hmul2(R[3], mx)))), ty);
    L.qz = add2(T::to(__hfma2(R[8], mz, __hfma2(R[7], my, __hmul2(R[6], mx)))), tz);
    const float2 fx = __fadd2_rd(fma2(L.qx, A.inv2, A.offx2), A.magic2);
    const float2 fy = __fadd2_rd(fma2(L.qy, A.inv2, A.offy2), A.magic2);
    const float2 fz = __fadd2_rd(fma2(L.qz, A.inv2, A.offz2), A.magic2);
    // unsigned arithmetic: an out-of-range voxel wraps to a large value
    const unsigned vxa = __float_as_uint(fx.x) - 0x4B400000u, vxb = __float_as_uint(fx.y) - 0x4B400000u;
    const unsigned vya = __float_as_uint(fy.x) - 0x4B400000u, vyb = __float_as_uint(fy.y) - 0x4B400000u;
    const unsigned vza = __float_as_uint(fz.x) - 0x4B400000u, vzb = __float_as_uint(fz.y) - 0x4B400000u;
    const bool ina = vxa < (unsigned)A.nx && vya < (unsigned)A.ny && vza < (unsigned)A.nz;
    const bool inb = vxb < (unsigned)A.nx && vyb < (unsigned)A.ny && vzb < (unsigned)A.nz;
    L.ma = -1;
    L.mb = -1;
    if (ina) L.ma = __ldg(A.nnf + (((int)vza * A.ny + (int)vya) * A.nx + (int)vxa));
    if (inb) L.mb = __ldg(A.nnf + (((int)vzb * A.ny + (int)vyb) * A.nx + (int)vxb));
    return L;
}

template <typename H2, int MINB>
__global__ void __launch_bounds__(PM_THREADS, MINB) k_likelihood_pm_h(const LkArgs A) {
    using T = Half2<H2>;
    __shared__ __align__(128) uint4 buf[2][2 * PM_CHUNK];
    __shared__ __align__(8) uint64_t bar[2];

    const int64_t pa = (int64_t)blockIdx.x * PM_PER_CTA + threadIdx.x;
    const int64_t pb = pa + PM_THREADS;
    const bool acta = pa < A.n, actb = pb < A.n;
    int64_t ia = acta ? A.order[pa] : 0, ib = actb ? A.order[pb] : 0;
    if (!MP_DCHECK(ia >= 0 && ia < A.n, "particle order entry", ia)) ia = 0;
    if (!MP_DCHECK(ib >= 0 && ib < A.n, "particle order entry", ib)) ib = 0;
    H2 R[9];
    float2 tx, ty, tz;
    {
        Quat qa, qb;
        float ta[3], tb[3], Ra[9], Rb[9];
        load_pose(A.poses, ia, qa, ta);
        load_pose(A.poses, ib, qb, tb);
        quat_rot_exact(qa, Ra);
        quat_rot_exact(qb, Rb);
#pragma unroll
        for (int k = 0; k < 9; ++k) R[k] = T::from(make_float2(Ra[k], Rb[k]));
        tx = make_float2(ta[0], tb[0]);
        ty = make_float2(ta[1], tb[1]);
        tz = make_float2(ta[2], tb[2]);
    }

    int nv = *A.nvalid;
    if (!MP_DCHECK(nv >= 0 && nv <= A.scan_cap, "valid scan points", nv)) nv = 0;
    const int nchunks = (nv + PM_CHUNK - 1) / PM_CHUNK;
    if (blockIdx.x == 0 && threadIdx.x == 0) atomicAdd(A.pairs, (unsigned long long)A.n * (unsigned long long)nv);
    if (threadIdx.x == 0) {
        mbar_init(&bar[0], 1);
        mbar_init(&bar[1], 1);
        mbar_fence_init();
    }
    __syncthreads();
    auto issue = [&](uint4* dst, uint64_t* b, int cc) {
        int m = min(PM_CHUNK, nv - cc * PM_CHUNK);
        if (!MP_DCHECK(cc >= 0 && m > 0 && ((reinterpret_cast<uintptr_t>(A.scan_h) & 15) == 0), "scan chunk", cc))
            return;
        uint32_t bytes = (uint32_t)m * 32u;
        fence_proxy_async_smem();   // the block's reads of dst (a reused buffer) before the copy's writes
        mbar_expect_tx(b, bytes + ((A.starve && cc == 0) ? 16u : 0u));
        bulk_g2s(dst, A.scan_h + 2 * (int64_t)cc * PM_CHUNK, bytes, b);
    };
    if (threadIdx.x == 0) {
        if (nchunks > 0) issue(buf[0], &bar[0], 0);
        if (nchunks > 1) issue(buf[1], &bar[1], 1);
    }

    Lk2Acc S;
    const float2 z2 = make_float2(0.f, 0.f);
#pragma unroll
    for (int k = 0; k < 6; ++k) { S.Hww[k] = z2; S.Hvv[k] = z2; }
#pragma unroll
    for (int k = 0; k < 9; ++k) S.Hwv[k] = z2;
#pragma unroll
    for (int k = 0; k < 3; ++k) { S.bw[k] = z2; S.nbv[k] = z2; }
    S.lc = z2;
    S.cnt = z2;

    bool failed = false;
    int c = 0;
    for (; c < nchunks; ++c) {
        const int b = c & 1;
        const uint32_t parity = (uint32_t)((c >> 1) & 1);
        bool got = mbar_wait_bounded(&bar[b], parity, A.budget);
        if (__syncthreads_or(!got)) { failed = true; break; }
        const int m = min(PM_CHUNK, nv - c * PM_CHUNK);
        if (acta) {
            const uint4* P = buf[b];
            // the same two-gather software pipeline as the FP32 form
            Lk2Look sb = lk2_none<float2>(), sc = lkh_lookup<H2>(A, R, tx, ty, tz, P);
            float4 ra0, rb0;
            float2 ra1, rb1;
            lk2_record(A, sc.ma, ra0, ra1);
            lk2_record(A, sc.mb, rb0, rb1);
            if (m > 1) sb = lkh_lookup<H2>(A, R, tx, ty, tz, P + 2);
            for (int k = 0; k < m; ++k) {
                const Lk2Look nb = (k + 2 < m) ? lkh_lookup<H2>(A, R, tx, ty, tz, P + 2 * (k + 2)) : lk2_none<float2>();
                float4 na0, nb0;
                float2 na1, nb1;
                lk2_record(A, sb.ma, na0, na1);
                lk2_record(A, sb.mb, nb0, nb1);
                const H2 nn[3] = {h2_bits<H2>(P[2 * k].w), h2_bits<H2>(P[2 * k + 1].x), h2_bits<H2>(P[2 * k + 1].y)};
                lk2_accumulate(A, S, R, tx, ty, tz, nn, sc, ra0, ra1, rb0, rb1);
                sc = sb;
                sb = nb;
                ra0 = na0; ra1 = na1; rb0 = nb0; rb1 = nb1;
            }
        }
        __syncthreads();
        if (threadIdx.x == 0 && c + 2 < nchunks) issue(buf[b], &bar[b], c + 2);
    }
    if (failed) {
        if (threadIdx.x == 0) {
            atomicOr(A.err, MP_ERR_WAIT);
            for (int k = c; k < min(c + 2, nchunks); ++k)
                mbar_wait_bounded(&bar[k & 1], (uint32_t)((k >> 1) & 1), A.budget);
        }
        return;
    }
    // the FP32 rotation of each particle for the sums' frame change
    float Rs[9];
    Quat q;
    float t[3];
    if (acta) {
        load_pose(A.poses, ia, q, t);
        quat_rot_exact(q, Rs);
        lk_store(A, Rs, lk2_half(A, S, 0, nv), pa);
    }
    if (actb) {
        load_pose(A.poses, ib, q, t);
        quat_rot_exact(q, Rs);
        lk_store(A, Rs, lk2_half(A, S, 1, nv), pb);
    }
}

}  // namespace

namespace {

// The shape of a launch over n particles. Up to 1024 of them, four warps share
// a particle (else a warp each, and half the SMs' schedulers would be idle). A
// warp takes up to 16 particles one after the other on the chunks its CTA has
// staged, as long as four waves of CTAs remain (4 instead of 16: 57.6 against
// 56.6 ms for 2^20 x 8192; 32: 54.5 against 52.9).
void lk_shape(int64_t n, LkArgs& A) {
    A.wpp = n <= 1024 ? LK_WARPS : 1;
    const int64_t per_round = LK_WARPS / A.wpp;
    A.rounds = (int)std::min<int64_t>(16, std::max<int64_t>(1, n / (per_round * 152 * LK_MINB * 4)));
}

int64_t lk_blocks(const LkArgs& A) {
    const int64_t per_cta = (int64_t)A.rounds * (LK_WARPS / A.wpp);
    return (A.n + per_cta - 1) / per_cta;
}

// Launches over a scan of n_scan points (at least one: it writes the zeros of
// a scan without valid points), of about equal parts.
int lk_segments(int n_scan, LkArgs& A) {
    const int chunks = std::max(1, (n_scan + LK_CHUNK * A.split - 1) / (LK_CHUNK * A.split));
    const int segs = (chunks + LK_SEG - 1) / LK_SEG;
    A.seg_len = (chunks + segs - 1) / segs;
    return segs;
}

// A map of more than LK_WIDE voxels across. Its sums keep one order, the scan's,
// unless the caller asks for a split (mp_set_likelihood_split; a batch's tuning
// does not): a lever arm of hundreds of voxels turns the last bits of a
// particle's step into other voxels for some of its points in the next, and with
// the particles close around the sensor the log posterior of two orders differed
// by 0.04 of its norm after a second step. Measured on two maps, 1000 voxels
// across (that) and 100 (1e-6); the line lies between them, unmeasured.
bool lk_wide(const mp_ctx* c) {
    return std::max(c->nnf_dims[0], std::max(c->nnf_dims[1], c->nnf_dims[2])) > LK_WIDE;
}

// Whether a launch takes the particle-major form: on wide maps, and from 80k particles on, which
// are 320 of the 456 CTAs the GPU holds. Measured, box room x 1024 points,
// particle-major / point-major: 32k particles 326 / 252 us, 64k 491 / 487, 96k
// 670 / 730, 128k 818 / 953, 256k 1511 / 1815, and 512k x 512 1405 / 2007 (the
// point-major form's lanes' points are 0.5 m apart there, each on a line of its
// own, and the queue adds shared-memory traffic to an L1 that is already 72%
// busy); outdoors x 8192 points 128k 8.2 / 8.1 ms, 512k 27.0 / 26.9, 1M 52.4 /
// 51.8, and with all particles around the sensor 256k 12.6 / 15.0 ms in their
// first step and 16.7 / 11.0 later. In 16 bits (box room x 1021 points) 64k 637
// / 577 us, 128k 1041 / 1142. The particle-major sums are added in scan order,
// point by point, whatever the launch. A scan split is the point-major form's.
bool lk_particle_major(const mp_ctx* c, int split) {
    return split == 1 && (c->n >= LK_PM_MIN || lk_wide(c));
}

LkArgs lk_args(mp_ctx* c) {
    LkArgs A;
    A.poses = c->poses[c->cur];
    A.order = c->visit;
    A.n = c->n;
    A.scan = c->scan_soa;
    A.scan_pm = c->scan_pair;
    A.items = 8;
    A.ticket = c->lk_ticket;
    A.nvalid = c->scan_nvalid;
    A.nnf = c->nnf;
    A.nx = c->nnf_dims[0]; A.ny = c->nnf_dims[1]; A.nz = c->nnf_dims[2];
    A.rec = c->map_rec;
    A.c_max = c->p.c_max;
    A.gn = c->gn;
    A.stride = c->cap;
    A.err = c->dev_error;
    A.budget = c->wait_budget > 0 ? c->wait_budget : MP_WAIT_BUDGET;
    A.starve = c->starve_tx;
    A.pairs = c->pairs;
    const float a = 1.f - c->p.eps_cov;
    auto pair = [](float v) { return make_float2(v, v); };
    A.inv2 = pair(c->nnf_inv_res);
    A.offx2 = pair(c->nnf_off[0]); A.offy2 = pair(c->nnf_off[1]); A.offz2 = pair(c->nnf_off[2]);
    A.magic2 = pair(12582912.0f);   // 1.5 * 2^23: round-down add gives floor in the low bits
    A.m1 = pair(-1.f);
    A.half2 = pair(0.5f);
    A.half_a2 = pair(0.5f * a);
    A.nhalf_a2 = pair(-0.5f * a);
    A.two_eps2 = pair(2.f * c->p.eps_cov);
    A.two2 = pair(2.f);
    A.quarter_a2 = pair(0.25f * a);
    A.scan_h = c->scan_h2;
    A.split = c->lk_split > 1 ? c->lk_split : 1;
    lk_shape(c->n, A);
    A.n_rec = c->n_map;
    A.scan_cap = c->p.max_scan;
    return A;
}

}  // namespace

namespace {

template <typename V>
int launch_point_major(mp_ctx* c, LkArgs A) {
    // a scan split (a tuning knob) adds the partial sums of its CTAs into a
    // zeroed output
    if (A.split > 1) MP_CUDA(c, cudaMemsetAsync(c->gn, 0, sizeof(float) * MP_GN * (size_t)c->cap, c->stream));
    const dim3 grid((unsigned)lk_blocks(A), (unsigned)A.split);
    const int segs = lk_segments(c->n_prep, A);
    for (A.seg = 0; A.seg < segs; ++A.seg) {
        MP_CUDA(c, launch_next(A.wpp > 1 ? k_likelihood<LK_WARPS, V> : k_likelihood<1, V>, grid, LK_THREADS, 0, c->stream, A));
        MP_LAUNCHED(c);
    }
    return MP_OK;
}

template <typename H2>
int launch_particle_major_16(mp_ctx* c, const LkArgs& A) {
    if (c->n_prep > 0) {
        k_scan_to_h2<H2><<<grid_for(c->n_prep, 256), 256, 0, c->stream>>>(c->scan_pair, c->scan_nvalid, c->n_prep,
                                                                          c->scan_h2);
        MP_LAUNCHED(c);
    }
    k_likelihood_pm_h<H2, PMH_MINB><<<grid_for(c->n, PM_PER_CTA), PM_THREADS, 0, c->stream>>>(A);
    MP_LAUNCHED(c);
    return MP_OK;
}

}  // namespace

bool mp_likelihood_in_scan_order(const mp_ctx* c) { return lk_particle_major(c, 1); }

int mp_launch_likelihood(mp_ctx* c) {
    LkArgs A = lk_args(c);
    if (c->precision != MP_PREC_FP32) A.split = 1;   // the split is the FP32 form's
    const bool pm = lk_particle_major(c, A.split);
    if (c->precision == MP_PREC_BF16)
        return pm ? launch_particle_major_16<__nv_bfloat162>(c, A) : launch_point_major<__nv_bfloat162>(c, A);
    if (c->precision == MP_PREC_FP16)
        return pm ? launch_particle_major_16<__half2>(c, A) : launch_point_major<__half2>(c, A);
    if (!pm) return launch_point_major<float2>(c, A);
    const int64_t blocks = (c->n + PM_PER_CTA - 1) / PM_PER_CTA;
    const int64_t slots = 152 * PM_MINB;
    if (lk_wide(c) && c->n <= LK_PM1_MAX) {
        k_likelihood_pm1<<<grid_for(c->n, PM_THREADS), PM_THREADS, 0, c->stream>>>(A);
    } else if (blocks <= slots || c->n_prep <= PM_CHUNK) {
        k_likelihood_pm<<<(unsigned)blocks, PM_THREADS, 0, c->stream>>>(A);
    } else {
        MP_CUDA(c, cudaMemsetAsync(c->lk_ticket, 0, sizeof(int) * (size_t)(blocks + 1), c->stream));
        // the test knob hands out no item 0: the second part of block 0 waits for the first
        // (a branch for it in the kernel moved its registers from 166 to 161: 3% slower)
        if (c->starve_bar) MP_CUDA(c, cudaMemsetAsync(c->lk_ticket, 1, 1, c->stream));
        k_likelihood_pm_parts<<<(unsigned)slots, PM_THREADS, 0, c->stream>>>(A);
    }
    MP_LAUNCHED(c);
    return MP_OK;
}

// Grouped likelihood (FP32): one launch for the instances in particle-major
// form, or, while those on wide maps have at most LK_PM1_MAX particles in all,
// one for them with one particle a thread and one for the rest (the same bits;
// a step of 24 instances of 1024 x 8192 points on a wide map 7.84 -> 6.00 ms, of 24 of
// 1024-8192 x 512-2048 2.26 -> 1.69; 8 of 32768, above the line, 6.2); of the others, per segment of the scan, one for those whose particles
// take a warp each and one for those whose particles take a CTA (the sums of
// an instance with a scan split zeroed first; block (bx, by) of the map =
// particle block bx, scan part by).
int mp_plan_likelihood(mp_group* G, int, std::vector<GOp>& plan) {
    std::vector<LkArgs> tab;
    std::vector<int64_t> blocks, blocks_pm, blocks_pm1;
    std::vector<int> ys, nseg, pm, wide;
    int64_t n_wide = 0;
    int segs = 0;
    for (int i = 0; i < G->size(); ++i) {
        mp_ctx* c = G->ctx[i];
        tab.push_back(lk_args(c));
        LkArgs& A = tab.back();
        blocks.push_back(lk_blocks(A));
        blocks_pm.push_back((c->n + PM_PER_CTA - 1) / PM_PER_CTA);
        blocks_pm1.push_back((c->n + PM_THREADS - 1) / PM_THREADS);
        ys.push_back(A.split);
        const bool by_particle = lk_particle_major(c, A.split);
        if (by_particle) (lk_wide(c) ? wide : pm).push_back(i);
        if (by_particle && lk_wide(c)) n_wide += c->n;
        nseg.push_back(by_particle ? 0 : lk_segments(G->n_scan[i], A));
        segs = std::max(segs, nseg.back());
        if (A.split > 1) plan_memset(plan, c->gn, sizeof(float) * MP_GN * (size_t)c->cap);
    }
    unsigned nblk = 0;
    if (n_wide > LK_PM1_MAX) {
        pm.insert(pm.end(), wide.begin(), wide.end());
        wide.clear();
    }
    if (!wide.empty()) {
        const LkArgs* t = G->upload(tab);
        const GBlk* m = G->block_map(blocks_pm1, &nblk, wide);
        plan_kernel<LkPm1Op>(plan, t, m, nblk);
    }
    if (!pm.empty()) {
        const LkArgs* t = G->upload(tab);
        const GBlk* m = G->block_map(blocks_pm, &nblk, pm);
        plan_kernel<LkPmOp>(plan, t, m, nblk);
    }
    for (int s = 0; s < segs; ++s) {
        std::vector<int> which[2];
        for (int i = 0; i < G->size(); ++i) {
            tab[i].seg = s;
            if (s < nseg[i]) which[tab[i].wpp > 1].push_back(i);
        }
        const LkArgs* t = G->upload(tab);
        if (!which[0].empty()) {
            const GBlk* m = G->block_map(blocks, &nblk, which[0], ys);
            plan_kernel<LkOp<1, float2>>(plan, t, m, nblk);
        }
        if (!which[1].empty()) {
            const GBlk* m = G->block_map(blocks, &nblk, which[1], ys);
            plan_kernel<LkOp<LK_WARPS, float2>>(plan, t, m, nblk);
        }
    }
    return G->err;
}
