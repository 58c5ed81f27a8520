// One FDiRW macro step as a deterministic gather (Eq. 8 / Eq. 14 with a banded p):
//
//     chat(s)  = sigma_s * c(s)                                   (FP64 renormalisation, Sec. 3.3)
//     c'(x)    = sum_o Q[o][x] * chat(x - o),  o in [-R, R]^3 in a fixed order
//
// Q is destination-indexed (Q[o][x] = stored kernel of source x - o at offset o), so a warp reads consecutive
// values of each plane (16-byte vector loads where the rows are whole vectors), every cache value exactly once
// per step.  chat is stored with a zero
// halo of R cells on every side, so x - o never leaves the buffer and no bounds test is needed.
//
// Accumulation (Sec. 3.3: multiply in the storage precision, accumulate in higher precision):
//   - FP64 storage: FP64 FMA.
//   - FP32/FP16/BF16 storage: GB300 issues FP64 FMAs at 1/73 of the FP32 rate (measured), so each row of
//     2R+1 terms is summed as an unevaluated pair of FP32 values (s, c) -- error-free product (FMA
//     residual) and error-free addition (Knuth TwoSum), with chat split into hi = fp32(v),
//     lo = fp32(v - hi) -- and the rows of a destination are summed as a second FP32 pair (ff_add);
//     one FP64 addition per destination forms the result.
//   - FDIRW_ACCUM_FP32: FP32 products and row sums (one FMA per term), rows as above; the caller then
//     restores the step's FP64 mass budget (launch_restore_mass).
// The work per step is HBM-bound in the cache read (N * (2R+1)^3 * storage bytes).
#include "fdirw_internal.h"
#include "ff.cuh"

#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <type_traits>

namespace fdirw {

namespace {

// Two FP32 values per packed instruction; a - b as b (-1) + a, which rounds once like the subtraction.
__device__ __forceinline__ uint64_t pack2(float lo, float hi) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void unpack2(uint64_t v, float& lo, float& hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
    uint64_t d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
    uint64_t d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ uint64_t sub2(uint64_t a, uint64_t b) { return fma2(b, 0xbf800000bf800000ull, a); }

// ff_madd and ff_add on two destinations at once: the same operations in the same order, each rounding the same value up
// to its sign (the product is formed as -p from nhi = -hi, so that nothing has to be negated per term).
__device__ __forceinline__ void ff_madd2(uint64_t& s, uint64_t& c, uint64_t q, uint64_t hi, uint64_t nhi, uint64_t lo) {
    const uint64_t np = mul2(q, nhi);
    const uint64_t e = fma2(q, lo, fma2(q, hi, np));
    const uint64_t t = sub2(s, np);
    const uint64_t bp = sub2(t, s);
    const uint64_t err = sub2(sub2(s, sub2(t, bp)), add2(np, bp));
    s = t;
    c = add2(c, add2(err, e));
}
__device__ __forceinline__ void ff_add2(uint64_t& A, uint64_t& B, uint64_t s, uint64_t c) {
    const uint64_t t = add2(A, s);
    const uint64_t bp = sub2(t, A);
    const uint64_t e = add2(sub2(A, sub2(t, bp)), sub2(s, bp));
    const uint64_t f = add2(e, add2(B, c));
    A = add2(t, f);
    B = sub2(f, sub2(A, t));
}

// VX consecutive stored values (16 bytes) as VX / 2 pairs (j0(i), j0(i) + D): neighbours for FP32, whose 16 bytes
// are register pairs already, values VX / 2 apart for the 16-bit types, whose widening places them anyway.
template <typename ST>
struct Quad {
    static constexpr int D = sizeof(ST) == 4 ? 1 : 4;
    static constexpr __host__ __device__ int j0(int i) { return sizeof(ST) == 4 ? 2 * i : i; }
};
template <typename ST>
__device__ __forceinline__ uint64_t pair_of(uint4 v, int i) {
    auto pr = [](uint32_t a, uint32_t b) { return pack2(__uint_as_float(a), __uint_as_float(b)); };
    if constexpr (sizeof(ST) == 4) return i ? pr(v.z, v.w) : pr(v.x, v.y);
    const uint32_t a = i < 2 ? v.x : v.y, b = i < 2 ? v.z : v.w;
    if constexpr (std::is_same<ST, __half>::value) {
        const __half2 ha = *reinterpret_cast<const __half2*>(&a), hb = *reinterpret_cast<const __half2*>(&b);
        return i & 1 ? pack2(__high2float(ha), __high2float(hb)) : pack2(__low2float(ha), __low2float(hb));
    } else {
        return i & 1 ? pr(a & 0xffff0000u, b & 0xffff0000u) : pr(a << 16, b << 16);
    }
}

// One row of VX destinations: s (and c, float-float) += q[o_x] chat(x - o_x), o_x ascending for every destination.  q: the
// row's 2R+1 vectors; ch(k): its scaled values, k = x - o_x + R.  The loop goes over k, so that the pair of scaled values
// at k (and its negative) is put together once for all destinations that it meets.  Float-float sums are bound by the
// issue slots (11 packed operations of two cycles a pair of terms), and with the pairs made at every use 45% of the
// instructions were moves and sign flips: us a step with BF16 storage before -> after, 192^3 R = 8 16680 -> 15790
// (10230 at the copy rate), 64^3 R = 3 68 -> 63, 128^3 R = 2 205 -> 178; FP32 128^3 R = 1 61 -> 51.
template <typename ST, int R, bool FF, typename F>
__device__ __forceinline__ void row_sums(const uint4 (&q)[2 * R + 1], F ch, uint64_t (&s)[8 / sizeof(ST)],
                                         uint64_t (&c)[8 / sizeof(ST)]) {
    using U = Quad<ST>;
    constexpr int NP = 8 / sizeof(ST), K1 = 2 * R + U::j0(NP - 1);
    float2 v[K1 + U::D + 1];                              // (hi, lo); FP32: (value, -)
#pragma unroll
    for (int k = 0; k <= K1 + U::D; k++) v[k] = ch(k);
#pragma unroll
    for (int k = K1; k >= 0; k--) {
        const uint64_t hi = pack2(v[k].x, v[k + U::D].x);
        uint64_t nhi = 0, lo = 0;
        if (FF) {
            nhi = pack2(-v[k].x, -v[k + U::D].x);
            lo = pack2(v[k].y, v[k + U::D].y);
        }
#pragma unroll
        for (int i = 0; i < NP; i++) {
            const int ox = U::j0(i) - k + R;
            if (ox < -R || ox > R) continue;
            const uint64_t w = pair_of<ST>(q[ox + R], i);
            if constexpr (FF) ff_madd2(s[i], c[i], w, hi, nhi, lo);
            else s[i] = fma2(w, hi, s[i]);
        }
    }
}

// The gather over destinations in cell order.  A block is 8 warps: VW of them side by side in the destinations, and
// 8 / VW row groups that split the (2R+1)^2 rows (o_z, o_y).  A destination's row sums are added up within a group in
// ascending order and the groups' sums in ascending order at the end, the same in every gather kernel of a mode (FP32
// sums: one group).
//
// Why the rows are split: a grid of up to about 100^3 cells has too few destinations to fill 152 SMs with one thread
// for all rows of each (32^3 FP32 ones are 32 blocks of 256), and beyond that the last wave of long threads idles most
// of the chip.  us a step before -> after, FP32 cache, float-float sums: 32^3 R = 3 49 -> 14, 48^3 R = 8 1972 -> 346,
// 112^3 R = 8 6487 -> 4110 (4060 at the copy rate); FP64 36^3 R = 6 600 -> 188.  At R <= 2 (at most 25 rows) eight
// groups cost more than they give (128^3 R = 2 BF16 cache 100 -> 125): one.
constexpr int vector_warps(int R) { return R <= 2 ? 8 : 1; }
__device__ __forceinline__ int row_groups(int R) { return R <= 2 ? 1 : 8; }

struct GatherArgs {
    const void* Q;
    const void* chat;
    Grid g;
    Pad p;
    int64_t qs;                    // plane stride
    int z0, zn, qnx;               // destination planes; values in a cache row (>= nx)
    double* out;
    bool acc_in;
};

// Cache rows of whole 16-byte vectors: a thread owns VX consecutive destinations of an x row, one load of a plane.
// The destinations past nx in a padded row are computed from whatever lies there and not stored.  MODE 0: FP64
// throughout.  MODE 1: float-float rows (FDIRW_ACCUM_FF).  MODE 2: FP32 rows (FDIRW_ACCUM_FP32); both sum the rows of a
// destination as a float-float pair, which one FP64 addition turns into the result.  Two blocks per SM: 128 registers keep a row's loads in flight (with three blocks and 80 registers the
// loads no longer overlap: 1.4 times as long).
template <typename ST, int R, int MODE, int VW>
__global__ void __launch_bounds__(256, MODE == 2 && R == 1 ? 4 : 2) gather_kernel(GatherArgs a) {
    constexpr int VX = 16 / sizeof(ST), W1 = 2 * R + 1, NROW = W1 * W1, NV = VW * 32, G = 8 / VW;
    constexpr int NP = MODE == 0 ? 1 : VX / 2, NK = VX + 2 * R;
    using T = typename std::conditional<MODE == 0, double, float>::type;
    __shared__ T part[MODE == 0 ? 1 : 2][VX][256];

    const int t = threadIdx.x, group = t / NV;
    // (a plane of 2^31 vectors would be a cache of 27 x 32 GB and more: 32-bit positions will do)
    const unsigned v = blockIdx.x * NV + (t - group * NV);
    double acc[2] = {0.0, 0.0};                          // MODE 0
    uint64_t A[NP], B[NP];                               // MODE 1, 2: running double-float sums of two destinations
#pragma unroll
    for (int i = 0; i < NP; i++) A[i] = B[i] = 0;

    const unsigned nxv = a.qnx / VX, nvec = nxv * a.g.ny * a.zn;
    if (v < nvec) {
        const unsigned rw = v / nxv;
        const int x = (int)(v - rw * nxv) * VX, z = a.z0 + (int)(rw / a.g.ny), y = (int)(rw % a.g.ny);
        const int64_t at = ((int64_t)(z + R) * a.p.py + (y + R)) * a.p.px + x;     // of (ox, oy, oz) = (R, 0, 0)
        const int last = a.g.nx - 1 - x + 2 * R;             // no scaled value past the padded x row is read
        const int r0 = group * NROW / G, r1 = (group + 1) * NROW / G;
        int oz = r0 / W1 - R, oy = r0 % W1 - R;
        const ST* q = reinterpret_cast<const ST*>(a.Q) + (int64_t)r0 * W1 * a.qs + (int64_t)v * VX;
        for (int r = r0; r < r1; r++) {
            const int64_t row = at - ((int64_t)oz * a.p.py + oy) * a.p.px;
            if constexpr (MODE == 0) {
                const double* ch = reinterpret_cast<const double*>(a.chat) + row;
                double w[NK];
#pragma unroll
                for (int k = 0; k < NK; k++) w[k] = __ldg(ch + (k <= 2 * R ? k : min(k, last)));
#pragma unroll
                for (int ox = -R; ox <= R; ox++) {
                    const double2 d = __ldcs(reinterpret_cast<const double2*>(q + (int64_t)(ox + R) * a.qs));
                    acc[0] = fma(d.x, w[R - ox], acc[0]);
                    acc[1] = fma(d.y, w[R - ox + 1], acc[1]);
                }
            } else {
                uint64_t s[NP], c[NP];
#pragma unroll
                for (int i = 0; i < NP; i++) s[i] = c[i] = 0;
                uint4 d[W1];                                 // streamed: read once per step
#pragma unroll
                for (int k = 0; k < W1; k++) d[k] = __ldcs(reinterpret_cast<const uint4*>(q + (int64_t)k * a.qs));
                row_sums<ST, R, MODE == 1>(d, [&](int k) {
                    const int64_t at_k = row + (k <= 2 * R ? k : min(k, last));
                    if constexpr (MODE == 1) return __ldg(reinterpret_cast<const float2*>(a.chat) + at_k);
                    else return make_float2(__ldg(reinterpret_cast<const float*>(a.chat) + at_k), 0.f);
                }, s, c);
                // The pair of a row restarts at zero, so its compensation stays within a few ulps of the row sum.
#pragma unroll
                for (int i = 0; i < NP; i++) ff_add2(A[i], B[i], s[i], c[i]);
            }
            q += W1 * a.qs;
            if (++oy > R) { oy = -R; oz++; }
        }
    }
    if constexpr (G == 1) {                              // nothing to add up
        if (v >= nvec) return;
        const unsigned rw = v / nxv;
        const int x = (int)(v - rw * nxv) * VX;
        double* o = a.out + x + (int64_t)a.g.nx * ((int64_t)rw + (int64_t)a.g.ny * a.z0);
        float SA[VX], SB[VX];
        if constexpr (MODE != 0) {
#pragma unroll
            for (int i = 0; i < NP; i++) {
                unpack2(A[i], SA[Quad<ST>::j0(i)], SA[Quad<ST>::j0(i) + Quad<ST>::D]);
                unpack2(B[i], SB[Quad<ST>::j0(i)], SB[Quad<ST>::j0(i) + Quad<ST>::D]);
            }
        }
#pragma unroll
        for (int j = 0; j < VX; j++)
            if (x + j < a.g.nx) {
                if constexpr (MODE == 0) o[j] = acc[j];
                else o[j] = (a.acc_in ? o[j] : 0.0) + ((double)SA[j] + (double)SB[j]);
            }
        return;
    }
    if constexpr (MODE == 0) {
        part[0][0][t] = acc[0];
        part[0][1][t] = acc[1];
    } else {
        using U = Quad<ST>;
#pragma unroll
        for (int i = 0; i < NP; i++) {
            unpack2(A[i], part[0][U::j0(i)][t], part[0][U::j0(i) + U::D][t]);
            unpack2(B[i], part[1][U::j0(i)][t], part[1][U::j0(i) + U::D][t]);
        }
    }
    __syncthreads();
    // The groups' sums in ascending order, consecutive threads on consecutive destinations.
    for (int d = t; d < NV * VX; d += 256) {
        const int w = d / VX, j = d - w * VX;
        const unsigned u = blockIdx.x * NV + w, rw = u / nxv;
        const int x = (int)(u - rw * nxv) * VX + j;
        if (u >= nvec || x >= a.g.nx) continue;
        double* o = a.out + x + (int64_t)a.g.nx * ((int64_t)rw + (int64_t)a.g.ny * a.z0);
        if constexpr (MODE == 0) {
            double sum = part[0][j][w];
#pragma unroll
            for (int k = 1; k < G; k++) sum += part[0][j][k * NV + w];
            *o = sum;
        } else {
            float SA = part[0][j][w], SB = part[1][j][w];
#pragma unroll
            for (int k = 1; k < G; k++) ff_add(SA, SB, part[0][j][k * NV + w], part[1][j][k * NV + w]);
            *o = (a.acc_in ? *o : 0.0) + ((double)SA + (double)SB);
        }
    }
}

// FDIRW_ACCUM_FP32 at R >= 3: the same split of the rows, but one destination's rows are added in the order of one
// sequential sum, because the next step rounds its scaled field to FP32: a last bit of the FP64 result can flip that
// rounding, and 6e-8 of the value with it, so a result is kept to the bit whatever the split.  The 8 warps of a block
// take 8 consecutive rows at a time and leave their row sums in shared memory; then each thread adds the 8 sums of its
// own destinations.  The next row's cache values are loaded before that, so they arrive while the block meets.
template <typename ST, int R>
__global__ void __launch_bounds__(256, 2) gather_ordered_kernel(GatherArgs a) {
    using U = Quad<ST>;
    constexpr int VX = 16 / sizeof(ST), W1 = 2 * R + 1, NROW = W1 * W1, NP = VX / 2, ND = 32 * VX;
    __shared__ __align__(16) float sums[2][8][ND];      // stored 16 bytes at a time
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const unsigned nxv = a.qnx / VX, nvec = nxv * a.g.ny * a.zn, v = blockIdx.x * 32 + lane;
    const bool valid = v < nvec;
    const unsigned rw = valid ? v / nxv : 0;
    const int x = valid ? (int)(v - rw * nxv) * VX : 0, z = a.z0 + (int)(rw / a.g.ny), y = (int)(rw % a.g.ny);
    const int last = a.g.nx - 1 - x + 2 * R;             // no scaled value past the padded x row is read
    const float* chat = reinterpret_cast<const float*>(a.chat) + ((int64_t)(z + R) * a.p.py + (y + R)) * a.p.px + x;
    const ST* q = reinterpret_cast<const ST*>(a.Q) + (valid ? (int64_t)v * VX : 0);
    uint4 d[W1];
    auto fetch = [&](int row) {
        const ST* p = q + (int64_t)row * W1 * a.qs;
#pragma unroll
        for (int k = 0; k < W1; k++) d[k] = __ldcs(reinterpret_cast<const uint4*>(p + (int64_t)k * a.qs));
    };
    fetch(warp);
    float A = 0.f, B = 0.f;                              // of destination t (threads below ND)
    int buf = 0;
    for (int r0 = 0; r0 < NROW; r0 += 8, buf ^= 1) {
        const int row = r0 + warp;
        if (row < NROW) {
            const int oz = row / W1 - R, oy = row % W1 - R;
            const float* ch = chat - ((int64_t)oz * a.p.py + oy) * a.p.px;
            uint64_t s[NP], c[NP];
#pragma unroll
            for (int i = 0; i < NP; i++) s[i] = c[i] = 0;
            row_sums<ST, R, false>(d, [&](int k) { return make_float2(__ldg(ch + (k <= 2 * R ? k : min(k, last))), 0.f); }, s, c);
            if (row + 8 < NROW) fetch(row + 8);
            float f[VX];
#pragma unroll
            for (int i = 0; i < NP; i++) unpack2(s[i], f[U::j0(i)], f[U::j0(i) + U::D]);
#pragma unroll
            for (int j = 0; j < VX; j += 4)
                *reinterpret_cast<float4*>(&sums[buf][warp][lane * VX + j]) = make_float4(f[j], f[j + 1], f[j + 2], f[j + 3]);
        }
        __syncthreads();
        if (t < ND) {
#pragma unroll
            for (int k = 0; k < 8; k++)
                if (r0 + k < NROW) ff_add(A, B, sums[buf][k][t], 0.f);
        }
    }
    if (t >= ND) return;
    const unsigned u = blockIdx.x * 32 + t / VX, ru = u / nxv;
    const int dx = (int)(u - ru * nxv) * VX + t % VX;
    if (u >= nvec || dx >= a.g.nx) return;
    double* o = a.out + dx + (int64_t)a.g.nx * ((int64_t)ru + (int64_t)a.g.ny * a.z0);
    *o = (a.acc_in ? *o : 0.0) + ((double)A + (double)B);
}

// Rows of a width that is no whole number of vectors (nx < VX, or a padded cache that would not fit), and R = 1: one
// destination per thread, runtime R, the sums of gather_kernel in the same order.  Bound by the latency of its loads.  us a
// step of a 7 x 40 x 40 box, BF16 cache, R = 8: float-float sums 1100 (without the unrolling by two 1716), FP32 sums 980
// (1663 with the compiler's); R = 3 48 (55) and 34 (42).
template <typename ST, int MODE>
__global__ void __launch_bounds__(256) gather_scalar_kernel(GatherArgs a, int R) {
    const int64_t nxy = (int64_t)a.g.nx * a.g.ny;
    const int64_t tid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (tid >= nxy * a.zn) return;
    const int64_t rw = tid / a.g.nx;
    const int x = (int)(tid - rw * a.g.nx), y = (int)(rw % a.g.ny), z = a.z0 + (int)(rw / a.g.ny);
    const int W1 = 2 * R + 1, NROW = W1 * W1, G = MODE == 2 ? 1 : row_groups(R);
    double sum = 0.0;                                     // MODE 0
    float SA = 0.f, SB = 0.f;                             // MODE 1, 2
    const ST* q = reinterpret_cast<const ST*>(a.Q) + rw * a.qnx + x;
    int row = 0, oz = -R, oy = -R;
    for (int k = 0; k < G; k++) {
        double acc = 0.0;
        float A = 0.f, B = 0.f;
        for (; row < (k + 1) * NROW / G; row++) {
            const int64_t at = ((int64_t)(z - oz + R) * a.p.py + (y - oy + R)) * a.p.px + x + R;
            float s = 0.f, c = 0.f;
            if constexpr (MODE == 0) {
                for (int ox = -R; ox <= R; ox++, q += a.qs)
                    acc = fma((double)*q, reinterpret_cast<const double*>(a.chat)[at - ox], acc);
            } else if constexpr (MODE == 1) {
#pragma unroll 2
                for (int ox = -R; ox <= R; ox++, q += a.qs)
                    ff_madd(s, c, widen(*q), reinterpret_cast<const float2*>(a.chat)[at - ox]);
            } else {
#pragma unroll 4
                for (int ox = -R; ox <= R; ox++, q += a.qs)
                    s = fmaf(widen(*q), reinterpret_cast<const float*>(a.chat)[at - ox], s);
            }
            if constexpr (MODE != 0) ff_add(A, B, s, c);
            if (++oy > R) { oy = -R; oz++; }
        }
        if (k == 0) { sum = acc; SA = A; SB = B; }
        else if constexpr (MODE != 0) ff_add(SA, SB, A, B);
        else sum += acc;
    }
    double* o = a.out + a.z0 * nxy + tid;
    if constexpr (MODE != 0) *o = (a.acc_in ? *o : 0.0) + ((double)SA + (double)SB);
    else *o = sum;
}

__global__ void scale_kernel(const double* __restrict__ c, const double* __restrict__ sigma, Grid g, int R, Pad p,
                             void* __restrict__ chat, int mode, int64_t i0, int64_t i1) {
    for (int64_t i = i0 + blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < i1; i += (int64_t)gridDim.x * blockDim.x) {
        const int x = (int)(i % g.nx);
        const int64_t r = i / g.nx;
        const int y = (int)(r % g.ny);
        const int z = (int)(r / g.ny);
        const int64_t pi = ((int64_t)(z + R) * p.py + (y + R)) * p.px + (x + R);
        const double v = sigma[i] * c[i];
        if (mode == 1) {
            const float hi = (float)v;
            const float lo = (float)(v - (double)hi);
            reinterpret_cast<float2*>(chat)[pi] = make_float2(hi, lo);
        } else if (mode == 2) {
            reinterpret_cast<float*>(chat)[pi] = (float)v;
        } else {
            reinterpret_cast<double*>(chat)[pi] = v;
        }
    }
}

// Fixed-order FP64 reduction, pass 1: block b sums the contiguous chunk b (thread-strided, then a tree).
__global__ void __launch_bounds__(256) mass_partial_kernel(const double* __restrict__ c, int64_t n,
                                                           double* __restrict__ partials) {
    __shared__ double sh[8];
    const int64_t chunk = (n + gridDim.x - 1) / gridDim.x;
    const int64_t lo = blockIdx.x * chunk;
    const int64_t hi = lo + chunk < n ? lo + chunk : n;
    double acc = 0.0;
    for (int64_t i = lo + threadIdx.x; i < hi; i += blockDim.x) acc += c[i];
    for (int off = 16; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x < 32) {
        double v = threadIdx.x < (blockDim.x >> 5) ? sh[threadIdx.x] : 0.0;
        for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
        if (threadIdx.x == 0) partials[blockIdx.x] = v;
    }
}

// Pass 2: one block of kMassBlocks threads sums the partials.
__global__ void __launch_bounds__(kMassBlocks) mass_final_kernel(const double* __restrict__ partials,
                                                                 double* __restrict__ out) {
    __shared__ double sh[kMassBlocks / 32];
    double v = partials[threadIdx.x];
    for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x < 32) {
        double w = sh[threadIdx.x];
        for (int off = 16; off > 0; off >>= 1) w += __shfl_xor_sync(0xffffffffu, w, off);
        if (threadIdx.x == 0) *out = w;
    }
}

// Mass restoration, pass 1: block b sums c and |c| over the contiguous chunk b (as mass_partial_kernel).
__global__ void __launch_bounds__(256) mass_abs_partial_kernel(const double* __restrict__ c, int64_t n,
                                                               double* __restrict__ partials) {
    __shared__ double sh[2][8];
    const int64_t chunk = (n + gridDim.x - 1) / gridDim.x;
    const int64_t lo = blockIdx.x * chunk;
    const int64_t hi = lo + chunk < n ? lo + chunk : n;
    double acc = 0.0, aab = 0.0;
    for (int64_t i = lo + threadIdx.x; i < hi; i += blockDim.x) {
        const double v = c[i];
        acc += v;
        aab += fabs(v);
    }
    for (int off = 16; off > 0; off >>= 1) {
        acc += __shfl_xor_sync(0xffffffffu, acc, off);
        aab += __shfl_xor_sync(0xffffffffu, aab, off);
    }
    if ((threadIdx.x & 31) == 0) { sh[0][threadIdx.x >> 5] = acc; sh[1][threadIdx.x >> 5] = aab; }
    __syncthreads();
    if (threadIdx.x < 32) {
        double v = threadIdx.x < (blockDim.x >> 5) ? sh[0][threadIdx.x] : 0.0;
        double w = threadIdx.x < (blockDim.x >> 5) ? sh[1][threadIdx.x] : 0.0;
        for (int off = 16; off > 0; off >>= 1) {
            v += __shfl_xor_sync(0xffffffffu, v, off);
            w += __shfl_xor_sync(0xffffffffu, w, off);
        }
        if (threadIdx.x == 0) { partials[blockIdx.x] = v; partials[kMassBlocks + blockIdx.x] = w; }
    }
}

// Pass 2: one block sums both partial sets and writes f = (m_in - S) / A into fix[1] (0 when A = 0) and
// the running maximum of |m_in - S| / |m_in| into fix[2].
__global__ void __launch_bounds__(kMassBlocks) mass_fix_kernel(const double* __restrict__ partials,
                                                               double* __restrict__ fix) {
    __shared__ double sh[2][kMassBlocks / 32];
    double v = partials[threadIdx.x], w = partials[kMassBlocks + threadIdx.x];
    for (int off = 16; off > 0; off >>= 1) {
        v += __shfl_xor_sync(0xffffffffu, v, off);
        w += __shfl_xor_sync(0xffffffffu, w, off);
    }
    if ((threadIdx.x & 31) == 0) { sh[0][threadIdx.x >> 5] = v; sh[1][threadIdx.x >> 5] = w; }
    __syncthreads();
    if (threadIdx.x < 32) {
        double S = sh[0][threadIdx.x], A = sh[1][threadIdx.x];
        for (int off = 16; off > 0; off >>= 1) {
            S += __shfl_xor_sync(0xffffffffu, S, off);
            A += __shfl_xor_sync(0xffffffffu, A, off);
        }
        if (threadIdx.x == 0) {
            fix[1] = A > 0.0 ? (fix[0] - S) / A : 0.0;
            // largest relative drift of the FP32-accumulated totals before restoration since fix[2] was reset
            if (fix[0] != 0.0) fix[2] = fmax(fix[2], fabs(fix[0] - S) / fabs(fix[0]));
        }
    }
}

// Pass 3: c[i] += f |c[i]|.
__global__ void mass_apply_kernel(double* __restrict__ c, int64_t n, const double* __restrict__ fix) {
    const double f = fix[1];
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        c[i] = fma(f, fabs(c[i]), c[i]);
}

// Per-structure mass restoration of batch contexts: kSegBlocks blocks per structure, block p summing the
// p-th contiguous part of its cells (c and |c|); then one warp per structure sums the parts in order.
__global__ void __launch_bounds__(256) seg_sums_kernel(const double* __restrict__ c, const int64_t* __restrict__ base,
                                                       int s0, double* __restrict__ partials) {
    __shared__ double sh[2][8];
    const int i = s0 + (int)(blockIdx.x / kSegBlocks), part = (int)(blockIdx.x % kSegBlocks);
    const int64_t b0 = base[i], n = base[i + 1] - b0;
    const int64_t chunk = (n + kSegBlocks - 1) / kSegBlocks;
    const int64_t lo = b0 + part * chunk;
    const int64_t hi = lo + chunk < b0 + n ? lo + chunk : b0 + n;
    double acc = 0.0, aab = 0.0;
    for (int64_t j = lo + threadIdx.x; j < hi; j += blockDim.x) {
        const double v = c[j];
        acc += v;
        aab += fabs(v);
    }
    for (int off = 16; off > 0; off >>= 1) {
        acc += __shfl_xor_sync(0xffffffffu, acc, off);
        aab += __shfl_xor_sync(0xffffffffu, aab, off);
    }
    if ((threadIdx.x & 31) == 0) { sh[0][threadIdx.x >> 5] = acc; sh[1][threadIdx.x >> 5] = aab; }
    __syncthreads();
    if (threadIdx.x < 32) {
        double v = threadIdx.x < (blockDim.x >> 5) ? sh[0][threadIdx.x] : 0.0;
        double w = threadIdx.x < (blockDim.x >> 5) ? sh[1][threadIdx.x] : 0.0;
        for (int off = 16; off > 0; off >>= 1) {
            v += __shfl_xor_sync(0xffffffffu, v, off);
            w += __shfl_xor_sync(0xffffffffu, w, off);
        }
        if (threadIdx.x == 0) { partials[2 * blockIdx.x] = v; partials[2 * blockIdx.x + 1] = w; }
    }
}

// One warp per structure i in [s0, s0 + nseg): target == true stores its total in fix[2 i]; otherwise
// fix[2 i + 1] = (fix[2 i] - S_i) / A_i (0 when A_i = 0).
__global__ void seg_fix_kernel(const double* __restrict__ partials, int s0, int nseg, double* __restrict__ fix,
                               bool target) {
    const int w = (int)((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
    if (w >= nseg) return;
    static_assert(kSegBlocks == 32, "one part per lane");
    double S = partials[2 * (w * kSegBlocks + lane)], A = partials[2 * (w * kSegBlocks + lane) + 1];
    for (int off = 16; off > 0; off >>= 1) {
        S += __shfl_xor_sync(0xffffffffu, S, off);
        A += __shfl_xor_sync(0xffffffffu, A, off);
    }
    const int i = s0 + w;
    if (lane == 0) {
        if (target) fix[2 * i] = S;
        else fix[2 * i + 1] = A > 0.0 ? (fix[2 * i] - S) / A : 0.0;
    }
}

__global__ void __launch_bounds__(256) seg_apply_kernel(double* __restrict__ c, const int64_t* __restrict__ base, int s0,
                                                        const double* __restrict__ fix) {
    const int i = s0 + (int)(blockIdx.x / kSegBlocks), part = (int)(blockIdx.x % kSegBlocks);
    const int64_t b0 = base[i], n = base[i + 1] - b0;
    const int64_t chunk = (n + kSegBlocks - 1) / kSegBlocks;
    const int64_t lo = b0 + part * chunk;
    const int64_t hi = lo + chunk < b0 + n ? lo + chunk : b0 + n;
    const double f = fix[2 * i + 1];
    for (int64_t j = lo + threadIdx.x; j < hi; j += blockDim.x) c[j] = fma(f, fabs(c[j]), c[j]);
}

template <typename ST>
__global__ void read_kernels_kernel(const ST* __restrict__ Q, int64_t qs, int qnx, const double* __restrict__ sigma, Grid g, int R,
                                    const int64_t* __restrict__ sources, int64_t n_src, double* __restrict__ out) {
    const int W1 = 2 * R + 1;
    const int64_t W = (int64_t)W1 * W1 * W1;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n_src * W; t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t q = t / W;
        const int o = (int)(t % W);
        const int64_t s = sources[q];
        const int ox = o % W1 - R, oy = (o / W1) % W1 - R, oz = o / (W1 * W1) - R;
        const int sx = (int)(s % g.nx);
        const int64_t r = s / g.nx;
        const int sy = (int)(r % g.ny), sz = (int)(r / g.ny);
        const int x = sx + ox, y = sy + oy, z = sz + oz;
        double v = 0.0;
        if (x >= 0 && x < g.nx && y >= 0 && y < g.ny && z >= 0 && z < g.nz) {
            const int64_t i = x + (int64_t)qnx * (y + (int64_t)g.ny * z);
            v = (double)widen(Q[(int64_t)o * qs + i]) * sigma[s];
        }
        out[t] = v;
    }
}
template <>
__global__ void read_kernels_kernel<double>(const double* __restrict__ Q, int64_t qs, int qnx,
                                            const double* __restrict__ sigma, Grid g, int R, const int64_t* __restrict__ sources, int64_t n_src,
                                            double* __restrict__ out) {
    const int W1 = 2 * R + 1;
    const int64_t W = (int64_t)W1 * W1 * W1;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n_src * W; t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t q = t / W;
        const int o = (int)(t % W);
        const int64_t s = sources[q];
        const int ox = o % W1 - R, oy = (o / W1) % W1 - R, oz = o / (W1 * W1) - R;
        const int sx = (int)(s % g.nx);
        const int64_t r = s / g.nx;
        const int sy = (int)(r % g.ny), sz = (int)(r / g.ny);
        const int x = sx + ox, y = sy + oy, z = sz + oz;
        double v = 0.0;
        if (x >= 0 && x < g.nx && y >= 0 && y < g.ny && z >= 0 && z < g.nz) {
            const int64_t i = x + (int64_t)qnx * (y + (int64_t)g.ny * z);
            v = Q[(int64_t)o * qs + i] * sigma[s];
        }
        out[t] = v;
    }
}

int blocks_for(int64_t n, int threads) {
    int64_t b = (n + threads - 1) / threads;
    return (int)(b < 1 ? 1 : b);
}

// Below this many vectors an FP32 gather splits the rows (gather_ordered_kernel), from there on a thread sums its rows
// alone.  us, split / alone, BF16 cache: R = 8 64^3 (33k vectors) 455 / 522, 96^3 (111k) 1356 / 1501, 128^3 (262k) 3095 /
// 3133, 144^3 (373k) 4506 / 4134; R = 4 48^3 (14k) 49 / 86, 64^3 86 / 88, 96^3 242 / 213; R = 3 64^3 43 / 51, 96^3 121 / 117.
constexpr int64_t ordered_below(int R) { return R <= 5 ? 65536 : 300000; }

template <typename ST, int R, int MODE>
cudaError_t gather_launch(const GatherArgs& a, cudaStream_t st) {
    constexpr int VX = 16 / sizeof(ST);
    // FP32 sums come in one order whatever the kernel, so the split is free to follow the size of the launch.
    constexpr int VW = MODE == 2 ? 8 : vector_warps(R);
    const bool vec = a.qnx % VX == 0 && reinterpret_cast<uintptr_t>(a.Q) % 16 == 0 && a.qs % VX == 0;
    const int64_t n = (vec ? (int64_t)a.qnx / VX : (int64_t)a.g.nx) * a.g.ny * a.zn;
    if (n <= 0) return cudaSuccess;
    // R = 1 has no rows to split (vector_warps): so few vectors of eight destinations leave the GPU to a handful of warps,
    // and a thread a destination is faster (BF16 cache, float-float sums, us: 10 x 9 x 8 11.8 -> 9.9, 40^3 14.0 -> 9.8).
    if (!vec || (R == 1 && MODE == 1 && sizeof(ST) == 2 && n <= 8000)) {
        const int64_t cells = (int64_t)a.g.nx * a.g.ny * a.zn;
        gather_scalar_kernel<ST, MODE><<<(unsigned)blocks_for(cells, 256), 256, 0, st>>>(a, R);
        return cudaGetLastError();
    }
    if constexpr (MODE == 2 && R > 2) {
        if (n < ordered_below(R)) {
            gather_ordered_kernel<ST, R><<<(unsigned)((n + 31) / 32), 256, 0, st>>>(a);
            return cudaGetLastError();
        }
    }
    gather_kernel<ST, R, MODE, VW><<<(unsigned)((n + VW * 32 - 1) / (VW * 32)), 256, 0, st>>>(a);
    return cudaGetLastError();
}

template <typename ST, int MODE>
cudaError_t gather_radius(const GatherArgs& a, int R, cudaStream_t st) {
    switch (R) {
        case 1: return gather_launch<ST, 1, MODE>(a, st);
        case 2: return gather_launch<ST, 2, MODE>(a, st);
        case 3: return gather_launch<ST, 3, MODE>(a, st);
        case 4: return gather_launch<ST, 4, MODE>(a, st);
        case 5: return gather_launch<ST, 5, MODE>(a, st);
        case 6: return gather_launch<ST, 6, MODE>(a, st);
        case 7: return gather_launch<ST, 7, MODE>(a, st);
        case 8: return gather_launch<ST, 8, MODE>(a, st);
        default: break;
    }
    if constexpr (MODE != 0) {
        if (R == 9) return gather_launch<ST, 9, MODE>(a, st);
        if (R == 10) return gather_launch<ST, 10, MODE>(a, st);
    }
    return cudaErrorInvalidValue;
}

// The gather of one part (radius R, chat with a halo of Rp): mode 0 FP64, 1 float-float, 2 FP32.
cudaError_t gather_part(const void* Q, Store store, int64_t qs, int qnx, const void* chat, int Rp, Grid g, int R,
                        int mode, bool accumulate, double* c_out, cudaStream_t st, int z0, int zn) {
    if (R < 1 || R > Rp || qnx < g.nx || (mode == 0) != (store == Store::F64) || (mode == 0 && accumulate))
        return cudaErrorInvalidValue;
    const Pad p = make_pad(g, Rp);
    // The kernels index chat as if its halo were R: move the base by (Rp - R) on every axis.
    const int64_t shift = ((int64_t)(Rp - R) * p.py + (Rp - R)) * p.px + (Rp - R);
    const void* ch = static_cast<const char*>(chat) + shift * (mode == 2 ? 4 : 8);
    const GatherArgs a{Q, ch, g, p, qs, z0, zn, qnx, c_out, accumulate};
    switch (store) {
        case Store::F64: return gather_radius<double, 0>(a, R, st);
        case Store::F32: return mode == 1 ? gather_radius<float, 1>(a, R, st) : gather_radius<float, 2>(a, R, st);
        case Store::F16: return mode == 1 ? gather_radius<__half, 1>(a, R, st) : gather_radius<__half, 2>(a, R, st);
        case Store::BF16: return mode == 1 ? gather_radius<__nv_bfloat16, 1>(a, R, st) : gather_radius<__nv_bfloat16, 2>(a, R, st);
    }
    return cudaErrorInvalidValue;
}

}  // namespace

cudaError_t launch_scale(const double* c, const double* sigma, Grid g, int R, void* chat, int mode,
                         cudaStream_t st, int z0, int zn) {
    const Pad p = make_pad(g, R);
    const int64_t nxy = (int64_t)g.nx * g.ny;
    const int64_t i0 = (int64_t)z0 * nxy, i1 = zn < 0 ? g.n : (int64_t)(z0 + zn) * nxy;
    if (i1 <= i0) return cudaSuccess;
    int b = blocks_for(i1 - i0, 256);
    if (b > 152 * 16) b = 152 * 16;
    scale_kernel<<<b, 256, 0, st>>>(c, sigma, g, R, p, chat, mode, i0, i1);
    return cudaGetLastError();
}

cudaError_t launch_gather_part(const void* Q, Store store, int64_t qs, int qnx, const void* chat, int Rp, Grid g,
                               int R, int mode, bool accumulate, double* c_out, cudaStream_t st) {
    return gather_part(Q, store, qs, qnx, chat, Rp, g, R, mode, accumulate, c_out, st, 0, g.nz);
}

cudaError_t launch_gather_slab(const void* Q, Store store, int64_t qs, int qnx, const void* chat, Grid g, int R,
                               int mode, int z0, int zn, double* c_out, cudaStream_t st) {
    return gather_part(Q, store, qs, qnx, chat, R, g, R, mode, false, c_out, st, z0, zn);
}

cudaError_t launch_mass(const double* c, int64_t n, double* partials, double* out, cudaStream_t st) {
    mass_partial_kernel<<<kMassBlocks, 256, 0, st>>>(c, n, partials);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    mass_final_kernel<<<1, kMassBlocks, 0, st>>>(partials, out);
    return cudaGetLastError();
}

cudaError_t launch_seg_target(const double* c, const int64_t* base, int s0, int s1, double* partials, double* fix,
                              cudaStream_t st) {
    const int nseg = s1 - s0;
    if (nseg <= 0) return cudaSuccess;
    seg_sums_kernel<<<nseg * kSegBlocks, 256, 0, st>>>(c, base, s0, partials);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    seg_fix_kernel<<<(nseg * 32 + 255) / 256, 256, 0, st>>>(partials, s0, nseg, fix, true);
    return cudaGetLastError();
}

cudaError_t launch_seg_restore(double* c, const int64_t* base, int s0, int s1, double* partials, double* fix,
                               cudaStream_t st) {
    const int nseg = s1 - s0;
    if (nseg <= 0) return cudaSuccess;
    seg_sums_kernel<<<nseg * kSegBlocks, 256, 0, st>>>(c, base, s0, partials);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    seg_fix_kernel<<<(nseg * 32 + 255) / 256, 256, 0, st>>>(partials, s0, nseg, fix, false);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    seg_apply_kernel<<<nseg * kSegBlocks, 256, 0, st>>>(c, base, s0, fix);
    return cudaGetLastError();
}

cudaError_t launch_restore_mass(double* c, int64_t n, double* partials, double* fix, cudaStream_t st) {
    mass_abs_partial_kernel<<<kMassBlocks, 256, 0, st>>>(c, n, partials);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    mass_fix_kernel<<<1, kMassBlocks, 0, st>>>(partials, fix);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    int b = blocks_for(n, 256);
    if (b > 152 * 16) b = 152 * 16;
    mass_apply_kernel<<<b, 256, 0, st>>>(c, n, fix);
    return cudaGetLastError();
}

cudaError_t launch_read_kernels(const void* Q, Store store, int64_t qs, int qnx, const double* sigma, Grid g, int R,
                                const int64_t* sources, int64_t n_src, double* out, cudaStream_t st) {
    const int64_t W = (int64_t)(2 * R + 1) * (2 * R + 1) * (2 * R + 1);
    int b = blocks_for(n_src * W, 256);
    if (b > 152 * 16) b = 152 * 16;
    switch (store) {
        case Store::F64:
            read_kernels_kernel<double><<<b, 256, 0, st>>>(reinterpret_cast<const double*>(Q), qs, qnx, sigma, g, R, sources, n_src, out);
            break;
        case Store::F32:
            read_kernels_kernel<float><<<b, 256, 0, st>>>(reinterpret_cast<const float*>(Q), qs, qnx, sigma, g, R, sources, n_src, out);
            break;
        case Store::F16:
            read_kernels_kernel<__half><<<b, 256, 0, st>>>(reinterpret_cast<const __half*>(Q), qs, qnx, sigma, g, R, sources, n_src, out);
            break;
        case Store::BF16:
            read_kernels_kernel<__nv_bfloat16><<<b, 256, 0, st>>>(reinterpret_cast<const __nv_bfloat16*>(Q), qs, qnx, sigma, g, R,
                                                                   sources, n_src, out);
            break;
    }
    return cudaGetLastError();
}

}  // namespace fdirw
