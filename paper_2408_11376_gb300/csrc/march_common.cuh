// Helpers shared by the march kernels: where a source lies, where its values go, the rounding to the
// storage type, the kernel masses, Tensor Memory accesses and packed FP32 pairs.
#pragma once

#include "fdirw_internal.h"

#include <cuda_bf16.h>
#include <cuda_fp16.h>

namespace fdirw {

namespace {

// Plane of the kernel cache for window cell (x, y, k) of a radius-R window: the cache is laid out for
// radius a.Rq >= R (offset o = (x - R, y - R, k - R), plane (ox + Rq) + Wq ((oy + Rq) + Wq (oz + Rq))).
__device__ __forceinline__ int64_t qplane(const MarchArgs& a, int R, int x, int y, int k) {
    const int Wq = 2 * a.Rq + 1, d = a.Rq - R;
    return (int64_t)(x + d) + (int64_t)Wq * ((y + d) + (int64_t)Wq * (k + d));
}

// Structure holding a source: its dimensions and first global cell (a batch concatenates structures;
// a single grid is structure 0 with base 0).  s becomes the source's index within its structure.
// qbase, qnx: first column of the structure in a destination-indexed cache and the values that an x row takes there.
struct SrcLoc {
    int nx, ny, nz, qnx;
    int64_t base, qbase;
};
__device__ __forceinline__ SrcLoc locate(const MarchArgs& a, bool ok, int64_t& s) {
    SrcLoc L{a.g.nx, a.g.ny, a.g.nz, 0, 0, 0};
    if (ok && a.nstruct > 0) {
        int lo = 0, hi = a.nstruct - 1;               // last structure whose first cell is <= s
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (__ldg(a.s_base + mid) <= s) lo = mid; else hi = mid - 1;
        }
        const int4 d = __ldg(a.s_dims + lo);
        const int64_t b = __ldg(a.s_base + lo);
        L = SrcLoc{d.x, d.y, d.z, 0, b, a.s_qbase ? __ldg(a.s_qbase + lo) : 0};
        s -= L.base;
    }
    L.qnx = a.q_vec > 1 ? (L.nx + a.q_vec - 1) / a.q_vec * a.q_vec : L.nx;
    return L;
}

// Coordinates of cell s of a structure nx x ny x nz (32-bit division where it is enough).
__device__ __forceinline__ void split_cell(int64_t s, int nx, int ny, int& x, int& y, int& z) {
    if (s <= 0x7fffffff) {
        const unsigned v = (unsigned)s, r = v / (unsigned)nx;
        x = (int)(v - r * (unsigned)nx);
        z = (int)(r / (unsigned)ny);
        y = (int)(r - (unsigned)z * (unsigned)ny);
    } else {
        x = (int)(s % nx);
        const int64_t r = s / nx;
        y = (int)(r % ny);
        z = (int)(r / ny);
    }
}

// Column of the kernel cache for a stored value: that of destination cell (x, y, z) of the structure
// (destination-indexed layout) or the source's position in the launch's source range (source-indexed layout of the
// radius buckets).
__device__ __forceinline__ int64_t qcol(const MarchArgs& a, const SrcLoc& L, int x, int y, int z, int64_t pos) {
    return a.src_major ? pos - a.src_begin : L.qbase + x + (int64_t)L.qnx * (y + (int64_t)L.ny * (z - a.dest_z0));
}

// Rounds v to the storage type, writes it to Q[idx] and returns the stored value widened to float
// (exact for every storage type).  Q == nullptr: round only.
__device__ __forceinline__ float put(void* Q, Store st, int64_t idx, float v) {
    if (st == Store::F32) {
        if (Q) reinterpret_cast<float*>(Q)[idx] = v;
        return v;
    } else if (st == Store::F16) {
        const __half h = __float2half_rn(v);
        if (Q) reinterpret_cast<__half*>(Q)[idx] = h;
        return __half2float(h);
    } else {
        const __nv_bfloat16 b = __float2bfloat16_rn(v);
        if (Q) reinterpret_cast<__nv_bfloat16*>(Q)[idx] = b;
        return __bfloat162float(b);
    }
}

// Stores the march's value for destination (x, y, z) at `plane` (put), or, for a destination outside the streamed
// slab, only rounds it to the storage type (sigma still sums it).
__device__ __forceinline__ float store_q(const MarchArgs& a, const SrcLoc& L, int64_t plane, int x, int y, int z,
                                         int64_t pos, float v) {
    if (a.dest_z1 > a.dest_z0 && (z < a.dest_z0 || z >= a.dest_z1)) return put(nullptr, a.store, 0, v);
    return put(a.Q, a.store, plane * a.q_stride + qcol(a, L, x, y, z, pos), v);
}

// Kernel masses of the FP32 march: every stored value as a multiple of 2^-60 (exact above 2^-36, rounded to
// nearest below; a kernel's values are <= 1 and sum to about 1), summed as 64-bit integers.  The total is off
// by at most W 2^-61 (2e-15 for 17^3 values; 7e-17 for random roundings, an FP64 sum's 1e-16), it does not
// depend on the order of the sum, and it needs no FP64 instruction per value (1/73 of the FP32 rate here).
__device__ __forceinline__ int64_t mass_fix(float v) { return __float2ll_rn(v * 0x1p60f); }
// The same for a run of values without a conversion each (F2I runs at 1/8 of the FP32 rate): v + 6 leaves v's
// multiples of 2^-21 in the mantissa bits (|v| < 2; a rounded substep can leave a value an ulp below 0 or above 1),
// the exact rest + 1.5 2^-20 those of 2^-43, and the rest of that + 1.5 2^-37 those of 2^-60 (rounded to nearest,
// ties as mass_fix).  Up to 500 values.
struct MassSum {
    uint32_t s1 = 0, s2 = 0, s3 = 0, n = 0;
    __device__ __forceinline__ void add(float v) {
        const float t1 = __fadd_rn(v, 6.f), r1 = __fsub_rn(v, __fsub_rn(t1, 6.f));
        const float t2 = __fadd_rn(r1, 0x1.8p-20f), r2 = __fsub_rn(r1, __fsub_rn(t2, 0x1.8p-20f));
        const float t3 = __fadd_rn(r2, 0x1.8p-37f);
        s1 += __float_as_uint(t1);
        s2 += __float_as_uint(t2);
        s3 += __float_as_uint(t3);
        n++;
    }
    __device__ __forceinline__ int64_t total() const {
        return ((int64_t)(int32_t)(s1 - n * 0x40C00000u) << 39) + ((int64_t)(int32_t)(s2 - n * 0x35C00000u) << 17) +
               (int64_t)(int32_t)(s3 - n * 0x2D400000u);
    }
};
__device__ __forceinline__ double mass_of(int64_t m) { return (double)m * 0x1p-60; }
__device__ __forceinline__ double mass_of(double m) { return m; }

// sigma_s = 1 / (sum of the N partials of slot) for every slot of the batch (FP64 partials in a fixed order):
// warp w takes slots w, w + nwarps, ...; lane l sums partials l, l + 32, ...; then a xor-butterfly.  Z sets of
// partials lie ZSTRIDE apart.
template <int N, int SPB, int Z = 1, int ZSTRIDE = 0, typename T>
__device__ __forceinline__ void finish_sigma(const T* red, int64_t batch_first, int64_t src_end, const int64_t* list,
                                             double* sigma) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nwarps = blockDim.x >> 5;
    for (int slot = warp; slot < SPB; slot += nwarps) {
        T acc = 0;
        for (int z = 0; z < Z; z++)
            for (int c = lane; c < N; c += 32) acc += red[z * ZSTRIDE + slot * N + c];
        for (int off = 16; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
        const int64_t s = batch_first + slot;
        if (lane == 0 && s < src_end) sigma[list ? list[s] : s] = acc > 0 ? 1.0 / mass_of(acc) : 0.0;
    }
}

__device__ __forceinline__ void tm_st16(uint32_t a, const uint32_t* v) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};"
                 :: "r"(a), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]),
                    "r"(v[8]), "r"(v[9]), "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15]) : "memory");
}
__device__ __forceinline__ void tm_st8(uint32_t a, const uint32_t* v) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};"
                 :: "r"(a), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]) : "memory");
}
__device__ __forceinline__ void tm_st4(uint32_t a, const uint32_t* v) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1,%2,%3,%4};"
                 :: "r"(a), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]) : "memory");
}
__device__ __forceinline__ void tm_ld16(uint32_t a, uint32_t (&r)[16]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                   "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
                 : "r"(a));
}
__device__ __forceinline__ void tm_ld4(uint32_t a, uint32_t (&r)[4]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(a));
}
// 12 words: 8 at a8, 4 at a4.
template <int N>
__device__ __forceinline__ void tm_ld12(uint32_t a8, uint32_t a4, uint32_t (&r)[N]) {
    static_assert(N >= 12, "room for 12 words");
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(a8));
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]) : "r"(a4));
}
// Waits for every outstanding tcgen05.ld of the thread; the registers are in-out operands so that no
// use of them is scheduled before the wait.
__device__ __forceinline__ void tm_wait_ld(uint32_t (&r)[16]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                   "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15])
                 :: "memory");
}

__device__ __forceinline__ uint64_t f2pack(float lo, float hi) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ uint64_t u2pack(uint32_t lo, uint32_t hi) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "r"(lo), "r"(hi));
    return r;
}
__device__ __forceinline__ float f2lo(uint64_t v) { return __uint_as_float((uint32_t)(v & 0xffffffffull)); }
__device__ __forceinline__ float f2hi(uint64_t v) { return __uint_as_float((uint32_t)(v >> 32)); }
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

// Where the stored values of one source of a CTA batch go (written by the source's first thread, read by
// every thread of the CTA in the epilogue).
struct SlotInfo {
    SrcLoc L;
    int64_t pos;
    int sx, sy, sz, ok;
};

// The cache stores of a CTA's batch, one window column of one source per thread and round, the batch's sources fastest:
// they have adjacent destinations in a plane, so one warp store covers about 32 / SPB planes.  Along a column both
// addresses advance by a constant (a plane of the cache and one of the grid).  u(x, y, k, slot): the marched value.
template <int R, int SPB, int THREADS, typename F>
__device__ __forceinline__ void store_columns(const MarchArgs& a, const SlotInfo* sinfo, F u) {
    constexpr int W1 = 2 * R + 1;
    for (int e = threadIdx.x; e < W1 * W1 * SPB; e += THREADS) {
        const int c = e / SPB, sl = e - c * SPB, y = c / W1, x = c - y * W1;
        const SlotInfo si = sinfo[sl];
        const int cx = si.sx - R + x, cy = si.sy - R + y, z0 = si.sz - R;
        if (!si.ok || cx < 0 || cx >= si.L.nx || cy < 0 || cy >= si.L.ny) continue;
        int k0 = z0 < 0 ? -z0 : 0, k1 = si.L.nz - z0 < W1 ? si.L.nz - z0 : W1;      // levels in the domain
        if (a.dest_z1 > a.dest_z0) {               // slab of z-planes: only its levels are stored
            k0 = max(k0, a.dest_z0 - z0);
            k1 = min(k1, a.dest_z1 - z0);
        }
        const int64_t at = qplane(a, R, x, y, 0) * a.q_stride + qcol(a, si.L, cx, cy, z0, si.pos);   // of level 0
        const int64_t step = (qplane(a, R, 0, 0, 1) - qplane(a, R, 0, 0, 0)) * a.q_stride +
                             (a.src_major ? 0 : (int64_t)si.L.qnx * si.L.ny);
        if (a.store == Store::F32) {
            float* q = reinterpret_cast<float*>(a.Q) + at;
#pragma unroll
            for (int k = 0; k < W1; k++, q += step)
                if (k >= k0 && k < k1) *q = u(x, y, k, sl);
        } else {
            uint16_t* q = reinterpret_cast<uint16_t*>(a.Q) + at;
            const bool half = a.store == Store::F16;
#pragma unroll
            for (int k = 0; k < W1; k++, q += step)
                if (k >= k0 && k < k1) {
                    const float v = u(x, y, k, sl);
                    *q = half ? __half_as_ushort(__float2half_rn(v)) : __bfloat16_as_ushort(__float2bfloat16_rn(v));
                }
        }
    }
}

// Coarse epilogue (Eq. 11 applied to the marched units of the blocks list[first .. first + n)): S[d] = FP64 sum of the
// marched field over the liquid cells of block J + d inside the window (z, y, x order; u is 0 elsewhere), m =
// sum of S in a fixed order, and column J of P: Qc[d][J + d] = N_J S[d] / (m N_{J+d}), or S[d] / N_{J+d}
// when the phase has open faces (a.abnd) and the column keeps the mass that stays (0 where block J + d
// has no liquid).  Every thread of the CTA takes part; S (W1^3 + 1 doubles) follows red in shared memory and holds as
// many sources as fit, their sums side by side: one source after the other left most of the CTA waiting (30^3, B = 3,
// R = 2, 24 sources a CTA, 3 substeps: 140 us a build, with fewer sources a CTA 19 now).
// u(x, y, k, q) is the marched value of a window cell of source first + q (0 on cells that are not liquid).
template <int R, typename F>
__device__ __forceinline__ void coarse_epilogue(const MarchArgs& a, F u, double* S, int64_t first, int n) {
    constexpr int W1 = 2 * R + 1;
    const int B = a.coarse_B, Rc = a.coarse_Rc, Wc = 2 * Rc + 1, Wc3 = Wc * Wc * Wc, bh = (B - 1) / 2;
    const int nx = a.g.nx, ny = a.g.ny, nz = a.g.nz, cap = (W1 * W1 * W1 + 1) / (Wc3 + 1);
    auto bar = [] { asm volatile("bar.sync 0;" ::: "memory"); };   // met by both z parts of a split march, each in its own code
    for (int q0 = 0; q0 < n; q0 += cap) {
        const int m = min(cap, n - q0);
        // per threads a source; q >= m: no source's
        const int per = blockDim.x / m, q = threadIdx.x / per;
        const int64_t s = first + q0 + (q < m ? q : 0), J = a.list ? a.list[s] : s;
        int bx, by, bz;
        split_cell(J, a.ncx, a.ncy, bx, by, bz);
        const int sx = bx * B + bh, sy = by * B + bh, sz = bz * B + bh;
        for (int d = q < m ? threadIdx.x - q * per : Wc3; d < Wc3; d += per) {
            const int cx = bx + d % Wc - Rc, cy = by + (d / Wc) % Wc - Rc, cz = bz + d / (Wc * Wc) - Rc;
            const int x0 = max(max(cx * B, sx - R), 0), x1 = min(min(cx * B + B - 1, sx + R), nx - 1);
            const int y0 = max(max(cy * B, sy - R), 0), y1 = min(min(cy * B + B - 1, sy + R), ny - 1);
            const int z0 = max(max(cz * B, sz - R), 0), z1 = min(min(cz * B + B - 1, sz + R), nz - 1);
            double acc = 0.0;
            for (int z = z0; z <= z1; z++)
                for (int y = y0; y <= y1; y++)
                    for (int x = x0; x <= x1; x++)
                        acc += (double)u(x - (sx - R), y - (sy - R), z - (sz - R), q0 + q);
            S[q * (Wc3 + 1) + d] = acc;
        }
        bar();
        for (int w = threadIdx.x >> 5; w < m; w += blockDim.x >> 5) {
            double v = 0.0;
            for (int d = threadIdx.x & 31; d < Wc3; d += 32) v += S[w * (Wc3 + 1) + d];
            for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
            if ((threadIdx.x & 31) == 0) S[w * (Wc3 + 1) + Wc3] = v;
        }
        bar();
        const double mass = q < m ? S[q * (Wc3 + 1) + Wc3] : 0.0, NJ = (double)a.ccount[J];
        for (int d = q < m ? threadIdx.x - q * per : Wc3; d < Wc3; d += per) {
            const int cx = bx + d % Wc - Rc, cy = by + (d / Wc) % Wc - Rc, cz = bz + d / (Wc * Wc) - Rc;
            if (cx < 0 || cx >= a.ncx || cy < 0 || cy >= a.ncy || cz < 0 || cz >= a.ncz) continue;
            const int64_t I = cx + (int64_t)a.ncx * (cy + (int64_t)a.ncy * cz);
            const int NI = a.ccount[I];
            const double part = S[q * (Wc3 + 1) + d];
            // Closed phase: renormalise the column to carry N_J; open faces: keep the mass that stays.
            double v = 0.0;
            if (NI > 0 && mass > 0.0) v = a.abnd ? part / (double)NI : (NJ * part) / (mass * (double)NI);
            a.Qc[(int64_t)d * a.coarse_n + I] = v;
        }
        bar();                                             // S is free again (and with the last one the marched values)
    }
}

}  // namespace

}  // namespace fdirw
