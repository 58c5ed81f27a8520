// Per-source windowed explicit FD march (Sec. 3.1: column s of p is the explicit-FD solution from a
// unit point source at s) and FP64 renormalisation of the stored kernel.
//
// Work decomposition (persistent grid, batches of SPB sources per CTA):
//   - one thread per z-column (ci, cj) of a source's (2R+1)^3 window; the column's 2R+1 cells live in
//     registers for the whole march;
//   - the FP32 path also keeps the 6 face coefficients of each cell in registers (they are constant over
//     the march), so a substep costs 1 MUL + 6 FMA + 1 ADD per cell; the z neighbours are in the same thread and
//     the x/y neighbours are read from a double-buffered shared-memory copy of every column (one
//     __syncthreads per substep);
//   - the FP64 path (the plain FP64 baseline) keeps u and the diagonal in registers and the face
//     coefficients in shared memory (FP64 registers would not fit), same exchange scheme, on the part of the window
//     that lies in the domain;
//   - after the march each thread rounds its cells to the storage type, writes them into the
//     destination-indexed cache Q[o][s + o] and sums the stored values (FP32 path: as 64-bit integers, FP64
//     path: in FP64 in a fixed order); sigma_s = 1 / sum.
// The mapping that runs unless a caller forces another one (2x2 column blocks) is in march_tm.cu.
// Window cells outside the domain carry no coefficients, so they stay 0; faces leaving the window or
// the domain have coefficient 0 (zero flux).  Bound: FP32 pipe + shared-memory bandwidth (FP32 path),
// FP64 pipe (FP64 path).  HBM traffic is only the coefficient loads (L2-resident) and the cache writes.
#include "fdirw_internal.h"
#include "march_common.cuh"

namespace fdirw {

namespace {

template <int R>
struct Shape {
    static constexpr int W1 = 2 * R + 1;
    static constexpr int COLS = W1 * W1;
    static constexpr int W = W1 * W1 * W1;
    static constexpr int SPB = (512 / COLS) > 0 ? (512 / COLS) : 1;
    // FP64 path: 2 exchange buffers + 3 face arrays of SPB*W doubles must fit in ~200 KB.
    static constexpr int SPB64_CAP = 200000 / (5 * W * 8);
    static constexpr int SPB64 = SPB64_CAP < 1 ? 1 : (SPB64_CAP < SPB ? SPB64_CAP : SPB);
    static constexpr int THREADS64 = ((SPB64 * COLS + 31) / 32) * 32;
};

// FP32 path thread mapping: P threads per window z-column, each owning KS consecutive cells.
template <int R, int P>
struct Map32 {
    static constexpr int W1 = 2 * R + 1;
    static constexpr int COLS = W1 * W1;
    static constexpr int KS = (W1 + P - 1) / P;
    static constexpr int TPS = P * COLS;                       // threads per source
    static constexpr int SPB = (512 / TPS) > 0 ? (512 / TPS) : 1;    // sources per CTA
    static constexpr int THREADS = ((SPB * TPS + 31) / 32) * 32;
    // Split mappings aim at ~1024 resident threads per SM; the single-column mapping needs the
    // registers of a whole SM for one CTA (6 coefficients + state per cell, 2R+1 cells per thread).
    static constexpr int MIN_BLOCKS = P == 1 ? 1 : ((1024 / THREADS) > 0 ? 1024 / THREADS : 1);
    static constexpr int BUF = SPB * COLS * W1;                // floats per exchange buffer
    static constexpr size_t SMEM = (size_t)((2 * BUF * 4 + 15) / 16) * 16 + (size_t)SPB * COLS * 8;
};

template <int R, int P>
__global__ void __launch_bounds__(Map32<R, P>::THREADS, Map32<R, P>::MIN_BLOCKS) march_f32_kernel(MarchArgs a) {
    using M = Map32<R, P>;
    constexpr int W1 = M::W1, COLS = M::COLS, KS = M::KS, TPS = M::TPS, SPB = M::SPB, BUF = M::BUF;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float* xbuf = reinterpret_cast<float*>(smem_raw);                                  // [2][SPB*COLS][W1]
    int64_t* red = reinterpret_cast<int64_t*>(smem_raw + ((2 * BUF * 4 + 15) / 16) * 16);  // [SPB*COLS]

    const int t = threadIdx.x;
    const bool active = t < SPB * TPS;
    const int slot = active ? t / TPS : 0;
    const int rr = active ? t - slot * TPS : 0;
    const int part = rr / COLS;
    const int col = rr - part * COLS;
    const int ci = col % W1, cj = col / W1;
    const int k0 = part * KS;                                  // first own cell of the column
    const int kn = (W1 - k0) < KS ? (W1 - k0) : KS;            // number of own cells
    const int64_t nbatch = (a.src_end - a.src_begin + SPB - 1) / SPB;

    const int base = (slot * COLS + col) * W1;
    const int xm = ci > 0 ? base - W1 : base;
    const int xp = ci < 2 * R ? base + W1 : base;
    const int ym = cj > 0 ? base - W1 * W1 : base;
    const int yp = cj < 2 * R ? base + W1 * W1 : base;
    const int kbelow = k0 > 0 ? k0 - 1 : k0;                   // cell read for the -z face of cell k0
    const int kabove = k0 + kn < W1 ? k0 + kn : k0;            // cell read for the +z face of the last cell

    for (int64_t b = blockIdx.x; b < nbatch; b += gridDim.x) {
        const int64_t first = a.src_begin + b * SPB;
        int64_t s = first + slot;
        const bool src_ok = active && s < a.src_end;
        if (src_ok && a.list) s = a.list[s];       // explicit source list (e.g. the surrogate's rejects)
        const int64_t pos = first + slot;                     // position of the source in the launch range
        const SrcLoc L = locate(a, src_ok, s);
        const int nx = L.nx, ny = L.ny, nz = L.nz;
        const int64_t nxy = (int64_t)nx * ny;
        const float* ax = a.ax + L.base;   // coefficients of the source's structure
        const float* ay = a.ay + L.base;
        const float* az = a.az + L.base;
        int sx = 0, sy = 0, sz = 0;
        if (src_ok) {
            sx = (int)(s % nx);
            const int64_t r = s / nx;
            sy = (int)(r % ny);
            sz = (int)(r / ny);
        }
        const int x = sx - R + ci, y = sy - R + cj;
        const bool col_ok = src_ok && x >= 0 && x < nx && y >= 0 && y < ny;

        // am = -(sum of the cell's face coefficients): the update is u += am*u + sum c*u_nb, i.e. the
        // increment is formed at full FP32 relative precision before it is added (1 - sum c rounded
        // once would bias near-delta kernels by half an ulp of 1 every substep).
        // cz[j] is the +z face of own cell j; czb is the -z face of own cell 0.
        float u[KS], am[KS], cxm[KS], cxp[KS], cym[KS], cyp[KS], cz[KS];
        float czb = 0.f;
#pragma unroll
        for (int j = 0; j < KS; j++) {
            const int k = k0 + j;
            const int z = sz - R + k;
            const bool ok = col_ok && j < kn && z >= 0 && z < nz;
            float vxm = 0.f, vxp = 0.f, vym = 0.f, vyp = 0.f, vz = 0.f;
            if (ok) {
                const int64_t i = (int64_t)x + (int64_t)nx * y + nxy * z;
                if (ci > 0 && x > 0) vxm = __ldg(ax + i - 1);
                if (ci < 2 * R && x + 1 < nx) vxp = __ldg(ax + i);
                if (cj > 0 && y > 0) vym = __ldg(ay + i - nx);
                if (cj < 2 * R && y + 1 < ny) vyp = __ldg(ay + i);
                if (k < 2 * R && z + 1 < nz) vz = __ldg(az + i);
                if (j == 0 && k > 0 && z > 0) czb = __ldg(az + i - nxy);
            }
            cxm[j] = vxm; cxp[j] = vxp; cym[j] = vym; cyp[j] = vyp; cz[j] = vz;
            u[j] = (src_ok && ci == R && cj == R && k == R) ? 1.f : 0.f;
        }
#pragma unroll
        for (int j = 0; j < KS; j++) {
            const float zm = j > 0 ? cz[j - 1] : czb;
            am[j] = -(((cxm[j] + cxp[j]) + (cym[j] + cyp[j])) + (zm + cz[j]));
        }

        for (int it = 0; it < a.n_sub; it++) {
            float* buf = xbuf + (it & 1) * BUF;
            if (active) {
#pragma unroll
                for (int j = 0; j < KS; j++)
                    if (j < kn) buf[base + k0 + j] = u[j];
            }
            __syncthreads();
            float prev = buf[base + kbelow];        // z-neighbour below own cell 0 (coefficient 0 if none)
            const float next_last = buf[base + kabove];
#pragma unroll
            for (int j = 0; j < KS; j++) {
                if (j < kn) {                      // the last part of a column may own fewer cells
                    const float cur = u[j];
                    const int k = k0 + j;
                    float v = am[j] * cur;
                    v = fmaf(cxm[j], buf[xm + k], v);
                    v = fmaf(cxp[j], buf[xp + k], v);
                    v = fmaf(cym[j], buf[ym + k], v);
                    v = fmaf(cyp[j], buf[yp + k], v);
                    v = fmaf(j > 0 ? cz[j - 1] : czb, prev, v);
                    v = fmaf(cz[j], (j + 1 < KS) ? (j + 1 < kn ? u[j + 1] : next_last) : next_last, v);
                    prev = cur;
                    u[j] = __fadd_rn(cur, v);
                }
            }
        }

        // Epilogue: round to storage and write Q[o][x] (x = s + o, the cell itself); the stored values
        // (exact in FP32) go back to shared memory so that each column is summed in k order by one
        // thread, whatever P is.
        float* sbuf = xbuf + (a.n_sub & 1) * BUF;   // not the buffer the last substep read
        if (active) {
#pragma unroll
            for (int j = 0; j < KS; j++) {
                if (j < kn) {
                    const int k = k0 + j;
                    const int z = sz - R + k;
                    float st = 0.f;
                    if (col_ok && z >= 0 && z < nz) st = store_q(a, L, qplane(a, R, ci, cj, k), x, y, z, pos, u[j]);
                    sbuf[base + k] = st;
                }
            }
        }
        __syncthreads();
        for (int c = t; c < SPB * COLS; c += blockDim.x) {
            int64_t colsum = 0;
#pragma unroll
            for (int k = 0; k < W1; k++) colsum += mass_fix(sbuf[c * W1 + k]);
            red[c] = colsum;
        }
        __syncthreads();
        finish_sigma<COLS, SPB>(red, first, a.src_end, a.list, a.sigma);
        __syncthreads();   // red and xbuf are reused by the next batch
    }
}

// The FP64 march.  Bound by the FP64 pipe (1/73 of the FP32 rate), so it computes no cell it need not: the threads of a
// batch are dealt out over the window columns that lie in the domain (the first threads to the first source's columns, and
// so on; warps past the last one idle), a column runs over its levels in the domain, and during the first substeps over
// those the source has reached (a substep moves a value one cell: |dx| + |dy| + |dz| <= substeps; the rest is still 0).
// The cells that are computed see the same operations in the same order.  36^3, R = 6, 120 substeps: 148 -> 114 ms; 20^3,
// R = 8, 60 substeps: 31.0 -> 15.7 ms; 64^3, R = 6, 30 substeps: 217 -> 176 ms.
// ALL: a thread a column and every level of it, in the domain or not.  The three levels of R = 1 are not worth their
// bounds (40 x 33 x 29, 60 substeps: 843 us with them, 790 without).
template <int R>
__global__ void __launch_bounds__(Shape<R>::THREADS64, 1) march_f64_kernel(MarchArgs a) {
    using S = Shape<R>;
    constexpr int W1 = S::W1, COLS = S::COLS, SPB = S::SPB64;
    constexpr bool ALL = R == 1;
    constexpr int BUF = SPB * COLS * W1;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double* xbuf = reinterpret_cast<double*>(smem_raw);   // [2][BUF]
    double* fx = xbuf + 2 * BUF;                           // +x face coefficient of each window cell
    double* fy = fx + BUF;                                 // +y
    double* fz = fy + BUF;                                 // +z
    double* red = fz + BUF;                                // [SPB*COLS]
    // Window of each source of the batch within the domain: first window column and widths, levels [k0, k1), threads
    // before it.
    __shared__ int c0x[SPB], c0y[SPB], wx[SPB], wxy[SPB], k0s[SPB], k1s[SPB], src[SPB][3], before[SPB + 1];

    const int t = threadIdx.x;
    const int nx = a.g.nx, ny = a.g.ny, nz = a.g.nz;
    const int64_t nxy = (int64_t)nx * ny;
    int64_t none = 0;
    const SrcLoc L = locate(a, false, none);
    const int64_t nbatch = (a.src_end - a.src_begin + SPB - 1) / SPB;

    // Columns outside the domain are not written: what lies there meets zero faces and has to be finite.
    for (int i = t; i < 2 * BUF; i += blockDim.x) xbuf[i] = 0.0;

    for (int64_t b = blockIdx.x; b < nbatch; b += gridDim.x) {
        const int64_t first = a.src_begin + b * SPB;
        bool own = false;
        int slot = 0, ci = 0, cj = 0, sx = 0, sy = 0, sz = 0, d0 = 0, d1 = 0;    // [d0, d1): levels in the domain
        if constexpr (ALL) {
            if (t < SPB * COLS) {
                slot = t / COLS;
                cj = (t - slot * COLS) / W1;
                ci = t - slot * COLS - cj * W1;
                int64_t s = first + slot;
                if (s < a.src_end) {
                    if (a.list) s = a.list[s];
                    split_cell(s, nx, ny, sx, sy, sz);
                    own = (unsigned)(sx - R + ci) < (unsigned)nx && (unsigned)(sy - R + cj) < (unsigned)ny;
                    d0 = own ? max(R - sz, 0) : 0;
                    d1 = own ? min(nz - 1 - sz, R) + R + 1 : 0;
                }
            }
        } else {
            if (t < SPB) {
                int64_t s = first + t;
                int n = 0;
                if (s < a.src_end) {
                    if (a.list) s = a.list[s];         // explicit source list (e.g. the surrogate's rejects)
                    int sx, sy, sz;
                    split_cell(s, nx, ny, sx, sy, sz);
                    c0x[t] = max(R - sx, 0);
                    c0y[t] = max(R - sy, 0);
                    wx[t] = min(nx - 1 - sx, R) + R - c0x[t] + 1;
                    k0s[t] = max(R - sz, 0);
                    k1s[t] = min(nz - 1 - sz, R) + R + 1;
                    src[t][0] = sx; src[t][1] = sy; src[t][2] = sz;
                    n = wx[t] * (min(ny - 1 - sy, R) + R - c0y[t] + 1);
                }
                wxy[t] = n;
            }
            __syncthreads();
            if (t <= SPB) {
                int n = 0;
#pragma unroll 8
                for (int q = 0; q < t; q++) n += wxy[q];
                before[t] = n;
            }
            for (int i = t; i < SPB * COLS; i += blockDim.x) red[i] = 0.0;
            __syncthreads();
            own = t < before[SPB];
            slot = own ? t / COLS : 0;                           // no source has more than COLS columns
            while (own && t >= before[slot + 1]) slot++;
            const int c = own ? t - before[slot] : 0, w = own ? wx[slot] : 1;
            cj = own ? c0y[slot] + c / w : 0;
            ci = own ? c0x[slot] + c % w : 0;
            sx = src[slot][0];
            sy = src[slot][1];
            sz = src[slot][2];
            d0 = own ? k0s[slot] : 0;
            d1 = own ? k1s[slot] : 0;
        }
        const int base = (slot * COLS + cj * W1 + ci) * W1;
        const int x = sx - R + ci, y = sy - R + cj;
        const int k0 = ALL ? 0 : d0, k1 = ALL ? W1 : d1;                 // levels that are computed
        const bool left = ci > 0 && x > 0, front = cj > 0 && y > 0;      // a lower neighbour in the window and the domain
        const int xm = left ? base - W1 : base, xp = ci < 2 * R ? base + W1 : base;
        const int ym = front ? base - W1 * W1 : base, yp = cj < 2 * R ? base + W1 * W1 : base;

        double u[W1];
#pragma unroll
        for (int k = 0; k < W1; k++) {
            u[k] = own && ci == R && cj == R && k == R ? 1.0 : 0.0;
            if (ALL ? own : k >= k0 && k < k1) {
                const int z = sz - R + k;
                const int64_t i = (int64_t)x + (int64_t)nx * y + nxy * z;
                const bool in = !ALL || (k >= d0 && k < d1);
                fx[base + k] = in && ci < 2 * R && x + 1 < nx ? __ldg(a.dx + i) : 0.0;
                fy[base + k] = in && cj < 2 * R && y + 1 < ny ? __ldg(a.dy + i) : 0.0;
                fz[base + k] = in && k < 2 * R && z + 1 < nz ? __ldg(a.dz + i) : 0.0;
            }
        }
        __syncthreads();
        double a0[W1];
#pragma unroll
        for (int k = 0; k < W1; k++) {
            a0[k] = 0.0;
            if (k >= k0 && k < k1) {
                const double vxm = left ? fx[xm + k] : 0.0;
                const double vym = front ? fy[ym + k] : 0.0;
                const double vzm = k > k0 ? fz[base + k - 1] : 0.0;
                a0[k] = 1.0 - (((vxm + fx[base + k]) + (vym + fy[base + k])) + (vzm + fz[base + k]));
            }
        }

        const int lateral = abs(ci - R) + abs(cj - R);
        for (int it = 0; it < a.n_sub; it++) {
            double* buf = xbuf + (it & 1) * BUF;
            if (!ALL || own)
#pragma unroll
                for (int k = 0; k < W1; k++)
                    if (k >= k0 && k < k1) buf[base + k] = u[k];
            __syncthreads();
            if (ALL && !own) continue;
            const int reach = it + 1 - lateral;                  // levels reached by the end of this substep
            const int ka = ALL ? 0 : max(k0, R - reach), kb = ALL ? W1 : min(k1, R + reach + 1);
            double prev = 0.0;
#pragma unroll
            for (int k = 0; k < W1; k++) {
                if (k < ka || k >= kb) continue;
                const double cur = u[k];
                double v = a0[k] * cur;
                if (left) v = fma(fx[xm + k], buf[xm + k], v);
                v = fma(fx[base + k], buf[xp + k], v);
                if (front) v = fma(fy[ym + k], buf[ym + k], v);
                v = fma(fy[base + k], buf[yp + k], v);
                if (k > k0) v = fma(fz[base + k - 1], prev, v);
                if (k + 1 < W1) v = fma(fz[base + k], u[k + 1 < W1 ? k + 1 : k], v);
                prev = cur;
                u[k] = v;
            }
        }

        double colsum = 0.0;
#pragma unroll
        for (int k = 0; k < W1; k++) {
            if (k < d0 || k >= d1) continue;
            const int z = sz - R + k;
            if (a.dest_z1 <= a.dest_z0 || (z >= a.dest_z0 && z < a.dest_z1))
                reinterpret_cast<double*>(a.Q)[qplane(a, R, ci, cj, k) * a.q_stride + qcol(a, L, x, y, z, 0)] = u[k];
            colsum += u[k];
        }
        if (ALL ? t < SPB * COLS : own) red[slot * COLS + cj * W1 + ci] = own ? colsum : 0.0;
        __syncthreads();
        finish_sigma<COLS, SPB>(red, first, a.src_end, a.list, a.sigma);
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------------------------------
// Column pairs with TMEM-resident faces and diagonals (mapping id 7; any R <= 10, made for R = 9, 10).
//
// Each thread owns two x-adjacent window columns (2 (2R+1) cells; the last pair of a window row is half
// padding), so the halo it exchanges through shared memory per substep is 4 words per cell (its two new
// values, the outer x neighbours and the y neighbours of both columns) instead of 5.  The 7 lateral faces
// of a pair's level (3 x, 4 y) and its 2 diagonals live in the thread's TMEM lane (8 + 1 words, loaded one
// level ahead); u and the z faces stay in registers, which leaves room below the register cap of a
// 256-thread CTA at R = 10 (mapping 5 runs 448 threads there and spills under a 128-register cap).  One
// CTA of 256 threads per SM, two threads per TMEM lane; the FP32 operations and their order are those of
// march_f32_kernel, so the results are bitwise those of every other mapping.
template <int R>
struct MapTmx {
    static constexpr int W1 = 2 * R + 1;
    static constexpr int COLS = W1 * W1;
    static constexpr int NBX = R + 1;                     // column pairs per window row
    static constexpr int TPS = NBX * W1;                  // threads per source
    static constexpr int THREADS = 256;
    static constexpr int SPB = THREADS / TPS;
    static constexpr int LEVEL = 2 * THREADS;             // floats per level: [sub-column][thread]
    static constexpr int BUF = W1 * LEVEL;
    static constexpr size_t SMEM_USED = (size_t)2 * BUF * 4 + (size_t)SPB * COLS * 8;
    static constexpr size_t SMEM = SMEM_USED > 120 * 1024 ? SMEM_USED : 120 * 1024;
    static_assert(SPB >= 1 && 9 * W1 <= 256, "a source must fit a CTA and its coefficients 256 TMEM columns");
};

__device__ __forceinline__ void tm_st1(uint32_t a, uint32_t v) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x1.b32 [%0], {%1};" :: "r"(a), "r"(v) : "memory");
}
// The 9 words of a pair's level: 8 at a8, 1 at a1.
__device__ __forceinline__ void tm_ld9(uint32_t a8, uint32_t a1, uint32_t (&r)[9]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(a8));
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x1.b32 {%0}, [%1];" : "=r"(r[8]) : "r"(a1));
}
__device__ __forceinline__ void tm_wait_ld9(uint32_t (&r)[9]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                   "+r"(r[8]) :: "memory");
}

template <int R>
__global__ void __launch_bounds__(MapTmx<R>::THREADS, 1) march_tmx_kernel(MarchArgs a) {
    using M = MapTmx<R>;
    constexpr int W1 = M::W1, COLS = M::COLS, NBX = M::NBX, TPS = M::TPS, SPB = M::SPB;
    constexpr int LEVEL = M::LEVEL, PLANE = M::THREADS, BUF = M::BUF;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float* xbuf = reinterpret_cast<float*>(smem_raw);                         // [2][W1][2][256]
    int64_t* red = reinterpret_cast<int64_t*>(smem_raw + (size_t)2 * BUF * 4);  // [SPB*COLS]
    __shared__ uint32_t s_taddr;

    const int t = threadIdx.x;
    const int warp = t >> 5;
    if (warp == 0) {
        const uint32_t dst = (uint32_t)__cvta_generic_to_shared(&s_taddr);
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" :: "r"(dst) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t taddr = s_taddr;
    const uint32_t tbase = taddr + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)(256 * (warp >> 2));
    const uint32_t regA = tbase, regB = tbase + (uint32_t)(8 * W1);      // level k: 8 words at 8k, 1 at 8 W1 + k

    const bool active = t < SPB * TPS;
    const int slot = active ? t / TPS : 0;
    const int b = active ? t - slot * TPS : 0;
    const int bi = b % NBX, bj = b / NBX;
    const int tl = (active && bi > 0) ? t - 1 : t;
    const int tr = (active && bi < NBX - 1) ? t + 1 : t;
    const int tb = (active && bj > 0) ? t - NBX : t;
    const int tt = (active && bj < W1 - 1) ? t + NBX : t;
    const int64_t nbatch = (a.src_end - a.src_begin + SPB - 1) / SPB;

    for (int64_t bt = blockIdx.x; bt < nbatch; bt += gridDim.x) {
        const int64_t first = a.src_begin + bt * SPB;
        int64_t s = first + slot;
        const bool src_ok = active && s < a.src_end;
        if (src_ok && a.list) s = a.list[s];
        const int64_t pos = first + slot;
        const SrcLoc L = locate(a, src_ok, s);
        const int nx = L.nx, ny = L.ny, nz = L.nz;
        const int64_t nxy = (int64_t)nx * ny;
        const float* ax = a.ax + L.base;
        const float* ay = a.ay + L.base;
        const float* az = a.az + L.base;
        int sx = 0, sy = 0, sz = 0;
        if (src_ok) {
            sx = (int)(s % nx);
            const int64_t r = s / nx;
            sy = (int)(r % ny);
            sz = (int)(r / ny);
        }
        auto cell_ok = [&](int x, int y, int k) -> bool {
            const int gx = sx - R + x, gy = sy - R + y, gz = sz - R + k;
            return src_ok && x >= 0 && x < W1 && y >= 0 && y < W1 && k >= 0 && k < W1 &&
                   gx >= 0 && gx < nx && gy >= 0 && gy < ny && gz >= 0 && gz < nz;
        };
        auto gidx = [&](int x, int y, int k) -> int64_t {
            return (int64_t)(sx - R + x) + (int64_t)nx * (sy - R + y) + nxy * (sz - R + k);
        };
        auto xface = [&](int x, int y, int k) -> float {
            return (x + 1 < W1 && cell_ok(x, y, k) && sx - R + x + 1 < nx) ? __ldg(ax + gidx(x, y, k)) : 0.f;
        };
        auto yface = [&](int x, int y, int k) -> float {
            return (y + 1 < W1 && cell_ok(x, y, k) && sy - R + y + 1 < ny) ? __ldg(ay + gidx(x, y, k)) : 0.f;
        };
        auto zface = [&](int x, int y, int k) -> float {
            return (k + 1 < W1 && cell_ok(x, y, k) && sz - R + k + 1 < nz) ? __ldg(az + gidx(x, y, k)) : 0.f;
        };

        // Sub-column sc at window (2 bi + sc, bj): state u[sc][k] and +z faces cz[sc][k] in registers.
        float u[2][W1], cz[2][W1];
#pragma unroll
        for (int sc = 0; sc < 2; sc++) {
            const int x = 2 * bi + sc, y = bj;
#pragma unroll
            for (int k = 0; k < W1; k++) {
                cz[sc][k] = zface(x, y, k);
                u[sc][k] = (src_ok && x == R && y == R && k == R) ? 1.f : 0.f;
            }
        }
#pragma unroll
        for (int k = 0; k < W1; k++) {
            const int x0 = 2 * bi, y = bj;
            float f[9];
            f[0] = bi > 0 ? xface(x0 - 1, y, k) : 0.f;        // -x face of sub-column 0
            f[1] = xface(x0, y, k);                            // between the two sub-columns
            f[2] = xface(x0 + 1, y, k);                        // +x face of sub-column 1
            f[3] = bj > 0 ? yface(x0, y - 1, k) : 0.f;        // -y face of sub-column 0
            f[4] = yface(x0, y, k);                            // +y face of sub-column 0
            f[5] = bj > 0 ? yface(x0 + 1, y - 1, k) : 0.f;    // -y face of sub-column 1
            f[6] = yface(x0 + 1, y, k);                        // +y face of sub-column 1
            // diagonals, same association as march_f32_kernel: -(((cxm+cxp)+(cym+cyp))+(czm+czp))
            f[7] = -(((f[0] + f[1]) + (f[3] + f[4])) + ((k > 0 ? cz[0][k > 0 ? k - 1 : 0] : 0.f) + cz[0][k]));
            f[8] = -(((f[1] + f[2]) + (f[5] + f[6])) + ((k > 0 ? cz[1][k > 0 ? k - 1 : 0] : 0.f) + cz[1][k]));
            uint32_t w[9];
#pragma unroll
            for (int q = 0; q < 9; q++) w[q] = __float_as_uint(f[q]);
            tm_st8(regA + (uint32_t)(8 * k), w);
            tm_st1(regB + (uint32_t)k, w[8]);
        }
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");

        #pragma unroll(2)   // two substeps per iteration: no register copies at the back edge
        for (int it = 0; it < a.n_sub; it++) {
            float* buf = xbuf + (it & 1) * BUF;
            if (active) {
#pragma unroll
                for (int k = 0; k < W1; k++)
#pragma unroll
                    for (int sc = 0; sc < 2; sc++) buf[k * LEVEL + sc * PLANE + t] = u[sc][k];
            }
            __syncthreads();
            uint32_t cb[2][9];
            tm_ld9(regA, regB, cb[0]);
            tm_wait_ld9(cb[0]);
            float prev[2] = {0.f, 0.f};
#pragma unroll
            for (int k = 0; k < W1; k++) {
                uint32_t (&cc)[9] = cb[k & 1];
                uint32_t (&cn)[9] = cb[(k + 1) & 1];
                if (k + 1 < W1) tm_ld9(regA + (uint32_t)(8 * (k + 1)), regB + (uint32_t)(k + 1), cn);
                const float* lv = buf + k * LEVEL;
                const float l = lv[1 * PLANE + tl], r = lv[0 * PLANE + tr];
                const float b0 = lv[0 * PLANE + tb], b1 = lv[1 * PLANE + tb];
                const float t0 = lv[0 * PLANE + tt], t1 = lv[1 * PLANE + tt];
                float c[9];
#pragma unroll
                for (int q = 0; q < 9; q++) c[q] = __uint_as_float(cc[q]);
                const float cxm[2] = {c[0], c[1]}, cxp[2] = {c[1], c[2]};
                const float cym[2] = {c[3], c[5]}, cyp[2] = {c[4], c[6]};
                const float amv[2] = {c[7], c[8]};
                const float uxm[2] = {l, u[0][k]}, uxp[2] = {u[1][k], r};
                const float uym[2] = {b0, b1}, uyp[2] = {t0, t1};
                float nu[2];
#pragma unroll
                for (int sc = 0; sc < 2; sc++) {
                    const float cur = u[sc][k];
                    float v = amv[sc] * cur;
                    v = fmaf(cxm[sc], uxm[sc], v);
                    v = fmaf(cxp[sc], uxp[sc], v);
                    v = fmaf(cym[sc], uym[sc], v);
                    v = fmaf(cyp[sc], uyp[sc], v);
                    v = fmaf(k > 0 ? cz[sc][k > 0 ? k - 1 : 0] : 0.f, prev[sc], v);
                    v = fmaf(cz[sc][k], k + 1 < W1 ? u[sc][k + 1 < W1 ? k + 1 : k] : 0.f, v);
                    nu[sc] = __fadd_rn(cur, v);
                }
#pragma unroll
                for (int sc = 0; sc < 2; sc++) { prev[sc] = u[sc][k]; u[sc][k] = nu[sc]; }
                if (k + 1 < W1) tm_wait_ld9(cn);
            }
        }

        // Epilogue: store, then per-column FP64 sums in k order (same order as march_f32_kernel).
        float* sbuf = xbuf + (a.n_sub & 1) * BUF;
        if (active) {
#pragma unroll
            for (int sc = 0; sc < 2; sc++) {
                const int x = 2 * bi + sc, y = bj;
#pragma unroll
                for (int k = 0; k < W1; k++) {
                    float stv = 0.f;
                    if (cell_ok(x, y, k)) stv = store_q(a, L, qplane(a, R, x, y, k), sx - R + x, sy - R + y, sz - R + k, pos, u[sc][k]);
                    sbuf[k * LEVEL + sc * PLANE + t] = stv;
                }
            }
        }
        __syncthreads();
        for (int c = t; c < SPB * COLS; c += blockDim.x) {
            const int sl = c / COLS, cc = c - sl * COLS;
            const int x = cc % W1, y = cc / W1;
            const int tt2 = sl * TPS + (x >> 1) + NBX * y;
            const int sc = x & 1;
            int64_t colsum = 0;
#pragma unroll
            for (int k = 0; k < W1; k++) colsum += mass_fix(sbuf[k * LEVEL + sc * PLANE + tt2]);
            red[c] = colsum;
        }
        __syncthreads();
        finish_sigma<COLS, SPB>(red, first, a.src_end, a.list, a.sigma);
        __syncthreads();
    }

    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" :: "r"(taddr) : "memory");
}

template <int R>
cudaError_t launch_tmx(const MarchArgs& a, int num_sms, cudaStream_t st) {
    using M = MapTmx<R>;
    const int64_t nsrc = a.src_end - a.src_begin;
    if (nsrc <= 0) return cudaSuccess;
    cudaError_t e = cudaFuncSetAttribute(march_tmx_kernel<R>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)M::SMEM);
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, march_tmx_kernel<R>, M::THREADS, M::SMEM);
    if (e != cudaSuccess) return e;
    if (per_sm != 1) return cudaErrorInvalidConfiguration;   // TMEM allocation assumes one CTA per SM
    const int64_t nbatch = (nsrc + M::SPB - 1) / M::SPB;
    const int64_t grid = nbatch < (int64_t)num_sms ? nbatch : (int64_t)num_sms;
    march_tmx_kernel<R><<<(unsigned)grid, M::THREADS, M::SMEM, st>>>(a);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------------------------------
// One thread per window column with the lateral face coefficients in TMEM (mapping id 5; any R <= 10).
//
// For R = 9, 10 a column of 2R+1 cells with 6 coefficients each no longer fits in registers next to
// enough threads.  Here u, the diagonal and the z faces stay in registers and the 4 lateral faces of the
// column (4(2R+1) words) live in the thread's TMEM lane, in groups of 4 cells (16 words, one
// tcgen05.ld.32x32b.x16 each) fetched one group ahead of the compute.  Up to 4 threads share a TMEM lane
// (128 columns each), so one CTA of up to 448 threads per SM owns all 512 columns.  The halo exchange
// and the FP32 operations (and their order) are those of march_f32_kernel.
template <int R>
struct MapTmc {
    static constexpr int W1 = 2 * R + 1;
    static constexpr int COLS = W1 * W1;
    static constexpr int THREADS = ((COLS + 31) / 32) * 32;
    static constexpr int NG = (W1 + 3) / 4;               // TMEM groups of 4 cells
    static constexpr int BUF = COLS * W1;
    static constexpr size_t SMEM_USED = (size_t)((2 * BUF * 4 + 15) / 16) * 16 + (size_t)COLS * 8;
    static constexpr size_t SMEM = SMEM_USED > 120 * 1024 ? SMEM_USED : 120 * 1024;
    static_assert(16 * NG <= 128, "lateral faces of a column must fit a 128-column TMEM slot");
    static_assert(THREADS <= 512, "at most 4 threads per TMEM lane");
    // Coarse mode adds the per-block sums (at most W1^3 blocks in a window, plus the total).
    static constexpr size_t SMEM_COARSE_USED = SMEM_USED + (size_t)(W1 * W1 * W1 + 1) * 8;
    static constexpr size_t SMEM_COARSE = SMEM_COARSE_USED > SMEM ? SMEM_COARSE_USED : SMEM;
};

// COARSE (coarse blocks with convection, or one per SM at most; otherwise they run in march_tm.cu): the source is coarse block a.list[pos]
// (Eqs. 10-15): its window is centred on the block's centre cell (radius R = window_R + (B - 1) / 2), the march starts
// from 1 on the block's liquid cells, and the epilogue maps the marched field onto the blocks of the window (column J of
// the coarse matrix, written destination-indexed) instead of storing a kernel.  The face coefficients differ by direction:
// a.ax/ay/az hold the coefficient of the lower cell in the upper cell's update and a.bx/by/bz that of the upper cell in
// the lower one's; the diagonal is minus the sum of the cell's outflow coefficients.  Otherwise both are a.ax/ay/az.
template <int R, bool COARSE>
__global__ void __launch_bounds__(MapTmc<R>::THREADS, 1) march_tmc_kernel(MarchArgs a) {
    using M = MapTmc<R>;
    constexpr int W1 = M::W1, COLS = M::COLS, NG = M::NG, BUF = M::BUF;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float* xbuf = reinterpret_cast<float*>(smem_raw);                                  // [2][COLS][W1]
    int64_t* red = reinterpret_cast<int64_t*>(smem_raw + ((2 * BUF * 4 + 15) / 16) * 16);  // [COLS]
    __shared__ uint32_t s_taddr;

    const int t = threadIdx.x, warp = t >> 5;
    if (warp == 0) {
        const uint32_t dst = (uint32_t)__cvta_generic_to_shared(&s_taddr);
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" :: "r"(dst) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t taddr = s_taddr;
    const uint32_t tbase = taddr + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)(128 * (warp >> 2));

    const bool active = t < COLS;
    const int col = active ? t : 0;
    const int ci = col % W1, cj = col / W1;
    const int64_t nbatch = a.src_end - a.src_begin;
    const int base = col * W1;
    const int xm = ci > 0 ? base - W1 : base;
    const int xp = ci < 2 * R ? base + W1 : base;
    const int ym = cj > 0 ? base - W1 * W1 : base;
    const int yp = cj < 2 * R ? base + W1 * W1 : base;

    for (int64_t b = blockIdx.x; b < nbatch; b += gridDim.x) {
        const int64_t first = a.src_begin + b;
        int64_t s = first;
        const bool src_ok = active && s < a.src_end;
        if (src_ok && a.list) s = a.list[s];
        const int64_t pos = first;                     // position of the source in the launch range
        const SrcLoc L = locate(a, src_ok, s);
        const int nx = L.nx, ny = L.ny, nz = L.nz;
        const int64_t nxy = (int64_t)nx * ny;
        const float* ax = a.ax + L.base;   // coefficients of the source's structure
        const float* ay = a.ay + L.base;
        const float* az = a.az + L.base;
        int sx = 0, sy = 0, sz = 0;
        int bx = 0, by = 0, bz = 0;
        const int bh = COARSE ? (a.coarse_B - 1) / 2 : 0;
        if (src_ok) {
            if constexpr (COARSE) {
                bx = (int)(s % a.ncx);
                by = (int)((s / a.ncx) % a.ncy);
                bz = (int)(s / ((int64_t)a.ncx * a.ncy));
                sx = bx * a.coarse_B + bh;       // centre of the block (may lie past a clipped domain edge)
                sy = by * a.coarse_B + bh;
                sz = bz * a.coarse_B + bh;
            } else {
                sx = (int)(s % nx);
                const int64_t r = s / nx;
                sy = (int)(r % ny);
                sz = (int)(r / ny);
            }
        }
        const int x = sx - R + ci, y = sy - R + cj;
        const bool col_ok = src_ok && x >= 0 && x < nx && y >= 0 && y < ny;

        float u[W1], am[W1], cz[W1];
        float czb[COARSE ? W1 : 1];              // COARSE: coefficient of the upper z neighbour (cz: of the lower)
        float zprev = 0.f, zprevb = 0.f;
        const float* bxp = COARSE ? a.bx + L.base : nullptr;
        const float* byp = COARSE ? a.by + L.base : nullptr;
        const float* bzp = COARSE ? a.bz + L.base : nullptr;
#pragma unroll
        for (int g = 0; g < NG; g++) {
            uint32_t w[16];
#pragma unroll
            for (int q = 0; q < 4; q++) {
                const int k = 4 * g + q;
                float vxm = 0.f, vxp = 0.f, vym = 0.f, vyp = 0.f, vz = 0.f;
                float oxm = 0.f, oxp = 0.f, oym = 0.f, oyp = 0.f, vzb = 0.f;   // COARSE: outflows, upper-z inflow
                if (k < W1) {
                    const int z = sz - R + k;
                    const bool ok = col_ok && z >= 0 && z < nz;
                    float u0 = (!COARSE && src_ok && ci == R && cj == R && k == R) ? 1.f : 0.f;
                    float vb = 0.f;                       // open faces of the cell (coarse, far field)
                    if (ok) {
                        const int64_t i = (int64_t)x + (int64_t)nx * y + nxy * z;
                        if (COARSE && a.liquid[i] && abs(ci - R) <= bh && abs(cj - R) <= bh && abs(k - R) <= bh) u0 = 1.f;
                        if (COARSE && a.abnd) vb = __ldg(a.abnd + i);
                        if (ci > 0 && x > 0) vxm = __ldg(ax + i - 1);
                        if (ci < 2 * R && x + 1 < nx) vxp = __ldg(COARSE ? bxp + i : ax + i);
                        if (cj > 0 && y > 0) vym = __ldg(ay + i - nx);
                        if (cj < 2 * R && y + 1 < ny) vyp = __ldg(COARSE ? byp + i : ay + i);
                        if (k < 2 * R && z + 1 < nz) vz = __ldg(az + i);
                        if constexpr (COARSE) {
                            if (ci > 0 && x > 0) oxm = __ldg(bxp + i - 1);
                            if (ci < 2 * R && x + 1 < nx) oxp = __ldg(ax + i);
                            if (cj > 0 && y > 0) oym = __ldg(byp + i - nx);
                            if (cj < 2 * R && y + 1 < ny) oyp = __ldg(ay + i);
                            if (k < 2 * R && z + 1 < nz) vzb = __ldg(bzp + i);
                        }
                    }
                    cz[k < W1 ? k : 0] = vz;
                    if constexpr (COARSE) {
                        // outflow through the -z face: the lower cell's upper-z inflow coefficient
                        czb[k < W1 ? k : 0] = vzb;
                        const float diag = ((oxm + oxp) + (oym + oyp)) + (zprevb + vz);
                        am[k < W1 ? k : 0] = -(diag + vb);
                        zprevb = vzb;
                    } else {
                        am[k < W1 ? k : 0] = -(((vxm + vxp) + (vym + vyp)) + (zprev + vz));
                    }
                    u[k < W1 ? k : 0] = u0;
                    zprev = vz;
                }
                w[4 * q + 0] = __float_as_uint(vxm);
                w[4 * q + 1] = __float_as_uint(vxp);
                w[4 * q + 2] = __float_as_uint(vym);
                w[4 * q + 3] = __float_as_uint(vyp);
            }
            tm_st16(tbase + (uint32_t)(16 * g), w);
        }
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");

        for (int it = 0; it < a.n_sub; it++) {
            float* buf = xbuf + (it & 1) * BUF;
            if (active) {
#pragma unroll
                for (int k = 0; k < W1; k++) buf[base + k] = u[k];
            }
            __syncthreads();
            uint32_t cb[2][16];                        // group g in cb[g & 1], g + 1 loading into the other
            tm_ld16(tbase, cb[0]);
            tm_wait_ld(cb[0]);
            float prev = 0.f;
#pragma unroll
            for (int g = 0; g < NG; g++) {
                uint32_t (&cc)[16] = cb[g & 1];
                uint32_t (&cn)[16] = cb[(g + 1) & 1];
                if (g + 1 < NG) tm_ld16(tbase + (uint32_t)(16 * (g + 1)), cn);
#pragma unroll
                for (int q = 0; q < 4; q++) {
                    const int k = 4 * g + q;
                    if (k < W1) {
                        const float cxm = __uint_as_float(cc[4 * q + 0]), cxp = __uint_as_float(cc[4 * q + 1]);
                        const float cym = __uint_as_float(cc[4 * q + 2]), cyp = __uint_as_float(cc[4 * q + 3]);
                        const float cur = u[k];
                        float v = am[k] * cur;
                        v = fmaf(cxm, buf[xm + k], v);
                        v = fmaf(cxp, buf[xp + k], v);
                        v = fmaf(cym, buf[ym + k], v);
                        v = fmaf(cyp, buf[yp + k], v);
                        v = fmaf(k > 0 ? cz[k > 0 ? k - 1 : 0] : 0.f, prev, v);
                        v = fmaf(COARSE ? czb[COARSE ? k : 0] : cz[k], k + 1 < W1 ? u[k + 1 < W1 ? k + 1 : k] : 0.f, v);
                        prev = cur;
                        u[k] = __fadd_rn(cur, v);
                    }
                }
                if (g + 1 < NG) tm_wait_ld(cn);
            }
        }

        float* sbuf = xbuf + (a.n_sub & 1) * BUF;
        if constexpr (COARSE) {
            if (active) {
#pragma unroll
                for (int k = 0; k < W1; k++) {
                    const int z = sz - R + k;
                    const bool ok = col_ok && z >= 0 && z < nz && a.liquid[(int64_t)x + (int64_t)nx * y + nxy * z];
                    sbuf[base + k] = ok ? u[k] : 0.f;
                }
            }
            __syncthreads();
            coarse_epilogue<R>(a, [&](int x, int y, int k, int) { return sbuf[(x + W1 * y) * W1 + k]; },
                               reinterpret_cast<double*>(red + COLS), first, 1);
        } else {
            if (active) {
#pragma unroll
                for (int k = 0; k < W1; k++) {
                    const int z = sz - R + k;
                    float stv = 0.f;
                    if (col_ok && z >= 0 && z < nz) stv = store_q(a, L, qplane(a, R, ci, cj, k), x, y, z, pos, u[k]);
                    sbuf[base + k] = stv;
                }
            }
            __syncthreads();
            for (int c = t; c < COLS; c += blockDim.x) {
                int64_t colsum = 0;
#pragma unroll
                for (int k = 0; k < W1; k++) colsum += mass_fix(sbuf[c * W1 + k]);
                red[c] = colsum;
            }
            __syncthreads();
            finish_sigma<COLS, 1>(red, first, a.src_end, a.list, a.sigma);
        }
        __syncthreads();
    }

    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" :: "r"(taddr) : "memory");
}

template <int R, bool COARSE = false>
cudaError_t launch_tmc(const MarchArgs& a, int num_sms, cudaStream_t st) {
    using M = MapTmc<R>;
    const int64_t nsrc = a.src_end - a.src_begin;
    if (nsrc <= 0) return cudaSuccess;
    cudaError_t e = cudaFuncSetAttribute(march_tmc_kernel<R, COARSE>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(COARSE ? M::SMEM_COARSE : M::SMEM));
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, march_tmc_kernel<R, COARSE>, M::THREADS, (COARSE ? M::SMEM_COARSE : M::SMEM));
    if (e != cudaSuccess) return e;
    if (per_sm != 1) return cudaErrorInvalidConfiguration;   // TMEM allocation assumes one CTA per SM
    const int64_t grid = nsrc < (int64_t)num_sms ? nsrc : (int64_t)num_sms;
    march_tmc_kernel<R, COARSE><<<(unsigned)grid, M::THREADS, (COARSE ? M::SMEM_COARSE : M::SMEM), st>>>(a);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------------------------------
// Mapping 6: one window column per thread for a PAIR of sources, every FP32 operation packed (f32x2).
//
// The two sources of a pair have the same window shape, so each thread marches the same column of
// both: the state, the diagonals and the z faces are register pairs (source A in the low half, B in
// the high half), the exchange buffer holds one 8-byte pair per cell, and the four lateral faces of
// both sources live in TMEM as aligned pairs (8 words per cell, 2 cells per 16-word load).  Each
// packed mul.rn / fma.rn / add.rn.f32x2 rounds each half exactly like the scalar instruction, and the
// operations come in the order of march_f32_kernel, so the kernels are bitwise those of mappings 1-5.
// Per cell-substep of a pair: 1 store + 4 loads of 8 bytes and 8 packed FP32 instructions.
template <int R>
struct MapTmp {
    static constexpr int W1 = 2 * R + 1;
    static constexpr int COLS = W1 * W1;
    static constexpr int PAIRS = (384 / COLS) > 0 ? (384 / COLS) : 1;   // source pairs per CTA
    static constexpr int THREADS = ((PAIRS * COLS + 31) / 32) * 32;
    static constexpr int SLOTS = (THREADS / 32 + 3) / 4;                // threads per TMEM lane
    static constexpr int SLOT_COLS = (512 / SLOTS) / 16 * 16;           // TMEM columns per thread
    static constexpr int NG = (W1 + 1) / 2;                             // 16-word groups of 2 cells
    static constexpr int BUF = PAIRS * COLS * W1;                       // 8-byte pairs per buffer
    static constexpr size_t SMEM_USED = (size_t)2 * BUF * 8 + (size_t)2 * PAIRS * COLS * 8;
    static constexpr size_t SMEM = SMEM_USED > 120 * 1024 ? SMEM_USED : 120 * 1024;
    static_assert(16 * NG <= SLOT_COLS, "the lateral faces of a column pair must fit the thread's TMEM slot");
    static_assert(R <= 8, "mapping 6 covers R <= 8");
};

template <int R>
__global__ void __launch_bounds__(MapTmp<R>::THREADS, 1) march_tmp_kernel(MarchArgs a) {
    using M = MapTmp<R>;
    constexpr int W1 = M::W1, COLS = M::COLS, NG = M::NG, BUF = M::BUF, PAIRS = M::PAIRS;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    uint64_t* xbuf = reinterpret_cast<uint64_t*>(smem_raw);                        // [2][PAIRS*COLS][W1]
    int64_t* red = reinterpret_cast<int64_t*>(smem_raw + (size_t)2 * BUF * 8);      // [2*PAIRS][COLS]
    __shared__ uint32_t s_taddr;

    const int t = threadIdx.x, warp = t >> 5;
    if (warp == 0) {
        const uint32_t dst = (uint32_t)__cvta_generic_to_shared(&s_taddr);
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" :: "r"(dst) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t taddr = s_taddr;
    const uint32_t tbase = taddr + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)(M::SLOT_COLS * (warp >> 2));

    const bool active = t < PAIRS * COLS;
    const int pair = active ? t / COLS : 0;
    const int col = active ? t - pair * COLS : 0;
    const int ci = col % W1, cj = col / W1;
    const int64_t nbatch = (a.src_end - a.src_begin + 2 * PAIRS - 1) / (2 * PAIRS);
    const int base = (pair * COLS + col) * W1;
    const int xm = ci > 0 ? base - W1 : base;
    const int xp = ci < 2 * R ? base + W1 : base;
    const int ym = cj > 0 ? base - W1 * W1 : base;
    const int yp = cj < 2 * R ? base + W1 * W1 : base;

    for (int64_t b = blockIdx.x; b < nbatch; b += gridDim.x) {
        const int64_t first = a.src_begin + b * 2 * PAIRS;
        // Per source of the pair (h = 0: low half, h = 1: high half): geometry and validity.
        int64_t pos[2], sidx[2];
        bool src_ok[2], col_ok[2];
        int sx[2], sy[2], sz[2], xs[2], ys[2], nzs[2], nxs[2], nys[2];
        int64_t nxy[2], cbase[2];
        SrcLoc Ls[2];
#pragma unroll
        for (int h = 0; h < 2; h++) {
            pos[h] = first + 2 * pair + h;
            src_ok[h] = active && pos[h] < a.src_end;
            int64_t s = pos[h];
            if (src_ok[h] && a.list) s = a.list[s];
            const SrcLoc L = locate(a, src_ok[h], s);
            nxs[h] = L.nx; nys[h] = L.ny; nzs[h] = L.nz;
            nxy[h] = (int64_t)L.nx * L.ny;
            cbase[h] = L.base;
            Ls[h] = L;
            sidx[h] = s;
            sx[h] = sy[h] = sz[h] = 0;
            if (src_ok[h]) {
                sx[h] = (int)(s % L.nx);
                const int64_t r = s / L.nx;
                sy[h] = (int)(r % L.ny);
                sz[h] = (int)(r / L.ny);
            }
            xs[h] = sx[h] - R + ci;
            ys[h] = sy[h] - R + cj;
            col_ok[h] = src_ok[h] && xs[h] >= 0 && xs[h] < L.nx && ys[h] >= 0 && ys[h] < L.ny;
        }

        uint64_t u[W1], am[W1], cz[W1];
        float zprev[2] = {0.f, 0.f};
#pragma unroll
        for (int g = 0; g < NG; g++) {
            uint32_t w[16];
#pragma unroll
            for (int q = 0; q < 2; q++) {
                const int k = 2 * g + q;
                float f[2][5] = {{0.f, 0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f, 0.f}};   // xm xp ym yp z+
                if (k < W1) {
                    float amv[2], uv[2];
#pragma unroll
                    for (int h = 0; h < 2; h++) {
                        const int z = sz[h] - R + k;
                        const bool ok = col_ok[h] && z >= 0 && z < nzs[h];
                        if (ok) {
                            const int64_t i = cbase[h] + (int64_t)xs[h] + (int64_t)nxs[h] * ys[h] + nxy[h] * z;
                            if (ci > 0 && xs[h] > 0) f[h][0] = __ldg(a.ax + i - 1);
                            if (ci < 2 * R && xs[h] + 1 < nxs[h]) f[h][1] = __ldg(a.ax + i);
                            if (cj > 0 && ys[h] > 0) f[h][2] = __ldg(a.ay + i - nxs[h]);
                            if (cj < 2 * R && ys[h] + 1 < nys[h]) f[h][3] = __ldg(a.ay + i);
                            if (k < 2 * R && z + 1 < nzs[h]) f[h][4] = __ldg(a.az + i);
                        }
                        amv[h] = -(((f[h][0] + f[h][1]) + (f[h][2] + f[h][3])) + (zprev[h] + f[h][4]));
                        uv[h] = (src_ok[h] && ci == R && cj == R && k == R) ? 1.f : 0.f;
                        zprev[h] = f[h][4];
                    }
                    const int kk = k < W1 ? k : 0;
                    cz[kk] = f2pack(f[0][4], f[1][4]);
                    am[kk] = f2pack(amv[0], amv[1]);
                    u[kk] = f2pack(uv[0], uv[1]);
                }
#pragma unroll
                for (int d = 0; d < 4; d++) {
                    w[8 * q + 2 * d] = __float_as_uint(f[0][d]);
                    w[8 * q + 2 * d + 1] = __float_as_uint(f[1][d]);
                }
            }
            tm_st16(tbase + (uint32_t)(16 * g), w);
        }
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");

        for (int it = 0; it < a.n_sub; it++) {
            uint64_t* buf = xbuf + (it & 1) * BUF;
            if (active) {
#pragma unroll
                for (int k = 0; k < W1; k++) buf[base + k] = u[k];
            }
            __syncthreads();
            uint32_t cb[2][16];
            tm_ld16(tbase, cb[0]);
            tm_wait_ld(cb[0]);
            uint64_t prev = 0ull;
#pragma unroll
            for (int g = 0; g < NG; g++) {
                uint32_t (&cc)[16] = cb[g & 1];
                uint32_t (&cn)[16] = cb[(g + 1) & 1];
                if (g + 1 < NG) tm_ld16(tbase + (uint32_t)(16 * (g + 1)), cn);
#pragma unroll
                for (int q = 0; q < 2; q++) {
                    const int k = 2 * g + q;
                    if (k < W1) {
                        const uint64_t cur = u[k];
                        uint64_t v = mul2(am[k], cur);
                        v = fma2(u2pack(cc[8 * q + 0], cc[8 * q + 1]), buf[xm + k], v);
                        v = fma2(u2pack(cc[8 * q + 2], cc[8 * q + 3]), buf[xp + k], v);
                        v = fma2(u2pack(cc[8 * q + 4], cc[8 * q + 5]), buf[ym + k], v);
                        v = fma2(u2pack(cc[8 * q + 6], cc[8 * q + 7]), buf[yp + k], v);
                        v = fma2(k > 0 ? cz[k > 0 ? k - 1 : 0] : 0ull, prev, v);
                        v = fma2(cz[k], k + 1 < W1 ? u[k + 1 < W1 ? k + 1 : k] : 0ull, v);
                        prev = cur;
                        u[k] = add2(cur, v);
                    }
                }
                if (g + 1 < NG) tm_wait_ld(cn);
            }
        }

        uint64_t* sbuf = xbuf + (a.n_sub & 1) * BUF;
        if (active) {
#pragma unroll
            for (int k = 0; k < W1; k++) {
                float stv[2];
#pragma unroll
                for (int h = 0; h < 2; h++) {
                    const int z = sz[h] - R + k;
                    stv[h] = 0.f;
                    if (col_ok[h] && z >= 0 && z < nzs[h]) {
                        stv[h] = store_q(a, Ls[h], qplane(a, R, ci, cj, k), xs[h], ys[h], z, pos[h], h == 0 ? f2lo(u[k]) : f2hi(u[k]));
                    }
                }
                sbuf[base + k] = f2pack(stv[0], stv[1]);
            }
        }
        __syncthreads();
        for (int c = t; c < PAIRS * COLS; c += blockDim.x) {
            const int pr = c / COLS, cl = c - pr * COLS;
            int64_t s0 = 0, s1 = 0;
#pragma unroll
            for (int k = 0; k < W1; k++) {
                const uint64_t v = sbuf[c * W1 + k];
                s0 += mass_fix(f2lo(v));
                s1 += mass_fix(f2hi(v));
            }
            red[(2 * pr) * COLS + cl] = s0;
            red[(2 * pr + 1) * COLS + cl] = s1;
        }
        __syncthreads();
        finish_sigma<COLS, 2 * PAIRS>(red, first, a.src_end, a.list, a.sigma);
        __syncthreads();
    }

    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" :: "r"(taddr) : "memory");
}

template <int R>
cudaError_t launch_tmp(const MarchArgs& a, int num_sms, cudaStream_t st) {
    using M = MapTmp<R>;
    const int64_t nsrc = a.src_end - a.src_begin;
    if (nsrc <= 0) return cudaSuccess;
    cudaError_t e = cudaFuncSetAttribute(march_tmp_kernel<R>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)M::SMEM);
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, march_tmp_kernel<R>, M::THREADS, M::SMEM);
    if (e != cudaSuccess) return e;
    if (per_sm != 1) return cudaErrorInvalidConfiguration;   // TMEM allocation assumes one CTA per SM
    const int64_t nbatch = (nsrc + 2 * M::PAIRS - 1) / (2 * M::PAIRS);
    const int64_t grid = nbatch < (int64_t)num_sms ? nbatch : (int64_t)num_sms;
    march_tmp_kernel<R><<<(unsigned)grid, M::THREADS, M::SMEM, st>>>(a);
    return cudaGetLastError();
}

template <int R, int P>
cudaError_t launch_f32(const MarchArgs& a, int num_sms, cudaStream_t st) {
    using M = Map32<R, P>;
    const int64_t nsrc = a.src_end - a.src_begin;
    if (nsrc <= 0) return cudaSuccess;
    cudaError_t e = cudaFuncSetAttribute(march_f32_kernel<R, P>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)M::SMEM);
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, march_f32_kernel<R, P>, M::THREADS, M::SMEM);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    const int64_t nbatch = (nsrc + M::SPB - 1) / M::SPB;
    const int64_t grid = nbatch < (int64_t)num_sms * per_sm ? nbatch : (int64_t)num_sms * per_sm;
    march_f32_kernel<R, P><<<(unsigned)grid, M::THREADS, M::SMEM, st>>>(a);
    return cudaGetLastError();
}

template <int R>
cudaError_t launch_f32_p(const MarchArgs& a, int P, int num_sms, cudaStream_t st) {
    switch (P) {
        case 1: return launch_f32<R, 1>(a, num_sms, st);
        case 2: return launch_f32<R, 2>(a, num_sms, st);
        case 3: return launch_f32<R, 3>(a, num_sms, st);
        case 4: return launch_march_blocks(a, num_sms, st);
        case 5: return a.bx ? launch_march_flow(a, num_sms, st) : launch_tmc<R>(a, num_sms, st);
        case 6: return launch_tmp<R>(a, num_sms, st);
        case 7: return launch_tmx<R>(a, num_sms, st);
        default: return cudaErrorInvalidValue;
    }
}

template <int R>
cudaError_t launch_f64(const MarchArgs& a, int num_sms, cudaStream_t st) {
    using S = Shape<R>;
    const int64_t nsrc = a.src_end - a.src_begin;
    if (nsrc <= 0) return cudaSuccess;
    const size_t smem = (size_t)(5 * S::SPB64 * S::W + S::SPB64 * S::COLS) * 8;
    cudaError_t e = cudaFuncSetAttribute(march_f64_kernel<R>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, march_f64_kernel<R>, S::THREADS64, smem);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    const int64_t nbatch = (nsrc + S::SPB64 - 1) / S::SPB64;
    const int64_t grid = nbatch < (int64_t)num_sms * per_sm ? nbatch : (int64_t)num_sms * per_sm;
    march_f64_kernel<R><<<(unsigned)grid, S::THREADS64, smem, st>>>(a);
    return cudaGetLastError();
}

cudaError_t dispatch(const MarchArgs& a, int P, int num_sms, cudaStream_t st) {
    if (a.store == Store::F64) {
        switch (a.R) {
            case 1: return launch_f64<1>(a, num_sms, st);
            case 2: return launch_f64<2>(a, num_sms, st);
            case 3: return launch_f64<3>(a, num_sms, st);
            case 4: return launch_f64<4>(a, num_sms, st);
            case 5: return launch_f64<5>(a, num_sms, st);
            case 6: return launch_f64<6>(a, num_sms, st);
            case 7: return launch_f64<7>(a, num_sms, st);
            case 8: return launch_f64<8>(a, num_sms, st);
            default: return cudaErrorInvalidValue;
        }
    }
    switch (a.R) {
        case 1: return launch_f32_p<1>(a, P, num_sms, st);
        case 2: return launch_f32_p<2>(a, P, num_sms, st);
        case 3: return launch_f32_p<3>(a, P, num_sms, st);
        case 4: return launch_f32_p<4>(a, P, num_sms, st);
        case 5: return launch_f32_p<5>(a, P, num_sms, st);
        case 6: return launch_f32_p<6>(a, P, num_sms, st);
        case 7: return launch_f32_p<7>(a, P, num_sms, st);
        case 8: return launch_f32_p<8>(a, P, num_sms, st);
        case 9: return P == 5 ? (a.bx ? launch_march_flow(a, num_sms, st) : launch_tmc<9>(a, num_sms, st))
                       : P == 4 ? launch_march_blocks(a, num_sms, st) : P == 7 ? launch_tmx<9>(a, num_sms, st)
                       : cudaErrorInvalidValue;
        case 10: return P == 5 ? (a.bx ? launch_march_flow(a, num_sms, st) : launch_tmc<10>(a, num_sms, st))
                        : P == 4 ? launch_march_blocks(a, num_sms, st) : P == 7 ? launch_tmx<10>(a, num_sms, st)
                        : cudaErrorInvalidValue;
        default: return cudaErrorInvalidValue;
    }
}

// Thread mapping of an FP32 march when the caller does not force one.  Mapping 4 is the fastest at every radius (ms for 48^3
// sources, BF16 kernels, 100 substeps, mappings 1-7; R = 9, 10 have 4, 5 and 7 only):
//   R = 2: 1.52 3.77 2.16 1.00 9.27 1.23 1.34    R = 6: 61.5 30.8 31.9 12.4 27.5 18.7 25.5
//   R = 3: 3.98 9.32 8.76 2.36 11.1 3.26 3.46    R = 8: 48.6 66.5 60.3 26.5 48.1 47.9 67.0
//   R = 4: 17.4 19.1 21.2 4.42 15.3 6.92 7.47    R = 9: 48.6 (4) 54.6 (5) 74.7 (7)
//   R = 5: 39.1 43.1 16.8 7.55 17.8 11.5 15.0    R = 10: 54.2 (4) 82.7 (5) 81.8 (7)
// R = 1 (us, 60 substeps, mappings 1 2 3 4 6 7): 512 sources 28 21 18 17 33 23, 32768 92 99 107 82 84 101, 64^3 679 727 807
// 508 546 682.
// With one source per SM at most (two at R = 5-7) one thread a column has the shorter substep up to R = 8 (us, 60 substeps,
// mappings 4 / 5: 152 sources R = 1 17 13, R = 3 25 16, R = 5 51 21, R = 8 72 45, R = 10 52 72; 216 sources R = 4 30 33, R = 5
// 51 37, R = 7 64 58, R = 8 72 87).
int default_mapping(const MarchArgs& a, int num_sms) {
    const int64_t few = (int64_t)num_sms * (a.R >= 5 && a.R <= 7 ? 2 : 1);
    return a.R <= 8 && a.src_end - a.src_begin <= few ? 5 : 4;
}

}  // namespace

int march_mapping(const MarchArgs& a, int parts_req, int num_sms) {
    if (a.store == Store::F64) return 1;
    if (a.bx) return 5;                           // direction-dependent coefficients: march_flow.cu
    if (parts_req >= 1 && parts_req <= 7 && (a.R <= 8 || parts_req == 4 || parts_req == 5 || parts_req == 7))
        return parts_req;
    return default_mapping(a, num_sms);
}

cudaError_t launch_march_coarse(const MarchArgs& a, int R, int num_sms, cudaStream_t st) {
    MarchArgs b = a;
    if (!a.bx) {
        if (a.src_end - a.src_begin > num_sms) return launch_march_blocks(a, num_sms, st);
        // One block per SM at most: what counts is the latency of a substep, and a thread a column has the shorter one
        // (15 x 14 x 13, B = 3, R = 2, 60 substeps: 31 us in 2x2 blocks, 21 so).  Both directions' faces are the same.
        b.bx = a.ax; b.by = a.ay; b.bz = a.az;
    }
    switch (R) {                                  // one column per thread; direction-dependent coefficients
        case 1: return launch_tmc<1, true>(b, num_sms, st);
        case 2: return launch_tmc<2, true>(b, num_sms, st);
        case 3: return launch_tmc<3, true>(b, num_sms, st);
        case 4: return launch_tmc<4, true>(b, num_sms, st);
        case 5: return launch_tmc<5, true>(b, num_sms, st);
        case 6: return launch_tmc<6, true>(b, num_sms, st);
        case 7: return launch_tmc<7, true>(b, num_sms, st);
        case 8: return launch_tmc<8, true>(b, num_sms, st);
        case 9: return launch_tmc<9, true>(b, num_sms, st);
        case 10: return launch_tmc<10, true>(b, num_sms, st);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_march(const MarchArgs& a, int num_sms, int parts_req, cudaStream_t st, int* parts_used) {
    const int P = march_mapping(a, parts_req, num_sms);
    if (parts_used) *parts_used = P;
    return dispatch(a, P, num_sms, st);
}

}  // namespace fdirw
