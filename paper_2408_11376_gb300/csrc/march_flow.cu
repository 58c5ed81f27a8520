// The FP32 march with direction-dependent faces (convection): across each face the lower cell's coefficient in the upper
// cell's update (A: a.ax/ay/az) differs from the upper cell's in the lower one's (B: a.bx/by/bz), and the diagonal is
// minus the sum of the cell's outflow coefficients (A of its +faces, B of its -faces).
//
// Each thread owns two x-adjacent window columns: the 2x2 blocks of the diffusion march need 20 coefficients a level here
// (no face is shared between two cells any more), which its share of registers and TMEM does not hold.  The halo exchange
// is 4 words per cell (one store, the outer x and both y neighbours) instead of the 5 of one column per thread, and two to
// three times as many sources share an SM.  As in march_tm.cu the levels go in pairs (j, j + R + 1), the middle level R as
// a scalar one: a pair's update is eight packed f32x2 instructions per column, in the order of operations of the
// one-column march (bitwise equal to it, and to the diffusion march without flow).
//
// A pair's coefficients are 20 words in TMEM, loaded in two halves while the other one computes:
//   X = {xm0, xp0, xm1, xp1 (8 words), am0, am1 (4)},  Y = {ym0, ym1, yp0, yp1 (8)}
// with xm/xp, ym/yp the inflow coefficients from the lower and the upper neighbour of column 0 or 1; u and the z
// coefficients of both directions stay in registers.
//
// 48^3 sources, BF16 kernels, ms a substep / ms outside the substeps, one column per thread and one source per SM before:
// R = 8 0.437 / 8.1 -> 0.294 / 4.1; R = 3 0.091 / 2.4 -> 0.021 / 0.34; R = 10 0.740 / 13.2 -> 0.521 / 10.3.  At R = 9 the
// 190 threads of one source leave lanes of an SM idle (0.472 / 9.9 -> 0.439 / 8.8).
#include "fdirw_internal.h"
#include "march_common.cuh"

namespace fdirw {

namespace {

template <int R>
struct MapFlow {
    static constexpr int W1 = 2 * R + 1;
    static constexpr int NBX = R + 1;                     // column pairs per window row (the last one half padding)
    static constexpr int TPS = NBX * W1;                  // threads per source
    // As many warps as the registers of a thread's state allow; SLOT TMEM columns a thread.
    static constexpr int THREADS = R == 10 ? 256 : R == 9 ? 192 : R == 8 ? 320 : 384;
    static constexpr int SLOT = THREADS <= 256 ? 256 : 168;
    static constexpr int SPB = THREADS / TPS;             // sources per CTA
    static constexpr int BUF = W1 * 2 * THREADS;          // floats per exchange buffer
    static constexpr int CA = 16 * R, CM = (20 * R + 7) / 8 * 8;      // TMEM columns of the diagonals, the middle level
    static_assert(SPB >= 1 && CM + 8 <= SLOT, "a source must fit a CTA and its coefficients their TMEM columns");
    static constexpr size_t SMEM_USED = (size_t)2 * BUF * 4 + (size_t)THREADS * 8 + (size_t)SPB * sizeof(SlotInfo);
    static constexpr size_t SMEM = SMEM_USED > 120 * 1024 ? SMEM_USED : 120 * 1024;
};

// Exchange buffer: float pairs [pair][column][thread], then the middle level's floats.
template <int R>
__device__ __forceinline__ int fpair_at(int p, int sc, int t) { return (p * 2 + sc) * MapFlow<R>::THREADS + t; }
template <int R>
__device__ __forceinline__ int fmid_at(int sc, int t) { return 4 * MapFlow<R>::THREADS * R + sc * MapFlow<R>::THREADS + t; }

__device__ __forceinline__ void tm_ld8(uint32_t a, uint32_t (&r)[8]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(a));
}
// Wait for the loads in flight; the registers are in-out operands so that no use of them comes before it.
__device__ __forceinline__ void tm_wait8(uint32_t (&r)[8]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]));
}
__device__ __forceinline__ void tm_wait84(uint32_t (&r)[8], uint32_t (&q)[4]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                   "+r"(q[0]), "+r"(q[1]), "+r"(q[2]), "+r"(q[3]));
}
template <int N>
__device__ __forceinline__ uint64_t pr(const uint32_t (&r)[N], int q) { return u2pack(r[2 * q], r[2 * q + 1]); }

template <int R>
__global__ void __launch_bounds__(MapFlow<R>::THREADS, 1) march_flow_kernel(MarchArgs a) {
    using M = MapFlow<R>;
    constexpr int W1 = M::W1, NBX = M::NBX, TPS = M::TPS, SPB = M::SPB, PT = M::THREADS, H = R + 1;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float* xbuf = reinterpret_cast<float*>(smem_raw);                                   // [2][BUF]
    int64_t* red = reinterpret_cast<int64_t*>(smem_raw + (size_t)2 * M::BUF * 4);       // [THREADS]
    SlotInfo* sinfo = reinterpret_cast<SlotInfo*>(red + PT);                            // [SPB]
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
    const uint32_t tbase = taddr + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)(M::SLOT * (warp >> 2));

    const bool active = t < SPB * TPS;
    const int slot = active ? t / TPS : 0;
    const int b = active ? t - slot * TPS : 0;
    const int bi = b % NBX, cj = b / NBX, x0 = 2 * bi;
    // Neighbours in a ring (past a window edge another row's or source's finite value, which meets a zero face): every
    // warp reads consecutive slots, free of bank conflicts.
    auto ring = [](int v) { return v < 0 ? v + PT : v >= PT ? v - PT : v; };
    const int tl = ring(t - 1), tr = ring(t + 1), tb = ring(t - NBX), tt = ring(t + NBX);
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
        int sx = 0, sy = 0, sz = 0;
        if (src_ok) split_cell(s, nx, ny, sx, sy, sz);
        if (active && b == 0) sinfo[slot] = SlotInfo{L, pos, sx, sy, sz, src_ok ? 1 : 0};

        // Faces as in march_tm.cu: stored with their lower cell, 0 outside the window or the domain; all but the z range
        // is fixed per thread.
        const int gx = sx - R + x0, gy = sy - R + cj, gz = sz - R;
        auto in = [](int v, int n) { return (unsigned)v < (unsigned)n; };
        const bool yin = src_ok && in(gy, ny);
        const bool xf[3] = {bi > 0 && yin && in(gx - 1, nx - 1), x0 + 1 < W1 && yin && in(gx, nx - 1),
                            x0 + 2 < W1 && yin && in(gx + 1, nx - 1)};
        const bool xc[2] = {src_ok && in(gx, nx), src_ok && x0 + 1 < W1 && in(gx + 1, nx)};
        const bool yf[2] = {cj > 0 && in(gy - 1, ny - 1), cj + 1 < W1 && in(gy, ny - 1)};
        const int64_t i0 = L.base + (int64_t)gx + (int64_t)nx * gy + nxy * gz;

        uint64_t U[2][R], za[2][R], zb[2][R], za0[2];   // u; A and B of the pairs' +z faces; A under pair 0
        float um[2], zbm[2], amm[2];                    // middle level: u, B of its +z face, diagonal
        float fa[2][W1 + 1], fb[2][W1 + 1];             // A and B of each level's -z face (prologue only)
#pragma unroll
        for (int sc = 0; sc < 2; sc++) {
            fa[sc][0] = fb[sc][0] = 0.f;
#pragma unroll
            for (int k = 0; k < W1; k++) {
                const bool ok = k + 1 < W1 && xc[sc] && yin && in(gz + k, nz - 1);
                const int64_t i = i0 + sc + nxy * k;
                fa[sc][k + 1] = ok ? __ldg(a.az + i) : 0.f;
                fb[sc][k + 1] = ok ? __ldg(a.bz + i) : 0.f;
            }
            const bool centre = src_ok && x0 + sc == R && cj == R;
#pragma unroll
            for (int j = 0; j < R; j++) {
                U[sc][j] = 0;                           // the source is on the middle level
                za[sc][j] = f2pack(fa[sc][j + 1], fa[sc][j + H + 1]);
                zb[sc][j] = f2pack(fb[sc][j + 1], fb[sc][j + H + 1]);
            }
            za0[sc] = f2pack(0.f, fa[sc][H]);
            zbm[sc] = fb[sc][H];
            um[sc] = centre ? 1.f : 0.f;
        }
        // f: xm0 xp0 xm1 xp1 am0 am1 ym0 ym1 yp0 yp1 of level k
        auto level = [&](int k, float (&f)[10]) {
            const bool zin = in(gz + k, nz);
            const int64_t i = i0 + nxy * k;
            float ax[3], bx[3];
#pragma unroll
            for (int q = 0; q < 3; q++) {
                ax[q] = zin && xf[q] ? __ldg(a.ax + i + q - 1) : 0.f;
                bx[q] = zin && xf[q] ? __ldg(a.bx + i + q - 1) : 0.f;
            }
            f[0] = ax[0]; f[1] = bx[1]; f[2] = ax[1]; f[3] = bx[2];
#pragma unroll
            for (int sc = 0; sc < 2; sc++) {
                const bool low = zin && xc[sc] && yf[0], up = zin && xc[sc] && yf[1];
                f[6 + sc] = low ? __ldg(a.ay + i + sc - nx) : 0.f;
                const float oym = low ? __ldg(a.by + i + sc - nx) : 0.f;
                f[8 + sc] = up ? __ldg(a.by + i + sc) : 0.f;
                const float oyp = up ? __ldg(a.ay + i + sc) : 0.f;
                // outflows, association of the one-column march: -(((xm+xp)+(ym+yp))+(zm+zp))
                f[4 + sc] = -(((bx[sc] + ax[sc + 1]) + (oym + oyp)) + (fb[sc][k] + fa[sc][k + 1]));
            }
        };
#pragma unroll
        for (int j = 0; j < R; j++) {
            float f[2][10];
            level(j, f[0]);
            level(j + H, f[1]);
            uint32_t w[20];
#pragma unroll
            for (int e = 0; e < 20; e++) w[e] = __float_as_uint(f[e & 1][e / 2]);
            tm_st8(tbase + (uint32_t)(16 * j), w);
            tm_st8(tbase + (uint32_t)(16 * j + 8), w + 12);
            tm_st4(tbase + (uint32_t)(M::CA + 4 * j), w + 8);
        }
        {
            float f[10];
            level(R, f);
            uint32_t w[8];
#pragma unroll
            for (int e = 0; e < 8; e++) w[e] = __float_as_uint(f[e < 4 ? e : e + 2]);
            tm_st8(tbase + (uint32_t)M::CM, w);
            amm[0] = f[4];
            amm[1] = f[5];
        }
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");

        {
            uint64_t* w = reinterpret_cast<uint64_t*>(xbuf);
#pragma unroll
            for (int j = 0; j < R; j++)
#pragma unroll
                for (int sc = 0; sc < 2; sc++) w[fpair_at<R>(j, sc, t)] = U[sc][j];
#pragma unroll
            for (int sc = 0; sc < 2; sc++) xbuf[fmid_at<R>(sc, t)] = um[sc];
        }
        uint32_t X[8], D[4], Y[8];
        auto load_x = [&](int j) {
            tm_ld8(tbase + (uint32_t)(16 * j), X);
            tm_ld4(tbase + (uint32_t)(M::CA + 4 * j), D);
        };
        load_x(0);
        __syncthreads();

#pragma unroll 2
        for (int it = 0; it < a.n_sub; it++) {
            const float* buf = xbuf + (it & 1) * M::BUF;
            const uint64_t* rd = reinterpret_cast<const uint64_t*>(buf);
            float* nbuf = xbuf + ((it & 1) ^ 1) * M::BUF;
            uint64_t* wr = reinterpret_cast<uint64_t*>(nbuf);
            uint64_t l = rd[fpair_at<R>(0, 1, tl)], r = rd[fpair_at<R>(0, 0, tr)];
            // z neighbours of pair 0 from below (hi: the middle level) and of the last pair from above (lo: the same)
            uint64_t prev[2];
            float over[2];
#pragma unroll
            for (int sc = 0; sc < 2; sc++) {
                prev[sc] = f2pack(0.f, um[sc]);
                over[sc] = f2hi(U[sc][0]);
            }
            tm_wait84(X, D);
#pragma unroll
            for (int j = 0; j < R; j++) {
                tm_ld8(tbase + (uint32_t)(16 * j + 8), Y);
                const uint64_t b0 = rd[fpair_at<R>(j, 0, tb)], b1 = rd[fpair_at<R>(j, 1, tb)];
                const uint64_t t0 = rd[fpair_at<R>(j, 0, tt)], t1 = rd[fpair_at<R>(j, 1, tt)];
                const uint64_t u0 = U[0][j], u1 = U[1][j];
                uint64_t V[2];
                V[0] = mul2(pr(D, 0), u0);
                V[1] = mul2(pr(D, 1), u1);
                V[0] = fma2(pr(X, 0), l, V[0]);
                V[1] = fma2(pr(X, 2), u0, V[1]);
                V[0] = fma2(pr(X, 1), u1, V[0]);
                V[1] = fma2(pr(X, 3), r, V[1]);
                tm_wait8(Y);
                if (j + 1 < R) {
                    load_x(j + 1);
                    l = rd[fpair_at<R>(j + 1, 1, tl)];
                    r = rd[fpair_at<R>(j + 1, 0, tr)];
                } else {
                    tm_ld8(tbase + (uint32_t)M::CM, X);
                }
                V[0] = fma2(pr(Y, 0), b0, V[0]);
                V[1] = fma2(pr(Y, 1), b1, V[1]);
                V[0] = fma2(pr(Y, 2), t0, V[0]);
                V[1] = fma2(pr(Y, 3), t1, V[1]);
#pragma unroll
                for (int sc = 0; sc < 2; sc++) V[sc] = fma2(j > 0 ? za[sc][j > 0 ? j - 1 : 0] : za0[sc], prev[sc], V[sc]);
#pragma unroll
                for (int sc = 0; sc < 2; sc++)
                    V[sc] = fma2(zb[sc][j], j + 1 < R ? U[sc][j + 1 < R ? j + 1 : j] : f2pack(um[sc], 0.f), V[sc]);
#pragma unroll
                for (int sc = 0; sc < 2; sc++) {
                    prev[sc] = U[sc][j];
                    U[sc][j] = add2(U[sc][j], V[sc]);
                    wr[fpair_at<R>(j, sc, t)] = U[sc][j];
                }
                tm_wait84(X, D);
            }
            {                                           // the middle level: the same coefficients as scalars
                const float ml = buf[fmid_at<R>(1, tl)], mr = buf[fmid_at<R>(0, tr)];
                const float mb[2] = {buf[fmid_at<R>(0, tb)], buf[fmid_at<R>(1, tb)]};
                const float mt[2] = {buf[fmid_at<R>(0, tt)], buf[fmid_at<R>(1, tt)]};
                const float ul[2] = {ml, um[0]}, ur[2] = {um[1], mr};
                float nu[2];
#pragma unroll
                for (int sc = 0; sc < 2; sc++) {
                    float v = amm[sc] * um[sc];
                    v = fmaf(__uint_as_float(X[2 * sc]), ul[sc], v);
                    v = fmaf(__uint_as_float(X[2 * sc + 1]), ur[sc], v);
                    v = fmaf(__uint_as_float(X[4 + sc]), mb[sc], v);
                    v = fmaf(__uint_as_float(X[6 + sc]), mt[sc], v);
                    v = fmaf(f2lo(za[sc][R - 1]), f2lo(prev[sc]), v);
                    v = fmaf(zbm[sc], over[sc], v);
                    nu[sc] = __fadd_rn(um[sc], v);
                }
#pragma unroll
                for (int sc = 0; sc < 2; sc++) { um[sc] = nu[sc]; nbuf[fmid_at<R>(sc, t)] = nu[sc]; }
                load_x(0);
            }
            __syncthreads();
        }
        tm_wait84(X, D);

        // Epilogue as in march_tm.cu.
        {
            MassSum m;
#pragma unroll
            for (int sc = 0; sc < 2; sc++) {
#pragma unroll
                for (int j = 0; j < R; j++) {
                    m.add(put(nullptr, a.store, 0, f2lo(U[sc][j])));
                    m.add(put(nullptr, a.store, 0, f2hi(U[sc][j])));
                }
                m.add(put(nullptr, a.store, 0, um[sc]));
            }
            red[t] = m.total();
        }
        const float* ubuf = xbuf + (a.n_sub & 1) * M::BUF;
        store_columns<R, SPB, PT>(a, sinfo, [&](int x, int y, int k, int sl) {
            const int th = sl * TPS + (x >> 1) + NBX * y, sc = x & 1;
            return ubuf[k == R ? fmid_at<R>(sc, th) : 2 * fpair_at<R>(k > R ? k - H : k, sc, th) + (k > R ? 1 : 0)];
        });
        __syncthreads();                                // red is complete; sinfo and xbuf are free for the next batch
        finish_sigma<TPS, SPB>(red, first, a.src_end, a.list, a.sigma);
    }

    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" :: "r"(taddr) : "memory");
}

template <int R>
cudaError_t launch_flow(const MarchArgs& a, int num_sms, cudaStream_t st) {
    using M = MapFlow<R>;
    const int64_t nsrc = a.src_end - a.src_begin;
    if (nsrc <= 0) return cudaSuccess;
    cudaError_t e = cudaFuncSetAttribute(march_flow_kernel<R>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)M::SMEM);
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, march_flow_kernel<R>, M::THREADS, M::SMEM);
    if (e != cudaSuccess) return e;
    if (per_sm != 1) return cudaErrorInvalidConfiguration;   // TMEM allocation assumes one CTA per SM
    const int64_t nbatch = (nsrc + M::SPB - 1) / M::SPB;
    const int64_t grid = nbatch < (int64_t)num_sms ? nbatch : (int64_t)num_sms;
    march_flow_kernel<R><<<(unsigned)grid, M::THREADS, M::SMEM, st>>>(a);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_march_flow(const MarchArgs& a, int num_sms, cudaStream_t st) {
    switch (a.R) {
        case 1: return launch_flow<1>(a, num_sms, st);
        case 2: return launch_flow<2>(a, num_sms, st);
        case 3: return launch_flow<3>(a, num_sms, st);
        case 4: return launch_flow<4>(a, num_sms, st);
        case 5: return launch_flow<5>(a, num_sms, st);
        case 6: return launch_flow<6>(a, num_sms, st);
        case 7: return launch_flow<7>(a, num_sms, st);
        case 8: return launch_flow<8>(a, num_sms, st);
        case 9: return launch_flow<9>(a, num_sms, st);
        case 10: return launch_flow<10>(a, num_sms, st);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace fdirw
