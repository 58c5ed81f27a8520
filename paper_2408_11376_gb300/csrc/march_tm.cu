// 2x2-block mapping of the FP32 march with TMEM-resident coefficients (mapping id 4).
//
// Each thread owns a 2x2 block of window columns (u in registers), so the halo it exchanges through shared
// memory per substep is 3 words per cell (one store, two loads) instead of the 5 of one column per thread.
// The 12 x/y face coefficients of a block level and its 4 diagonals do not fit in registers beside u and the
// z faces; they live in Tensor Memory, one TMEM lane per thread, and are streamed back with tcgen05.ld while
// the previous half of a level pair computes.
//
// The levels of a thread are taken in pairs (j, j + H), H = half of them rounded up: u, the faces and the diagonals
// of a pair are natural 64-bit register pairs, a neighbour's pair is one 8-byte shared load, and so are the pair's z
// neighbours (the pairs j - 1 and j + 1), so that a pair's whole update is eight packed f32x2 instructions.  (With
// adjacent levels in a pair the z terms had to be scalar: 14% more issue slots.)  Only where the two halves meet are
// pairs put together from single registers; an odd count leaves the middle level H - 1 as a scalar one.  Each packed
// instruction rounds each half like the scalar one and the operations of a cell come in the order of
// march_f32_kernel, so the results are bitwise those of every other mapping.
//
// A pair's coefficients come in two halves, each loaded while the other one computes (32 registers in all; each
// half works on the four cells side by side, so four independent chains are in flight):
//   X = {L0, I0, R0, L1, I1, R1, am0, am1, am2, am3},  Y = {B0, B1, J0, J1, T0, T1}   (pairs of levels)
// with L/I/R the x faces left of, inside and right of the block in row 0 or 1, B/J/T the y faces below, inside
// and above it in column 0 or 1, am the diagonals of the four cells (sub-column sc = column + 2 row).
//
// R <= 8: each thread has all 2R+1 levels; SPB sources per CTA.  R = 9, 10: a thread's state would not
// fit its registers, so each column block is split in z between two threads of different warps (the first
// takes LO levels); the two meet at one face through the exchange buffer.
//
// What bounds it: the shared-memory exchange.  8.2 cell-substeps a clock and SM at every radius (padding cells of
// the blocks included) are 25 of the 32 words a clock; the FP32 pipe is half busy.  64^3 sources, BF16 kernels, ms a
// substep / ms outside the substeps (coefficients, sums, cache stores), scalar levels before: R = 8: 0.721 / 28.0
// -> 0.554 / 8.1; R = 6: 0.333 / 13.0 -> 0.261 / 3.5; R = 3: 0.056 / 2.2 -> 0.048 / 0.8; R = 10 against one column
// per thread (mapping 5): 1.73 / 23.5 -> 1.10 / 15.3 (grouped stores; 23.4 without).
//
// One CTA per SM (two or three threads per TMEM lane; the CTA allocates all 512 columns once and frees them before it
// exits, and its shared-memory request keeps a second CTA off the SM so an allocation never waits).
#include "fdirw_internal.h"
#include "march_common.cuh"

#include <type_traits>

namespace fdirw {

namespace {

template <int R>
struct MapTm {
    static constexpr int W1 = 2 * R + 1;
    static constexpr int NB = R + 1;                      // blocks per window axis (last one half padding)
    static constexpr int TPS = NB * NB;                   // threads per source and z part
    static constexpr int ZS = R <= 8 ? 1 : 2;             // z parts
    // R <= 4: the state leaves room for 12 warps (3 threads per TMEM lane) instead of 8; 64^3 sources, ms a substep /
    // outside: R = 3 0.0477 / 0.80 -> 0.0461 / 0.68, R = 4 0.0930 / 1.18 -> 0.0927 / 1.02.
    static constexpr int THREADS = R <= 4 ? 384 : 256;
    static constexpr int SLOT = R <= 4 ? 160 : 256;       // TMEM columns of a thread
    static constexpr int PT = THREADS / ZS;               // threads of a z part
    static constexpr int SPB = PT / TPS;                  // sources per CTA
    static constexpr int LO = ZS == 1 ? W1 : 10;          // levels of the first z part
    static constexpr int BUF = W1 * 4 * PT;               // floats per exchange buffer
    static constexpr size_t SMEM_USED = (size_t)2 * BUF * 4 + (size_t)THREADS * 8 + (size_t)SPB * sizeof(SlotInfo);
    static constexpr size_t SMEM = SMEM_USED > 120 * 1024 ? SMEM_USED : 120 * 1024;
    // Stored values of a group of sources (see march_part): 4 of 16 bits or 2 of 32 each.
    static constexpr size_t SMEM_GROUP_USED = 8 * (size_t)W1 * W1 * W1 + SMEM_USED + 3 * sizeof(SlotInfo);
    static constexpr size_t SMEM_GROUP = SMEM_GROUP_USED > SMEM ? SMEM_GROUP_USED : SMEM;
    // Coarse mode adds the per-block sums (at most W1^3 blocks in a window, plus the total).
    static constexpr size_t SMEM_COARSE_USED = SMEM_USED + (size_t)(W1 * W1 * W1 + 1) * 8;
    static constexpr size_t SMEM_COARSE = SMEM_COARSE_USED > SMEM ? SMEM_COARSE_USED : SMEM;
    static_assert(SPB >= 1, "a source must fit one CTA");
};

// TMEM columns of a z part of NK levels (at most 256 per thread).  The pairs p < AP take 32 columns each: X at 32 p (16
// words, am2 and am3 at 32 p + 24) and Y at 32 p + 16 (8 words, the last 4 at 32 p + 28).  The others keep their
// diagonals in registers and take 24: X as 8 + 4 words, Y as 8 + 4.  The middle level of an odd count takes 16.
template <int NK>
struct ColsTm {
    static constexpr int NP = NK / 2, MID = NK & 1;
    static constexpr int AP0 = (256 - 16 * MID - 24 * NP) / 8;
    static constexpr int AP = AP0 < NP ? AP0 : NP;
    static constexpr int NR = NP - AP;                    // pairs whose diagonals stay in registers
    static constexpr int C8 = 32 * AP, C4 = C8 + 16 * NR, CT = C4 + 8 * NR;
    static_assert(AP >= 0 && CT % 16 == 0 && CT + 16 * MID <= 256, "a thread's coefficients fit its TMEM columns");
};

// Exchange buffer: float pairs [pair][sub-column][thread of the part] of both parts, then the middle level's floats.
template <int R>
__device__ __forceinline__ int pair_at(int p, int sc, int th) { return (p * 4 + sc) * MapTm<R>::PT + th; }
template <int R>
__device__ __forceinline__ int mid_at(int sc, int th) { return 8 * MapTm<R>::PT * R + sc * MapTm<R>::PT + th; }
// Float index of window level k.
template <int R>
__device__ __forceinline__ int level_at(int k, int sc, int th) {
    using M = MapTm<R>;
    const int part = k >= M::LO ? 1 : 0, nk = part ? M::W1 - M::LO : M::LO, j = k - part * M::LO;
    const int h = (nk + 1) / 2, p = (part ? M::LO / 2 : 0) + (j >= h ? j - h : j);
    return (nk & 1) && j == h - 1 ? mid_at<R>(sc, th) : 2 * pair_at<R>(p, sc, th) + (j >= h ? 1 : 0);
}

template <int NK>
__device__ __forceinline__ void load_x(uint32_t tbase, int p, uint32_t (&r)[16], uint32_t (&r4)[4]) {
    using C = ColsTm<NK>;
    if (p < C::AP) {
        tm_ld16(tbase + (uint32_t)(32 * p), r);
        tm_ld4(tbase + (uint32_t)(32 * p + 24), r4);
    } else {
        tm_ld12(tbase + (uint32_t)(C::C8 + 16 * (p - C::AP)), tbase + (uint32_t)(C::C4 + 8 * (p - C::AP)), r);
    }
}
template <int NK>
__device__ __forceinline__ void load_y(uint32_t tbase, int p, uint32_t (&r)[12]) {
    using C = ColsTm<NK>;
    if (p < C::AP) tm_ld12(tbase + (uint32_t)(32 * p + 16), tbase + (uint32_t)(32 * p + 28), r);
    else tm_ld12(tbase + (uint32_t)(C::C8 + 16 * (p - C::AP) + 8), tbase + (uint32_t)(C::C4 + 8 * (p - C::AP) + 4), r);
}

// Wait for the loads in flight; the registers are in-out operands so that no use of them comes before it.
__device__ __forceinline__ void tm_wait_x(uint32_t (&r)[16], uint32_t (&q)[4]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                   "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15]),
                   "+r"(q[0]), "+r"(q[1]), "+r"(q[2]), "+r"(q[3]));
}
__device__ __forceinline__ void tm_wait_y(uint32_t (&r)[12]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                   "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]));
}

template <int N>
__device__ __forceinline__ uint64_t pr(const uint32_t (&r)[N], int q) { return u2pack(r[2 * q], r[2 * q + 1]); }

// One z part (levels K0 .. K0 + NK - 1 of the window) of every source of the CTA's batches.
// SPREAD: a batch is a.spb sources, at most the SPB that fit (else SPB).
// COARSE: the source is coarse block a.list[pos] (Eqs. 10-15): its window is centred on the block's centre cell
// (radius R = window_R + (B - 1) / 2), the march starts from 1 on the block's liquid cells, an open face (a.abnd) adds
// to the diagonal, and the epilogue maps the marched field onto the blocks of the window instead of storing a kernel.
// G > 1 (one source at a time per CTA, R = 9, 10): the CTA marches G consecutive sources, keeps their rounded values in
// shared memory and stores them together.  A plane gets G adjacent values then instead of one, and the stores, half of the
// time outside the substeps, are as many sectors fewer (64^3 sources, R = 10, BF16, no substeps: 21.4 -> 15.3 ms; 100 substeps: 129 -> 122).
template <int R, bool COARSE, int G, bool SPREAD, int K0, int NK>
__device__ __forceinline__ void march_part(const MarchArgs& a, unsigned char* smem_raw, uint32_t tbase) {
    using M = MapTm<R>;
    using C = ColsTm<NK>;
    constexpr int W1 = M::W1, NB = M::NB, TPS = M::TPS, PT = M::PT, SPB = M::SPB;
    constexpr int NP = C::NP, AP = C::AP, NR = C::NR, P0 = K0 / 2, H = NP + C::MID;
    constexpr bool MID = C::MID, BELOW = K0 > 0, ABOVE = K0 + NK < W1;
    static_assert(K0 % 2 == 0 && (ABOVE ? !MID : MID), "one part has an odd count of levels");
    float* xbuf = reinterpret_cast<float*>(smem_raw);                                   // [2][BUF]
    int64_t* red = reinterpret_cast<int64_t*>(smem_raw + (size_t)2 * M::BUF * 4);       // [THREADS]
    SlotInfo* sinfo = reinterpret_cast<SlotInfo*>(red + M::THREADS);                    // [SPB * G]
    static_assert(G == 1 || (SPB == 1 && !COARSE), "groups are of single sources");
    using Word = typename std::conditional<G == 4, uint16_t, float>::type;              // a stored value of a group
    Word* stage = reinterpret_cast<Word*>(sinfo + SPB * G);                             // [W1^3][G]
    auto bar = [] { asm volatile("bar.sync 0;" ::: "memory"); };   // met by both z parts, each in its own code

    const int t = threadIdx.x;
    const int th = M::ZS == 1 ? t : t & (PT - 1);
    const int spb = SPREAD ? a.spb : SPB;          // sources that the CTA takes at a time
    const bool active = th < spb * TPS;
    // A warp without a source only meets the others at their barriers.  The zeros that its ring neighbours read stay.
    const bool idle = SPREAD && (th & ~31) >= spb * TPS;
    if (idle)
        for (float* buf = xbuf; buf < xbuf + 2 * M::BUF; buf += M::BUF)
            for (int sc = 0; sc < 4; sc++) {
                for (int p = 0; p < R; p++) reinterpret_cast<uint64_t*>(buf)[pair_at<R>(p, sc, th)] = 0;
                buf[mid_at<R>(sc, th)] = 0.f;
            }
    const int slot = active ? th / TPS : 0;
    const int b = active ? th - slot * TPS : 0;
    const int bi = b % NB, bj = b / NB;
    // Neighbour blocks, in a ring: past a window edge this is a thread of another row or source, whose (finite)
    // value meets a zero face.  Every warp then reads 32 consecutive slots, which no bank serves twice; reading
    // the own slot there instead cost 10% of the shared-memory wavefronts in bank conflicts.
    auto ring = [](int v) { return v < 0 ? v + PT : v >= PT ? v - PT : v; };
    const int tl = ring(th - 1), tr = ring(th + 1), tb = ring(th - NB), tt = ring(th + NB);
    const int x0 = 2 * bi, y0 = 2 * bj;
    const int64_t nbatch = (a.src_end - a.src_begin + spb * G - 1) / (spb * G);

    for (int64_t bt = blockIdx.x; bt < nbatch; bt += gridDim.x) {
    if (G > 1 && K0 == 0 && t < G) sinfo[t].ok = 0;           // set by the sources that exist
    for (int g = 0; g < G; g++) {
        const int64_t first = a.src_begin + bt * (spb * G) + g;
        if (G > 1 && first >= a.src_end) break;               // (uniform over the CTA)
        auto end = [&]() -> int64_t {                         // of the sources that this batch may reach
            if constexpr (SPREAD) return first + spb < a.src_end ? first + spb : a.src_end;
            return a.src_end;
        };
        if (SPREAD && t >= spb && t < SPB) sinfo[t].ok = 0;
      if (idle) {
        for (int it = 0; it <= a.n_sub; it++) bar();
      } else {
        int64_t s = first + slot;
        const bool src_ok = active && s < end();
        if (src_ok && a.list) s = a.list[s];       // explicit source list (e.g. the surrogate's rejects)
        const int64_t pos = first + slot;          // position of the source in the launch range
        const SrcLoc L = locate(a, src_ok, s);
        const int nx = L.nx, ny = L.ny, nz = L.nz;
        const int64_t nxy = (int64_t)nx * ny;
        int sx = 0, sy = 0, sz = 0;
        const int bh = COARSE ? (a.coarse_B - 1) / 2 : 0;
        if (src_ok) {
            if constexpr (COARSE) {
                split_cell(s, a.ncx, a.ncy, sx, sy, sz);
                sx = sx * a.coarse_B + bh;         // centre of the block (may lie past a clipped domain edge)
                sy = sy * a.coarse_B + bh;
                sz = sz * a.coarse_B + bh;
            } else {
                split_cell(s, nx, ny, sx, sy, sz);
            }
        }
        if (active && b == 0 && K0 == 0)
            sinfo[G > 1 ? g : slot] = SlotInfo{L, pos, sx, sy, sz, src_ok ? 1 : 0};

        // A face is stored with its lower cell and taken when that cell is in the domain and both cells are in
        // the window and the domain (0 otherwise).  All but the z range is fixed per thread, so the 16 faces
        // of a block level are 16 loads at fixed offsets from 7 row pointers that advance by one plane.
        const int gx = sx - R + x0, gy = sy - R + y0, gz = sz - R + K0;
        auto in = [](int v, int n) { return (unsigned)v < (unsigned)n; };
        const bool xf[3] = {bi > 0 && in(gx - 1, nx - 1), x0 + 1 < W1 && in(gx, nx - 1), x0 + 2 < W1 && in(gx + 1, nx - 1)};
        const bool yf[3] = {bj > 0 && in(gy - 1, ny - 1), y0 + 1 < W1 && in(gy, ny - 1), y0 + 2 < W1 && in(gy + 1, ny - 1)};
        const bool xc[2] = {src_ok && in(gx, nx), src_ok && x0 + 1 < W1 && in(gx + 1, nx)};
        const bool yc[2] = {src_ok && in(gy, ny), src_ok && y0 + 1 < W1 && in(gy + 1, ny)};
        const int64_t i0 = L.base + (int64_t)gx + (int64_t)nx * gy + nxy * gz;
        const float* px = a.ax + i0;
        const float* py = a.ay + i0;
        const float* pz = a.az + i0;

        uint64_t U[4][NP], cz[4][NP], cz0[4];      // +z faces of the pairs; -z faces of pair 0
        float um[4] = {0.f, 0.f, 0.f, 0.f};        // middle level
        uint64_t amr[NR > 0 ? NR : 1][4];          // diagonals of the pairs p >= AP
        float zf[4][NK + 1];                       // -z face of each level, +z face of the last (prologue only)
#pragma unroll
        for (int sc = 0; sc < 4; sc++) {
            const float* p = pz + (sc & 1) + (int64_t)nx * (sc >> 1);
            const bool ok = xc[sc & 1] && yc[sc >> 1];
            zf[sc][0] = (BELOW && ok && in(gz - 1, nz - 1)) ? __ldg(p - nxy) : 0.f;
#pragma unroll
            for (int j = 0; j < NK; j++) {
                zf[sc][j + 1] = K0 + j + 1 < W1 && ok && in(gz + j, nz - 1) ? __ldg(p) : 0.f;
                p += nxy;
            }
            const bool centre = src_ok && x0 + (sc & 1) == R && y0 + (sc >> 1) == R;
            const bool near = COARSE && ok && abs(x0 + (sc & 1) - R) <= bh && abs(y0 + (sc >> 1) - R) <= bh;
            auto u0 = [&](int j) -> float {
                if (!COARSE) return centre && K0 + j == R ? 1.f : 0.f;
                if (!near || abs(K0 + j - R) > bh || !in(gz + j, nz)) return 0.f;
                return a.liquid[i0 + (sc & 1) + (int64_t)nx * (sc >> 1) + nxy * j] ? 1.f : 0.f;
            };
#pragma unroll
            for (int j = 0; j < NP; j++) {
                U[sc][j] = f2pack(u0(j), u0(j + H));
                cz[sc][j] = f2pack(zf[sc][j + 1], zf[sc][j + H + 1]);
            }
            cz0[sc] = f2pack(zf[sc][0], zf[sc][H]);
            if (MID) um[sc] = u0(NP);
        }
        // The 12 lateral faces and 4 diagonals of local level j.
        auto level = [&](int j, float (&f)[16]) {
            const bool zin = in(gz + j, nz);
            const float* qx0 = px + nxy * j;
            const float* qx1 = qx0 + nx;
            const float* qy1 = py + nxy * j;
            const float* qy0 = qy1 - nx;
            const float* qy2 = qy1 + nx;
            const bool z0 = zin && yc[0], z1 = zin && yc[1], w0 = zin && xc[0], w1 = zin && xc[1];
            f[0] = z0 && xf[0] ? __ldg(qx0 - 1) : 0.f;     // L0
            f[1] = z0 && xf[1] ? __ldg(qx0) : 0.f;         // I0
            f[2] = z0 && xf[2] ? __ldg(qx0 + 1) : 0.f;     // R0
            f[3] = z1 && xf[0] ? __ldg(qx1 - 1) : 0.f;     // L1
            f[4] = z1 && xf[1] ? __ldg(qx1) : 0.f;         // I1
            f[5] = z1 && xf[2] ? __ldg(qx1 + 1) : 0.f;     // R1
            f[10] = w0 && yf[0] ? __ldg(qy0) : 0.f;        // B0
            f[11] = w1 && yf[0] ? __ldg(qy0 + 1) : 0.f;    // B1
            f[12] = w0 && yf[1] ? __ldg(qy1) : 0.f;        // J0
            f[13] = w1 && yf[1] ? __ldg(qy1 + 1) : 0.f;    // J1
            f[14] = w0 && yf[2] ? __ldg(qy2) : 0.f;        // T0
            f[15] = w1 && yf[2] ? __ldg(qy2 + 1) : 0.f;    // T1
            // same association as march_f32_kernel: -(((cxm+cxp)+(cym+cyp))+(czm+czp))
#pragma unroll
            for (int sc = 0; sc < 4; sc++) {
                const int x = (sc & 1) + 3 * (sc >> 1), y = 10 + sc;
                float sum = ((f[x] + f[x + 1]) + (f[y] + f[y + 2])) + (zf[sc][j] + zf[sc][j + 1]);
                if constexpr (COARSE) {
                    const bool open = a.abnd && zin && xc[sc & 1] && yc[sc >> 1];
                    sum = sum + (open ? __ldg(a.abnd + i0 + (sc & 1) + (int64_t)nx * (sc >> 1) + nxy * j) : 0.f);
                }
                f[6 + sc] = -sum;
            }
        };
#pragma unroll
        for (int m = 0; m < NP; m++) {
            float f[2][16];
            level(m, f[0]);
            level(m + H, f[1]);
            uint32_t w[32];
#pragma unroll
            for (int e = 0; e < 32; e++) w[e] = __float_as_uint(f[e & 1][e / 2]);
            if (m < AP) {
                tm_st16(tbase + (uint32_t)(32 * m), w);
                tm_st8(tbase + (uint32_t)(32 * m + 16), w + 20);
                tm_st4(tbase + (uint32_t)(32 * m + 24), w + 16);
                tm_st4(tbase + (uint32_t)(32 * m + 28), w + 28);
            } else {
                tm_st8(tbase + (uint32_t)(C::C8 + 16 * (m - AP)), w);
                tm_st4(tbase + (uint32_t)(C::C4 + 8 * (m - AP)), w + 8);
                tm_st8(tbase + (uint32_t)(C::C8 + 16 * (m - AP) + 8), w + 20);
                tm_st4(tbase + (uint32_t)(C::C4 + 8 * (m - AP) + 4), w + 28);
#pragma unroll
                for (int sc = 0; sc < 4; sc++) amr[m >= AP ? m - AP : 0][sc] = u2pack(w[12 + 2 * sc], w[13 + 2 * sc]);
            }
        }
        if (MID) {
            float f[16];
            level(NP, f);
            uint32_t w[16];
#pragma unroll
            for (int e = 0; e < 16; e++) w[e] = __float_as_uint(f[e]);
            tm_st16(tbase + (uint32_t)C::CT, w);
        }
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");

        auto publish = [&](float* buf) {           // u of every level into an exchange buffer
            uint64_t* w = reinterpret_cast<uint64_t*>(buf);
#pragma unroll
            for (int m = 0; m < NP; m++)
#pragma unroll
                for (int sc = 0; sc < 4; sc++) w[pair_at<R>(P0 + m, sc, th)] = U[sc][m];
            if (MID)
#pragma unroll
                for (int sc = 0; sc < 4; sc++) buf[mid_at<R>(sc, th)] = um[sc];
        };
        uint32_t X[16], X4[4], Y[12];
        publish(xbuf);
        load_x<NK>(tbase, 0, X, X4);
        bar();

#pragma unroll 2
        for (int it = 0; it < a.n_sub; it++) {
            const float* buf = xbuf + (it & 1) * M::BUF;
            const uint64_t* rd = reinterpret_cast<const uint64_t*>(buf);
            float* nbuf = xbuf + ((it & 1) ^ 1) * M::BUF;
            uint64_t* wr = reinterpret_cast<uint64_t*>(nbuf);
            uint64_t l0 = rd[pair_at<R>(P0, 1, tl)], r0 = rd[pair_at<R>(P0, 0, tr)];
            uint64_t l1 = rd[pair_at<R>(P0, 3, tl)], r1 = rd[pair_at<R>(P0, 2, tr)];
            // z neighbours of pair 0 from below (hi: the level under the upper half) and of the last pair from above
            // (lo: the level over the lower half); the other part's u through the buffer
            uint64_t prev[4];
            float over[4], next[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int sc = 0; sc < 4; sc++) {
                float below = 0.f;
                if (BELOW) below = buf[level_at<R>(K0 > 0 ? K0 - 1 : 0, sc, th)];
                if (ABOVE) next[sc] = buf[level_at<R>(ABOVE ? K0 + NK : 0, sc, th)];
                prev[sc] = f2pack(below, MID ? um[sc] : f2lo(U[sc][NP - 1]));
                over[sc] = f2hi(U[sc][0]);
            }
            tm_wait_x(X, X4);
#pragma unroll
            for (int m = 0; m < NP; m++) {
                // diagonal and x terms while the y faces load
                load_y<NK>(tbase, m, Y);
                const uint64_t b0 = rd[pair_at<R>(P0 + m, 2, tb)], b1 = rd[pair_at<R>(P0 + m, 3, tb)];
                const uint64_t t0 = rd[pair_at<R>(P0 + m, 0, tt)], t1 = rd[pair_at<R>(P0 + m, 1, tt)];
                const uint64_t u0 = U[0][m], u1 = U[1][m], u2 = U[2][m], u3 = U[3][m];
                const int mr = m >= AP ? m - AP : 0;
                uint64_t V[4];
                V[0] = mul2(m < AP ? pr(X, 6) : amr[mr][0], u0);
                V[1] = mul2(m < AP ? pr(X, 7) : amr[mr][1], u1);
                V[2] = mul2(m < AP ? pr(X4, 0) : amr[mr][2], u2);
                V[3] = mul2(m < AP ? pr(X4, 1) : amr[mr][3], u3);
                V[0] = fma2(pr(X, 0), l0, V[0]);
                V[1] = fma2(pr(X, 1), u0, V[1]);
                V[2] = fma2(pr(X, 3), l1, V[2]);
                V[3] = fma2(pr(X, 4), u2, V[3]);
                V[0] = fma2(pr(X, 1), u1, V[0]);
                V[1] = fma2(pr(X, 2), r0, V[1]);
                V[2] = fma2(pr(X, 4), u3, V[2]);
                V[3] = fma2(pr(X, 5), r1, V[3]);
                tm_wait_y(Y);
                // y and z terms while the next pair's x faces load (the middle level's 16 words after the last)
                if (m + 1 < NP) {
                    load_x<NK>(tbase, m + 1, X, X4);
                    l0 = rd[pair_at<R>(P0 + m + 1, 1, tl)];
                    r0 = rd[pair_at<R>(P0 + m + 1, 0, tr)];
                    l1 = rd[pair_at<R>(P0 + m + 1, 3, tl)];
                    r1 = rd[pair_at<R>(P0 + m + 1, 2, tr)];
                } else if (MID) {
                    tm_ld16(tbase + (uint32_t)C::CT, X);
                } else {
                    load_x<NK>(tbase, 0, X, X4);
                }
                V[0] = fma2(pr(Y, 0), b0, V[0]);
                V[1] = fma2(pr(Y, 1), b1, V[1]);
                V[2] = fma2(pr(Y, 2), u0, V[2]);
                V[3] = fma2(pr(Y, 3), u1, V[3]);
                V[0] = fma2(pr(Y, 2), u2, V[0]);
                V[1] = fma2(pr(Y, 3), u3, V[1]);
                V[2] = fma2(pr(Y, 4), t0, V[2]);
                V[3] = fma2(pr(Y, 5), t1, V[3]);
#pragma unroll
                for (int sc = 0; sc < 4; sc++) V[sc] = fma2(m > 0 ? cz[sc][m > 0 ? m - 1 : 0] : cz0[sc], prev[sc], V[sc]);
#pragma unroll
                for (int sc = 0; sc < 4; sc++) {
                    const uint64_t up = m + 1 < NP ? U[sc][m + 1 < NP ? m + 1 : m] : f2pack(MID ? um[sc] : over[sc], next[sc]);
                    V[sc] = fma2(cz[sc][m], up, V[sc]);
                }
#pragma unroll
                for (int sc = 0; sc < 4; sc++) {
                    prev[sc] = U[sc][m];
                    U[sc][m] = add2(U[sc][m], V[sc]);
                }
#pragma unroll
                for (int sc = 0; sc < 4; sc++) wr[pair_at<R>(P0 + m, sc, th)] = U[sc][m];
                tm_wait_x(X, X4);
            }
            if (MID) {                             // the middle level: the same words as scalars
                const float tl0 = buf[mid_at<R>(1, tl)], tl1 = buf[mid_at<R>(3, tl)];
                const float tr0 = buf[mid_at<R>(0, tr)], tr1 = buf[mid_at<R>(2, tr)];
                const float tb0 = buf[mid_at<R>(2, tb)], tb1 = buf[mid_at<R>(3, tb)];
                const float tt0 = buf[mid_at<R>(0, tt)], tt1 = buf[mid_at<R>(1, tt)];
                float c[16];
#pragma unroll
                for (int q = 0; q < 16; q++) c[q] = __uint_as_float(X[q]);
                const float cxm[4] = {c[0], c[1], c[3], c[4]}, cxp[4] = {c[1], c[2], c[4], c[5]};
                const float uxm[4] = {tl0, um[0], tl1, um[2]}, uxp[4] = {um[1], tr0, um[3], tr1};
                const float uym[4] = {tb0, tb1, um[0], um[1]}, uyp[4] = {um[2], um[3], tt0, tt1};
                float nu[4];
#pragma unroll
                for (int sc = 0; sc < 4; sc++) {
                    float v = c[6 + sc] * um[sc];
                    v = fmaf(cxm[sc], uxm[sc], v);
                    v = fmaf(cxp[sc], uxp[sc], v);
                    v = fmaf(c[10 + sc], uym[sc], v);
                    v = fmaf(c[12 + sc], uyp[sc], v);
                    v = fmaf(f2lo(cz[sc][NP - 1]), f2lo(prev[sc]), v);
                    v = fmaf(f2hi(cz0[sc]), over[sc], v);
                    nu[sc] = __fadd_rn(um[sc], v);
                }
#pragma unroll
                for (int sc = 0; sc < 4; sc++) { um[sc] = nu[sc]; nbuf[mid_at<R>(sc, th)] = nu[sc]; }
                load_x<NK>(tbase, 0, X, X4);
            }
            bar();
        }
        tm_wait_x(X, X4);

        if constexpr (!COARSE) {
            // Each thread sums its own rounded values (cells outside the window or the domain are 0).
            MassSum m;
#pragma unroll
            for (int sc = 0; sc < 4; sc++) {
#pragma unroll
                for (int q = 0; q < NP; q++) {
                    m.add(put(nullptr, a.store, 0, f2lo(U[sc][q])));
                    m.add(put(nullptr, a.store, 0, f2hi(U[sc][q])));
                }
                if (MID) m.add(put(nullptr, a.store, 0, um[sc]));
            }
            red[(K0 > 0 ? PT : 0) + th] = m.total();
        }
        if constexpr (G > 1) {
            if (active) {
#pragma unroll
                for (int sc = 0; sc < 4; sc++) {
                    const int x = x0 + (sc & 1), y = y0 + (sc >> 1);
                    if (x >= W1 || y >= W1) continue;
                    Word* w = stage + G * (x + W1 * (y + W1 * K0)) + g;
                    auto keep = [&](int j, float v) {
                        if constexpr (G == 4)
                            w[G * W1 * W1 * j] = a.store == Store::F16 ? __half_as_ushort(__float2half_rn(v))
                                                                       : __bfloat16_as_ushort(__float2bfloat16_rn(v));
                        else
                            w[G * W1 * W1 * j] = v;
                    };
#pragma unroll
                    for (int q = 0; q < NP; q++) {
                        keep(q, f2lo(U[sc][q]));
                        keep(q + H, f2hi(U[sc][q]));
                    }
                    if (MID) keep(NP, um[sc]);
                }
            }
        }
      }
        // Epilogue.  xbuf's buffer n_sub & 1 holds every u (published by the last substep).
        const float* ubuf = xbuf + (a.n_sub & 1) * M::BUF;
        if constexpr (COARSE) {
            // u is 0 on cells that are not liquid: their faces carry nothing and they start at 0
            coarse_epilogue<R>(a, [&](int x, int y, int k, int q) {
                return ubuf[level_at<R>(k, (x & 1) + 2 * (y & 1), q * TPS + (x >> 1) + NB * (y >> 1))];
            }, reinterpret_cast<double*>(sinfo + SPB), first, end() - first < spb ? (int)(end() - first) : spb);
            continue;
        }
        if constexpr (G == 1) {
            store_columns<R, SPB, M::THREADS>(a, sinfo, [&](int x, int y, int k, int sl) {
                return ubuf[level_at<R>(k, (x & 1) + 2 * (y & 1), sl * TPS + (x >> 1) + NB * (y >> 1))];
            });
        }
        bar();                                     // red (and stage) complete; xbuf is free for the next source
        finish_sigma<TPS, SPB, M::ZS, PT>(red, first, end(), a.list, a.sigma);
    }
    if constexpr (G > 1) {
        store_columns<R, G, M::THREADS>(a, sinfo, [&](int x, int y, int k, int sl) {
            const Word w = stage[G * (x + W1 * (y + W1 * k)) + sl];
            if constexpr (G == 4) return a.store == Store::F16 ? __half2float(__ushort_as_half(w))
                                                               : __bfloat162float(__ushort_as_bfloat16(w));
            else return w;
        });
        bar();                                     // sinfo is free for the next group
    }
    }
}

template <int R, bool COARSE, int G, bool SPREAD>
__global__ void __launch_bounds__(MapTm<R>::THREADS, 1) march_tm_kernel(MarchArgs a) {
    using M = MapTm<R>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ uint32_t s_taddr;
    const int warp = threadIdx.x >> 5;
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
    if constexpr (M::ZS == 1) {
        march_part<R, COARSE, G, SPREAD, 0, M::W1>(a, smem_raw, tbase);
    } else {
        if (warp < M::PT / 32) march_part<R, COARSE, G, SPREAD, 0, M::LO>(a, smem_raw, tbase);
        else march_part<R, COARSE, G, SPREAD, M::LO, M::W1 - M::LO>(a, smem_raw, tbase);
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" :: "r"(taddr) : "memory");
}

// Sources of a CTA when a launch of nsrc is spread evenly over as many waves of CTAs as full ones (of spb) need.
int even_spb(int64_t nsrc, int spb, int num_sms) {
    const int64_t wave = (int64_t)num_sms * spb, ctas = (nsrc + wave - 1) / wave * num_sms;
    return (int)((nsrc + ctas - 1) / ctas);
}

template <int R, bool COARSE, int G, bool SPREAD>
cudaError_t launch_tm(const MarchArgs& a, int num_sms, cudaStream_t st) {
    using M = MapTm<R>;
    const int64_t nsrc = a.src_end - a.src_begin;
    if (nsrc <= 0) return cudaSuccess;
    const size_t smem = COARSE ? M::SMEM_COARSE : G > 1 ? M::SMEM_GROUP : M::SMEM;
    auto kernel = march_tm_kernel<R, COARSE, G, SPREAD>;
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, M::THREADS, smem);
    if (e != cudaSuccess) return e;
    if (per_sm != 1) return cudaErrorInvalidConfiguration;   // TMEM allocation assumes one CTA per SM
    MarchArgs b = a;
    b.spb = SPREAD ? even_spb(nsrc, M::SPB, num_sms) : M::SPB;
    const int64_t nbatch = (nsrc + b.spb * G - 1) / (b.spb * G);
    const int64_t grid = nbatch < (int64_t)num_sms ? nbatch : (int64_t)num_sms;
    kernel<<<(unsigned)grid, M::THREADS, smem, st>>>(b);
    return cudaGetLastError();
}

template <int R>
cudaError_t launch_tm(const MarchArgs& a, int num_sms, cudaStream_t st) {
    using M = MapTm<R>;
    const int64_t nsrc = a.src_end - a.src_begin;
    // Coarse blocks are few: shares at every radius (us a build, 60 substeps, full CTAs -> shares: 30^3, B = 3, R = 2
    // 175 -> 33; B = 5, R = 5 124 -> 62; 60 x 50 x 40, B = 5, R = 2 330 -> 79).
    if (a.coarse_B > 0) return launch_tm<R, true, 1, (M::SPB > 1)>(a, num_sms, st);
    if constexpr (M::ZS > 1) {
        // Groups where a last, partly filled wave of them costs less than a tenth; source-indexed columns are adjacent
        // whatever the order of the stores is, and gain the same.
        const int G = a.store == Store::F32 ? 2 : 4;
        if (nsrc >= (int64_t)num_sms * G * 10)
            return G == 2 ? launch_tm<R, false, 2, false>(a, num_sms, st) : launch_tm<R, false, 4, false>(a, num_sms, st);
    }
    if constexpr (R <= 4) {
        // A launch that does not fill every CTA: an even share each, warps without a source out of the march (us, 60
        // substeps, BF16, full CTAs -> shares: 1000 sources R = 1 32 -> 18, R = 2 39 -> 23, R = 3 53 -> 27; 512 sources
        // R = 4 63 -> 33; 8000 sources R = 3 145 -> 141).  In a kernel of its own: the loop of full CTAs loses 3% to it.
        // From R = 5 on a CTA is full with 7 sources and less.
        if (nsrc > 0 && even_spb(nsrc, M::SPB, num_sms) < M::SPB) return launch_tm<R, false, 1, true>(a, num_sms, st);
    }
    return launch_tm<R, false, 1, false>(a, num_sms, st);
}

}  // namespace

cudaError_t launch_march_blocks(const MarchArgs& a, int num_sms, cudaStream_t st) {
    switch (a.R) {
        case 1: return launch_tm<1>(a, num_sms, st);
        case 2: return launch_tm<2>(a, num_sms, st);
        case 3: return launch_tm<3>(a, num_sms, st);
        case 4: return launch_tm<4>(a, num_sms, st);
        case 5: return launch_tm<5>(a, num_sms, st);
        case 6: return launch_tm<6>(a, num_sms, st);
        case 7: return launch_tm<7>(a, num_sms, st);
        case 8: return launch_tm<8>(a, num_sms, st);
        case 9: return launch_tm<9>(a, num_sms, st);
        case 10: return launch_tm<10>(a, num_sms, st);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace fdirw
