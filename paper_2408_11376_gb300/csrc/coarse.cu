// Coarse-mesh FDiRW (Sec. 3.1, Eqs. 10-15, without the boundary term p_BC c_far).
//
//   nodes      the liquid cells of each B x B x B block form one representative node (B odd; blocks
//              clipped by the domain keep their cells); N_I = liquid cells of block I
//   phase      faces with a non-liquid cell on either side carry no flux; non-liquid cells keep c
//   P          column J: the remapped unit of block J (1 on its liquid cells, Eq. 12) marched n_sub
//              explicit substeps on the block's window widened by R cells, then mapped (Eq. 11):
//              P[I][J] = N_J S_I / (m N_I), S_I the marched mass on block I, m the total.  The march is
//              mapping 4 in coarse mode (march_tm.cu), with convection or one block per SM at most one thread a column
//              (march.cu); P is stored FP64, destination-indexed over the (2 Rc + 1)^3 block offsets, Rc = ceil(R / B)
//   step       mapping (Eq. 13): C_I = mean of c over the liquid cells of block I, FP64 (map_kernel's order);
//              FDiRW calculation (Eq. 14): C'_I = sum_d P[I][I - d] C_{I - d}, FP64 (coarse_gather_kernel's order);
//              re-mapping (Eq. 15): c'_i = C'_I on every liquid cell of block I.
#include "fdirw.h"
#include "fdirw_internal.h"
#include "ctx.h"

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <string>
#include <vector>

using namespace fdirw::host;

namespace fdirw {

struct Coarse {
    int B = 1, Rc = 0, Rw = 0;                   // block side, band radius, march window radius
    int ncx = 0, ncy = 0, ncz = 0;
    int64_t nc = 0, nodes = 0;                   // blocks, blocks with liquid
    uint8_t* liquid = nullptr;                   // N
    int32_t* count = nullptr;                    // nc
    int64_t* list = nullptr;                     // blocks with liquid, ascending
    double* Qc = nullptr;                        // Wc^3 planes of nc values
    double* C = nullptr;                         // nc
    double* Cn = nullptr;                        // nc
    bool built = false;
    // Far-field boundary (open outer surface): lam * open-face conductance per cell, P_BC per block,
    // device scalars [c_far, mass before, mass after], FP32 ping-pong fields of the P_BC march.
    bool open = false;
    double V_far = 0.0;
    float* abnd = nullptr;
    double* pbc = nullptr;
    double* far = nullptr;
    float* ubuf = nullptr;
    // Coupled macro step: FP64 solid-phase face conductances, a scratch field, phase-mass partials.
    double* gs = nullptr;                        // 3 N: +x/+y/+z solid-solid faces
    double* tmp = nullptr;                       // 2 N
    bool gs_ready = false;                       // gs has been computed
    double gs_max = -1.0;                        // largest per-cell sum of gs; negative: not known yet
    double* qpart = nullptr;                     // kMassBlocks
    double* qout = nullptr;                      // [Q_L, Q_S] per step, n_steps_cap * 2
    int64_t qcap = 0;
};

namespace {

int grid_blocks(int64_t n, int threads) {
    int64_t b = (n + threads - 1) / threads;
    if (b > 152 * 16) b = 152 * 16;
    return (int)(b < 1 ? 1 : b);
}

// Coordinates of cell i (32-bit division where it is enough: a 64-bit one per axis cost more than the rest of the
// one-cell-per-thread kernels below).
__device__ __forceinline__ void cell_of(int64_t i, const Grid& g, int& x, int& y, int& z) {
    if (g.n <= 0x7fffffff) {
        const unsigned v = (unsigned)i, r = v / (unsigned)g.nx, q = r / (unsigned)g.ny;
        x = (int)(v - r * (unsigned)g.nx);
        y = (int)(r - q * (unsigned)g.ny);
        z = (int)q;
    } else {
        x = (int)(i % g.nx);
        y = (int)(i / g.nx % g.ny);
        z = (int)(i / ((int64_t)g.nx * g.ny));
    }
}

// The largest of the warps' values (bits of non-negative doubles) into *max_bits, one atomic per warp (one per cell
// serialised on the one address: 569 us for 96^3 cells, 136 so).
__device__ __forceinline__ void max_bits_of(double v, unsigned long long* max_bits) {
    unsigned long long b = (unsigned long long)__double_as_longlong(v);
    for (int off = 16; off > 0; off >>= 1) {
        const unsigned long long o = __shfl_xor_sync(0xffffffffu, b, off);
        b = o > b ? o : b;
    }
    if ((threadIdx.x & 31) == 0) atomicMax(max_bits, b);
}

// Zero the coefficient of every face with a non-liquid cell on either side.
__global__ void mask_faces_kernel(Grid g, const uint8_t* __restrict__ liquid, float* __restrict__ ax,
                                  float* __restrict__ ay, float* __restrict__ az) {
    const int64_t nxy = (int64_t)g.nx * g.ny;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < g.n; i += (int64_t)gridDim.x * blockDim.x) {
        int x, y, z;
        cell_of(i, g, x, y, z);
        const bool l = liquid[i] != 0;
        if (!l || x + 1 >= g.nx || !liquid[i + 1]) ax[i] = 0.f;
        if (!l || y + 1 >= g.ny || !liquid[i + g.nx]) ay[i] = 0.f;
        if (!l || z + 1 >= g.nz || !liquid[i + nxy]) az[i] = 0.f;
    }
}

// Liquid cells per block (one thread per block, cells in z, y, x order).
__global__ void count_kernel(Grid g, const uint8_t* __restrict__ liquid, int B, int ncx, int ncy, int64_t nc,
                             int32_t* __restrict__ count) {
    for (int64_t I = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; I < nc; I += (int64_t)gridDim.x * blockDim.x) {
        const int bx = (int)(I % ncx), by = (int)((I / ncx) % ncy), bz = (int)(I / ((int64_t)ncx * ncy));
        int n = 0;
        for (int z = bz * B; z < min(bz * B + B, g.nz); z++)
            for (int y = by * B; y < min(by * B + B, g.ny); y++)
                for (int x = bx * B; x < min(bx * B + B, g.nx); x++)
                    n += liquid[x + (int64_t)g.nx * (y + (int64_t)g.ny * z)] ? 1 : 0;
        count[I] = n;
    }
}

// Eq. 13: C_I = (sum of c over the liquid cells of block I) / N_I.  LANES lanes per block, 32 / LANES blocks per warp:
// lane l takes the block's (x, y) columns l, l + LANES, ... and walks each in z, then a xor-butterfly.  One thread for a
// block's 125 cells leaves most of a small grid's GPU idle; a whole warp spends the FP64 pipe (16 clocks an instruction
// and SM) on sums and divisions of idle lanes.  B = 5, us at 96^3 / 192^3: one thread 27 / 48, a warp 14 / 80, eight lanes
// 11 / 34.
template <int LANES>
__global__ void map_kernel(Grid g, const uint8_t* __restrict__ liquid, int B, int ncx, int ncy, int64_t nc,
                           const int32_t* __restrict__ count, const double* __restrict__ c, double* __restrict__ C) {
    constexpr int NB = 32 / LANES;
    const int lane = threadIdx.x & 31, l = lane % LANES;
    const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5), nxy = (int64_t)g.nx * g.ny;
    Grid blocks = g;
    blocks.nx = ncx;
    blocks.ny = ncy;
    blocks.n = nc;
    for (int64_t w = blockIdx.x * (int64_t)(blockDim.x >> 5) + (threadIdx.x >> 5); NB * w < nc; w += warps) {
        const int64_t I = NB * w + lane / LANES;
        double s = 0.0;
        if (I < nc) {
            int bx, by, bz;
            cell_of(I, blocks, bx, by, bz);
            if constexpr (LANES == 1) {
                for (int z = bz * B; z < min(bz * B + B, g.nz); z++)
                    for (int y = by * B; y < min(by * B + B, g.ny); y++)
                        for (int x = bx * B; x < min(bx * B + B, g.nx); x++) {
                            const int64_t i = x + (int64_t)g.nx * y + nxy * z;
                            if (liquid[i]) s += c[i];
                        }
            } else {
                const int nz = min(B, g.nz - bz * B);
                for (int e = l; e < B * B; e += LANES) {
                    const int dy = e / B, x = bx * B + e - dy * B, y = by * B + dy;
                    if (x >= g.nx || y >= g.ny) continue;
                    const int64_t i = x + (int64_t)g.nx * y + nxy * ((int64_t)bz * B);
#pragma unroll 5
                    for (int z = 0; z < nz; z++)
                        if (liquid[i + z * nxy]) s += c[i + z * nxy];
                }
            }
        }
#pragma unroll
        for (int off = 1; off < LANES; off <<= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
        if (l == 0 && I < nc) C[I] = count[I] > 0 ? s / (double)count[I] : 0.0;
    }
}

// Open faces: gb_i = D_i times the faces of liquid cell i on the grid's outer surface; abnd = fp32(lam gb)
// (one rounding, as the face coefficients); the largest per-cell sum of masked face conductances plus gb
// (bits of a non-negative double, for atomicMax) for the stability check.
__global__ void open_faces_kernel(Grid g, const double* __restrict__ D, const uint8_t* __restrict__ liquid,
                                  double lam, float* __restrict__ abnd, unsigned long long* __restrict__ max_bits) {
    const int64_t nxy = (int64_t)g.nx * g.ny;
    double most = 0.0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < g.n; i += (int64_t)gridDim.x * blockDim.x) {
        int x, y, z;
        cell_of(i, g, x, y, z);
        double gb = 0.0, sum = 0.0;
        if (liquid[i]) {
            const int faces = (x == 0) + (x == g.nx - 1) + (y == 0) + (y == g.ny - 1) + (z == 0) + (z == g.nz - 1);
            gb = D[i] * (double)faces;
            auto face = [&](int64_t j) {
                const double a = D[i], b = D[j];
                return (liquid[j] && a + b > 0.0) ? 2.0 * a * b / (a + b) : 0.0;
            };
            if (x > 0) sum += face(i - 1);
            if (x + 1 < g.nx) sum += face(i + 1);
            if (y > 0) sum += face(i - g.nx);
            if (y + 1 < g.ny) sum += face(i + g.nx);
            if (z > 0) sum += face(i - nxy);
            if (z + 1 < g.nz) sum += face(i + nxy);
            sum += gb;
        }
        abnd[i] = (float)(lam * gb);
        most = fmax(most, sum);
    }
    max_bits_of(most, max_bits);
}

// One explicit substep of the liquid phase over the whole grid with every far-field ghost at 1 (the
// P_BC march): u' = u + (am u + sum c u_nb + abnd), am = -(sum of the cell's coefficients + abnd), in the
// FP32 increment form and association of the windowed kernels.
// FLOW (convection): the inflow from the upper neighbour uses B and the diagonal sums the cell's outflows (A of its
// +faces, B of its -faces), as the block-source march.
// Bound: L2 (the six arrays fit it) and the launch.  A thread walks kPbcZ cells up a z column, the column's u and z faces
// in registers; no index division (one cell per thread with 64-bit ones: 9.8 us a substep at 96^3, 5.4 so).
constexpr int kPbcZ = 6;
template <bool FLOW>
__global__ void __launch_bounds__(256) pbc_substep_kernel(Grid g, const float* __restrict__ ax, const float* __restrict__ ay,
                                                          const float* __restrict__ az, const float* __restrict__ bx,
                                                          const float* __restrict__ by, const float* __restrict__ bz,
                                                          const float* __restrict__ abnd, const float* __restrict__ u,
                                                          float* __restrict__ un) {
    const int x = blockIdx.x * 32 + (threadIdx.x & 31);
    if (x >= g.nx) return;
    const int64_t nxy = (int64_t)g.nx * g.ny;
    for (int64_t y = blockIdx.y * 8 + (threadIdx.x >> 5); y < g.ny; y += gridDim.y * 8)
    for (int64_t z0 = blockIdx.z * kPbcZ; z0 < g.nz; z0 += gridDim.z * kPbcZ) {
        int64_t i = x + (int64_t)g.nx * y + nxy * z0;
        const float* ux = FLOW ? bx : ax;                 // coefficient of the upper neighbour in this cell
        const float* uy = FLOW ? by : ay;
        const float* uz = FLOW ? bz : az;
        const bool xm = x > 0, xp = x + 1 < g.nx, ym = y > 0, yp = y + 1 < g.ny;
        float czm = z0 > 0 ? az[i - nxy] : 0.f, ozm = FLOW && z0 > 0 ? uz[i - nxy] : czm;
        float below = z0 > 0 ? u[i - nxy] : 0.f, cur = u[i];
        const int64_t z1 = z0 + kPbcZ < g.nz ? z0 + kPbcZ : g.nz;
        for (int64_t z = z0; z < z1; z++, i += nxy) {
            const bool zp = z + 1 < g.nz;
            const float above = zp ? u[i + nxy] : 0.f;
            const float cxm = xm ? ax[i - 1] : 0.f, cxp = xp ? ux[i] : 0.f;
            const float cym = ym ? ay[i - g.nx] : 0.f, cyp = yp ? uy[i] : 0.f;
            const float czp = zp ? uz[i] : 0.f;
            // outflows: the cell's own +faces (A) and the lower neighbours' B; equal to the inflows without flow
            const float oxm = FLOW && xm ? ux[i - 1] : cxm, oxp = FLOW && xp ? ax[i] : cxp;
            const float oym = FLOW && ym ? uy[i - g.nx] : cym, oyp = FLOW && yp ? ay[i] : cyp;
            const float ozp = FLOW && zp ? az[i] : czp;
            const float vb = abnd[i];
            const float am = -((((oxm + oxp) + (oym + oyp)) + (ozm + ozp)) + vb);
            float v = am * cur;
            v = fmaf(cxm, xm ? u[i - 1] : 0.f, v);
            v = fmaf(cxp, xp ? u[i + 1] : 0.f, v);
            v = fmaf(cym, ym ? u[i - g.nx] : 0.f, v);
            v = fmaf(cyp, yp ? u[i + g.nx] : 0.f, v);
            v = fmaf(czm, below, v);
            v = fmaf(czp, above, v);
            v = __fadd_rn(v, vb);                           // inflow from the ghosts at c_far = 1
            un[i] = __fadd_rn(cur, v);
            below = cur;
            cur = above;
            czm = ozp;                                      // the face's A, into the cell above
            ozm = czp;                                      // its B, out of it
        }
    }
}

__global__ void widen_kernel(const float* __restrict__ u, int64_t n, double* __restrict__ out) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        out[i] = (double)u[i];
}

// Interface exchange of Eqs. 4-6 on every liquid/solid face, pre-step values, rate over dt; each cell adds
// its faces' transfers in the order -z, -y, -x, +x, +y, +z (the order in which a raster sweep over the
// lower cell of each face reaches them), f_L and f_S clamped at 0.  FP64 without contraction.
//
// The factor of a cell, k f_L of a liquid one and f_S of a solid one, is formed once per cell that has an interface face:
// two FP64 divisions on either side of every face were what the exchange spent its time on (the FP64 pipe runs at 1/73 of
// the FP32 rate): 96^3, 237 us a step before, 78 us for both kernels now.
__global__ void rate_kernel(Grid g, const uint8_t* __restrict__ liquid, double k, double cS, double cL,
                            const double* __restrict__ c, double* __restrict__ rate) {
    const int64_t nxy = (int64_t)g.nx * g.ny;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < g.n; i += (int64_t)gridDim.x * blockDim.x) {
        int x, y, z;
        cell_of(i, g, x, y, z);
        const bool l = liquid[i] != 0;
        auto other = [&](int64_t j) { return (liquid[j] != 0) != l; };
        const bool edge = (z > 0 && other(i - nxy)) || (y > 0 && other(i - g.nx)) || (x > 0 && other(i - 1)) ||
                          (x + 1 < g.nx && other(i + 1)) || (y + 1 < g.ny && other(i + g.nx)) ||
                          (z + 1 < g.nz && other(i + nxy));
        if (!edge) continue;
        const double v = c[i];
        rate[i] = l ? __dmul_rn(k, v > cL ? __ddiv_rn(__dadd_rn(v, -cL), cL) : 0.0)
                    : v < cS ? __ddiv_rn(__dadd_rn(cS, -v), cS) : 0.0;
    }
}

__global__ void absorb_kernel(Grid g, const uint8_t* __restrict__ liquid, double dt, const double* __restrict__ rate,
                              const double* __restrict__ c, double* __restrict__ out) {
    const int64_t nxy = (int64_t)g.nx * g.ny;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < g.n; i += (int64_t)gridDim.x * blockDim.x) {
        int x, y, z;
        cell_of(i, g, x, y, z);
        const bool l = liquid[i] != 0;
        double v = c[i];                                 // the liquid side loses, the solid side gains
        // transfer from the liquid cell to the solid one across the face to cell j; none unless the phases differ
        auto face = [&](int64_t j) {
            if ((liquid[j] != 0) == l) return;
            const double m = __dmul_rn(__dmul_rn(rate[i], rate[j]), dt);
            v = l ? __dsub_rn(v, m) : __dadd_rn(v, m);
        };
        if (z > 0) face(i - nxy);
        if (y > 0) face(i - g.nx);
        if (x > 0) face(i - 1);
        if (x + 1 < g.nx) face(i + 1);
        if (y + 1 < g.ny) face(i + g.nx);
        if (z + 1 < g.nz) face(i + nxy);
        out[i] = v;
    }
}

// FP64 harmonic conductances of the faces between two solid cells (+x, +y, +z of each cell).
__global__ void solid_faces_kernel(Grid g, const double* __restrict__ D, const uint8_t* __restrict__ liquid,
                                   double* __restrict__ gx, double* __restrict__ gy, double* __restrict__ gz) {
    const int64_t nxy = (int64_t)g.nx * g.ny;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < g.n; i += (int64_t)gridDim.x * blockDim.x) {
        int x, y, z;
        cell_of(i, g, x, y, z);
        auto h = [&](int64_t j) {
            const double a = D[i], b = D[j];
            return (!liquid[i] && !liquid[j] && __dadd_rn(a, b) > 0.0)
                       ? __ddiv_rn(__dmul_rn(__dmul_rn(2.0, a), b), __dadd_rn(a, b)) : 0.0;
        };
        gx[i] = x + 1 < g.nx ? h(i + 1) : 0.0;
        gy[i] = y + 1 < g.ny ? h(i + g.nx) : 0.0;
        gz[i] = z + 1 < g.nz ? h(i + nxy) : 0.0;
    }
}

// One flux-form substep of the solid phase, FP64, faces in the order -x, +x, -y, +y, -z, +z.
__global__ void solid_substep_kernel(Grid g, const double* __restrict__ gx, const double* __restrict__ gy,
                                     const double* __restrict__ gz, double lam, const double* __restrict__ u,
                                     double* __restrict__ un) {
    const int64_t nxy = (int64_t)g.nx * g.ny;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < g.n; i += (int64_t)gridDim.x * blockDim.x) {
        int x, y, z;
        cell_of(i, g, x, y, z);
        const double ui = u[i];
        double acc = 0.0;
        if (x > 0) acc = __dadd_rn(acc, __dmul_rn(gx[i - 1], __dadd_rn(u[i - 1], -ui)));
        if (x + 1 < g.nx) acc = __dadd_rn(acc, __dmul_rn(gx[i], __dadd_rn(u[i + 1], -ui)));
        if (y > 0) acc = __dadd_rn(acc, __dmul_rn(gy[i - g.nx], __dadd_rn(u[i - g.nx], -ui)));
        if (y + 1 < g.ny) acc = __dadd_rn(acc, __dmul_rn(gy[i], __dadd_rn(u[i + g.nx], -ui)));
        if (z > 0) acc = __dadd_rn(acc, __dmul_rn(gz[i - nxy], __dadd_rn(u[i - nxy], -ui)));
        if (z + 1 < g.nz) acc = __dadd_rn(acc, __dmul_rn(gz[i], __dadd_rn(u[i + nxy], -ui)));
        un[i] = __dadd_rn(ui, __dmul_rn(lam, acc));
    }
}

// Largest per-cell sum of the solid-solid conductances (bits of a non-negative double).
__global__ void solid_max_kernel(Grid g, const double* __restrict__ gx, const double* __restrict__ gy,
                                 const double* __restrict__ gz, unsigned long long* __restrict__ max_bits) {
    const int64_t nxy = (int64_t)g.nx * g.ny;
    double most = 0.0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < g.n; i += (int64_t)gridDim.x * blockDim.x) {
        int x, y, z;
        cell_of(i, g, x, y, z);
        double sum = __dadd_rn(__dadd_rn(gx[i], gy[i]), gz[i]);
        if (x > 0) sum = __dadd_rn(sum, gx[i - 1]);
        if (y > 0) sum = __dadd_rn(sum, gy[i - g.nx]);
        if (z > 0) sum = __dadd_rn(sum, gz[i - nxy]);
        most = fmax(most, sum);
    }
    max_bits_of(most, max_bits);
}

// Fixed-order FP64 totals of a field's liquid cells, of its solid ones and of all (in one pass: the total in the order of
// launch_mass): block b sums chunk b, then one block sums the partials.
__global__ void __launch_bounds__(256) phase_partial_kernel(const double* __restrict__ c, const uint8_t* __restrict__ liquid,
                                                            int64_t n, double* __restrict__ partials,
                                                            double* __restrict__ totals) {
    __shared__ double sh[3][8];
    const int64_t chunk = (n + gridDim.x - 1) / gridDim.x;
    const int64_t lo = blockIdx.x * chunk;
    const int64_t hi = lo + chunk < n ? lo + chunk : n;
    double acc[3] = {0.0, 0.0, 0.0};
    for (int64_t i = lo + threadIdx.x; i < hi; i += blockDim.x) {
        const double v = c[i];
        if (liquid[i]) acc[0] += v; else acc[1] += v;
        acc[2] += v;
    }
#pragma unroll
    for (int q = 0; q < 3; q++) {
        for (int off = 16; off > 0; off >>= 1) acc[q] += __shfl_xor_sync(0xffffffffu, acc[q], off);
        if ((threadIdx.x & 31) == 0) sh[q][threadIdx.x >> 5] = acc[q];
    }
    __syncthreads();
    if (threadIdx.x < 32) {
#pragma unroll
        for (int q = 0; q < 3; q++) {
            double v = threadIdx.x < (blockDim.x >> 5) ? sh[q][threadIdx.x] : 0.0;
            for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
            if (threadIdx.x == 0) (q == 2 ? totals : partials + q * kMassBlocks)[blockIdx.x] = v;
        }
    }
}

// phases: [Q_L, Q_S] of the step; the total is the mass after it, far[2], for Eq. 7's update of far[0].
__global__ void __launch_bounds__(kMassBlocks) phase_final_kernel(const double* __restrict__ partials,
                                                                  const double* __restrict__ totals, double* phases,
                                                                  double* far, double V_far) {
    __shared__ double sh[3][kMassBlocks / 32];
#pragma unroll
    for (int q = 0; q < 3; q++) {
        double v = (q == 2 ? totals : partials + q * kMassBlocks)[threadIdx.x];
        for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
        if ((threadIdx.x & 31) == 0) sh[q][threadIdx.x >> 5] = v;
    }
    __syncthreads();
    if (threadIdx.x < 32) {
#pragma unroll
        for (int q = 0; q < 3; q++) {
            double w = sh[q][threadIdx.x];
            for (int off = 16; off > 0; off >>= 1) w += __shfl_xor_sync(0xffffffffu, w, off);
            if (threadIdx.x == 0) {
                if (q < 2) {
                    phases[q] = w;
                } else {
                    far[2] = w;
                    far[0] = ((far[1] + V_far * far[0]) - w) / V_far;
                }
            }
        }
    }
}

// Eq. 7 for the step just taken: c_far = (m_in + V_far c_far - m_out) / V_far.
__global__ void far_update_kernel(double* far, double V_far) {
    far[0] = ((far[1] + V_far * far[0]) - far[2]) / V_far;
}

// Eq. 14: C'_I = sum over block offsets d of P[I][I - d] C_{I - d}, FP64, plus P_BC[I] c_far when the outer surface is
// open.  PARTS = 8: a CTA takes 32 consecutive blocks, a lane each; warp w adds the offsets d = w, w + 8, ... in ascending
// order, then the eight sums go pairwise.  PARTS = 1: one thread takes all offsets of a block in ascending order.  In both
// a warp reads 32 consecutive values of a plane.
template <int PARTS>
__global__ void __launch_bounds__(PARTS == 1 ? 128 : 32 * PARTS) coarse_gather_kernel(int ncx, int ncy, int ncz, int Rc,
                                                                                      const double* __restrict__ Qc,
                                                                                      const double* __restrict__ C,
                                                                                      const double* __restrict__ pbc,
                                                                                      const double* __restrict__ far,
                                                                                      double* __restrict__ Cn) {
    constexpr int LANES = PARTS == 1 ? 128 : 32;
    __shared__ double sums[PARTS][LANES];
    const int64_t nc = (int64_t)ncx * ncy * ncz;
    const int Wc = 2 * Rc + 1, n = Wc * Wc * Wc, lane = threadIdx.x % LANES, part = threadIdx.x / LANES;
    const Grid blocks{ncx, ncy, ncz, nc};
    for (int64_t I0 = (int64_t)blockIdx.x * LANES; I0 < nc; I0 += (int64_t)gridDim.x * LANES) {
        const int64_t I = I0 + lane;
        double acc = 0.0;
        if (I < nc) {
            int bx, by, bz;
            cell_of(I, blocks, bx, by, bz);
            auto in = [](int v, int m) { return (unsigned)v < (unsigned)m; };
            auto add = [&](int d, int jx, int jy, int jz) {
                if (in(jx, ncx) && in(jy, ncy) && in(jz, ncz))
                    acc = fma(Qc[(int64_t)d * nc + I], C[jx + (int64_t)ncx * (jy + (int64_t)ncy * jz)], acc);
            };
            if constexpr (PARTS == 1) {
                int d = 0;
                for (int dz = -Rc; dz <= Rc; dz++)
                    for (int dy = -Rc; dy <= Rc; dy++)
                        for (int dx = -Rc; dx <= Rc; dx++, d++) add(d, bx - dx, by - dy, bz - dz);
            } else {
                int dx = part % Wc, dy = part / Wc % Wc, dz = part / (Wc * Wc);      // offset d + Rc
                for (int d = part; d < n; d += PARTS) {
                    add(d, bx + Rc - dx, by + Rc - dy, bz + Rc - dz);
                    for (dx += PARTS; dx >= Wc;) {
                        dx -= Wc;
                        if (++dy == Wc) { dy = 0; dz++; }
                    }
                }
            }
        }
        if constexpr (PARTS > 1) {
            sums[part][lane] = acc;
            __syncthreads();
            if (part == 0)
                acc = ((sums[0][lane] + sums[1][lane]) + (sums[2][lane] + sums[3][lane])) +
                      ((sums[4][lane] + sums[5][lane]) + (sums[6][lane] + sums[7][lane]));
            __syncthreads();
        }
        if (part == 0 && I < nc) {
            if (pbc) acc = __dadd_rn(acc, __dmul_rn(pbc[I], far[0]));
            Cn[I] = acc;
        }
    }
}

// Eq. 15: c'_i = C'_I on liquid cells, c'_i = c_i elsewhere (in place allowed: each cell reads itself).
__global__ void remap_kernel(Grid g, const uint8_t* __restrict__ liquid, int B, int ncx, int ncy,
                             const double* __restrict__ Cn, const double* c_in, double* c_out) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < g.n; i += (int64_t)gridDim.x * blockDim.x) {
        int x, y, z;
        cell_of(i, g, x, y, z);
        c_out[i] = liquid[i] ? Cn[(x / B) + (int64_t)ncx * ((y / B) + (int64_t)ncy * (z / B))] : c_in[i];
    }
}

// Columns of P for listed blocks on the source-major band layout [n][Wc^3] (offset d = I - J).
__global__ void read_coarse_kernel(const double* __restrict__ Qc, int ncx, int ncy, int ncz, int Rc,
                                   const int64_t* __restrict__ blocks, int64_t n, double* __restrict__ out) {
    const int Wc = 2 * Rc + 1;
    const int64_t W3 = (int64_t)Wc * Wc * Wc, nc = (int64_t)ncx * ncy * ncz;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n * W3; t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t q = t / W3;
        const int d = (int)(t % W3);
        const int64_t J = blocks[q];
        const int bx = (int)(J % ncx), by = (int)((J / ncx) % ncy), bz = (int)(J / ((int64_t)ncx * ncy));
        const int cx = bx + d % Wc - Rc, cy = by + (d / Wc) % Wc - Rc, cz = bz + d / (Wc * Wc) - Rc;
        double v = 0.0;
        if (cx >= 0 && cx < ncx && cy >= 0 && cy < ncy && cz >= 0 && cz < ncz)
            v = Qc[(int64_t)d * nc + cx + (int64_t)ncx * (cy + (int64_t)ncy * cz)];
        out[t] = v;
    }
}

// Lanes per block: few blocks leave the GPU idle with one each; of many, lanes that share a block's sum cost FP64
// instructions (16 clocks each on an SM) that add nothing.  us, 1 / 4 / 8 lanes: B = 5 96^3 (8000 blocks) 21 / 10 / 10,
// 128^3 (18k) 27 / 12 / 14, 224^3 (91k) 33 / 42 / 51; B = 3 64^3 (11k) 10 / 8 / 8, 96^3 (33k) 10 / 10 / 12, 160^3 (157k)
// 16 / 29 / 45; B = 1 96^3 33 / 119 / 244.
cudaError_t launch_map(fdirw_ctx* c, const double* field, double* means) {
    const Coarse& k = *c->coarse;
    auto launch = [&](auto kernel, int lanes, int threads) {
        kernel<<<grid_blocks(k.nc, threads / lanes), threads, 0, c->stream>>>(c->g, k.liquid, k.B, k.ncx, k.ncy, k.nc, k.count,
                                                                              field, means);
        return cudaGetLastError();
    };
    if (k.B == 1 || k.nc > 40000) return launch(map_kernel<1>, 1, 128);
    if (k.nc > 12000) return launch(map_kernel<4>, 4, 256);
    return launch(map_kernel<8>, 8, 256);
}

// Eight threads per block where one each leaves the chain of a block's terms bare, that is with few blocks or many terms.
// us, 1 / 8: Rc = 1 8000 blocks 8 / 6, 157k 13 / 21, 885k 72 / 113; Rc = 2 8000 23 / 8, 33k 23 / 14, 157k 53 / 59, 885k 279 /
// 310; Rc = 3 8000 51 / 17, 80k 119 / 70, 262k 247 / 213, 885k 718 / 722.
cudaError_t launch_coarse_gather(fdirw_ctx* c) {
    const Coarse& k = *c->coarse;
    const double* pbc = k.open ? k.pbc : nullptr;
    if (k.nc <= 40000 || k.Rc >= 3)
        coarse_gather_kernel<8><<<grid_blocks(k.nc, 32), 256, 0, c->stream>>>(k.ncx, k.ncy, k.ncz, k.Rc, k.Qc, k.C, pbc, k.far, k.Cn);
    else
        coarse_gather_kernel<1><<<grid_blocks(k.nc, 128), 128, 0, c->stream>>>(k.ncx, k.ncy, k.ncz, k.Rc, k.Qc, k.C, pbc, k.far, k.Cn);
    return cudaGetLastError();
}

}  // namespace

int coarse_kernels(fdirw_ctx* c) {
    Coarse& k = *c->coarse;
    if (k.built) return FDIRW_OK;
    const uint64_t W3 = (uint64_t)(2 * k.Rc + 1) * (2 * k.Rc + 1) * (2 * k.Rc + 1);
    FDIRW_CUDA(c, cudaMemsetAsync(k.Qc, 0, W3 * (uint64_t)k.nc * 8, c->stream));
    MarchArgs a{};
    a.g = c->g;
    a.R = k.Rw;
    a.Rq = k.Rw;
    a.n_sub = c->n_sub;
    a.ax = reinterpret_cast<const float*>(c->coef[0]);
    a.ay = reinterpret_cast<const float*>(c->coef[1]);
    a.az = reinterpret_cast<const float*>(c->coef[2]);
    a.src_begin = 0;
    a.src_end = k.nodes;
    a.list = k.list;
    a.coarse_B = k.B;
    a.coarse_Rc = k.Rc;
    a.ncx = k.ncx;
    a.ncy = k.ncy;
    a.ncz = k.ncz;
    a.coarse_n = k.nc;
    a.liquid = k.liquid;
    a.ccount = k.count;
    a.Qc = k.Qc;
    a.abnd = k.open ? k.abnd : nullptr;
    if (c->flow) {                                     // convection: direction-dependent faces
        a.bx = reinterpret_cast<const float*>(c->coefb[0]);
        a.by = reinterpret_cast<const float*>(c->coefb[1]);
        a.bz = reinterpret_cast<const float*>(c->coefb[2]);
    }
    FDIRW_CUDA(c, cudaEventRecord(c->ev[0], c->stream));
    if (k.nodes > 0 && c->n_sub >= 0) FDIRW_CUDA(c, launch_march_coarse(a, k.Rw, c->num_sms, c->stream));
    FDIRW_CUDA(c, cudaEventRecord(c->ev[1], c->stream));
    if (k.open) {
        // P_BC: the liquid from 0 with every ghost at 1, n_sub substeps over the whole grid, then Eq. 11.
        float* u0 = k.ubuf;
        float* u1 = k.ubuf + c->g.n;
        FDIRW_CUDA(c, cudaMemsetAsync(u0, 0, (size_t)c->g.n * 4, c->stream));
        const dim3 tiles((c->g.nx + 31) / 32, std::min((c->g.ny + 7) / 8, 65535), std::min((c->g.nz + kPbcZ - 1) / kPbcZ, 65535));
        for (int t = 0; t < c->n_sub; t++) {
            (a.bx ? pbc_substep_kernel<true> : pbc_substep_kernel<false>)<<<tiles, 256, 0, c->stream>>>(
                c->g, a.ax, a.ay, a.az, a.bx, a.by, a.bz, k.abnd, u0, u1);
            FDIRW_CUDA(c, cudaGetLastError());
            std::swap(u0, u1);
        }
        widen_kernel<<<grid_blocks(c->g.n, 256), 256, 0, c->stream>>>(u0, c->g.n, c->cbuf);
        FDIRW_CUDA(c, launch_map(c, c->cbuf, k.pbc));
    }
    c->kernels_timed = true;
    c->parts_used = c->flow || k.nodes <= c->num_sms ? 5 : 4;
    k.built = true;
    c->kernels_ready = true;
    return FDIRW_OK;
}

// phases (nullable, device): receives the liquid and the solid total of c_out after the last step (far field only).
static int coarse_steps(fdirw_ctx* c, const double* c_in, double* c_out, int32_t n_steps, double* mass_out, double* phases) {
    Coarse& k = *c->coarse;
    const Kind kin = classify(c_in, c->device), kout = classify(c_out, c->device);
    if (kin == Kind::Foreign || kout == Kind::Foreign)
        return fail(c, FDIRW_ERR_ARG, "c_in/c_out are device memory of another device");
    if (!k.built) {
        const int rc = coarse_kernels(c);
        if (rc != FDIRW_OK) return rc;
    }
    const size_t bytes = (size_t)c->g.n * 8;
    const double* src = c_in;
    if (kin == Kind::Host) {
        FDIRW_CUDA(c, cudaMemcpyAsync(c->cbuf, c_in, bytes, cudaMemcpyHostToDevice, c->stream));
        src = c->cbuf;
    }
    double* dst = kout == Kind::Device ? c_out : c->cbuf;
    if (mass_out) {
        FDIRW_CUDA(c, launch_mass(src, c->g.n, c->partials, c->dmass, c->stream));
        FDIRW_CUDA(c, cudaMemcpyAsync(&c->mass_in, c->dmass, 8, cudaMemcpyDeviceToHost, c->stream));
    }
    if (n_steps == 0) {
        if (dst != src) FDIRW_CUDA(c, cudaMemcpyAsync(dst, src, bytes, cudaMemcpyDeviceToDevice, c->stream));
    } else {
        const double* cur = src;
        for (int t = 0; t < n_steps; t++) {
            FDIRW_CUDA(c, launch_map(c, cur, k.C));
            const bool last = t + 1 == n_steps;
            if (last) FDIRW_CUDA(c, cudaEventRecord(c->ev[2], c->stream));
            if (k.open) FDIRW_CUDA(c, launch_mass(cur, c->g.n, c->partials, k.far + 1, c->stream));
            FDIRW_CUDA(c, launch_coarse_gather(c));
            if (last) FDIRW_CUDA(c, cudaEventRecord(c->ev[3], c->stream));
            remap_kernel<<<grid_blocks(c->g.n, 256), 256, 0, c->stream>>>(c->g, k.liquid, k.B, k.ncx, k.ncy, k.Cn, cur, dst);
            FDIRW_CUDA(c, cudaGetLastError());
            if (k.open && phases && last) {
                phase_partial_kernel<<<kMassBlocks, 256, 0, c->stream>>>(dst, k.liquid, c->g.n, c->partials, k.qpart);
                phase_final_kernel<<<1, kMassBlocks, 0, c->stream>>>(c->partials, k.qpart, phases, k.far, k.V_far);
                FDIRW_CUDA(c, cudaGetLastError());
            } else if (k.open) {
                FDIRW_CUDA(c, launch_mass(dst, c->g.n, c->partials, k.far + 2, c->stream));
                far_update_kernel<<<1, 1, 0, c->stream>>>(k.far, k.V_far);
                FDIRW_CUDA(c, cudaGetLastError());
            }
            cur = dst;
        }
        c->gather_timed = true;
    }
    if (mass_out) {
        FDIRW_CUDA(c, launch_mass(dst, c->g.n, c->partials, c->dmass, c->stream));
        FDIRW_CUDA(c, cudaMemcpyAsync(&c->mass_out, c->dmass, 8, cudaMemcpyDeviceToHost, c->stream));
    }
    if (kout == Kind::Host) FDIRW_CUDA(c, cudaMemcpyAsync(c_out, dst, bytes, cudaMemcpyDeviceToHost, c->stream));
    if (mass_out || kout == Kind::Host) FDIRW_CUDA(c, cudaStreamSynchronize(c->stream));
    if (mass_out) *mass_out = c->mass_out;
    return FDIRW_OK;
}

int coarse_step(fdirw_ctx* c, const double* c_in, double* c_out, int32_t n_steps, double* mass_out) {
    return coarse_steps(c, c_in, c_out, n_steps, mass_out, nullptr);
}

// One liquid step of a coupled macro step on device fields.
static int coarse_coupled(fdirw_ctx* c, const double* c_in, double* c_out, double* phases) {
    return coarse_steps(c, c_in, c_out, 1, nullptr, phases);
}

int coarse_info(fdirw_ctx* c, fdirw_info* out) {
    out->coarse_block = c->coarse->B;
    out->coarse_nodes = c->coarse->nodes;
    out->cache_bytes = (uint64_t)(2 * c->coarse->Rc + 1) * (2 * c->coarse->Rc + 1) * (2 * c->coarse->Rc + 1) *
                       (uint64_t)c->coarse->nc * 8;
    return FDIRW_OK;
}

const uint8_t* coarse_liquid(fdirw_ctx* c) { return c->coarse ? c->coarse->liquid : nullptr; }

const float* coarse_open_faces(fdirw_ctx* c) { return (c->coarse && c->coarse->open) ? c->coarse->abnd : nullptr; }

void coarse_invalidate(fdirw_ctx* c) {
    if (c->coarse) c->coarse->built = false;
}

void coarse_release(fdirw_ctx* c) {
    Coarse* k = c->coarse;
    if (!k) return;
    void* p;
    p = k->liquid; dfree(p);
    p = k->count; dfree(p);
    p = k->list; dfree(p);
    p = k->Qc; dfree(p);
    p = k->C; dfree(p);
    p = k->Cn; dfree(p);
    p = k->abnd; dfree(p);
    p = k->pbc; dfree(p);
    p = k->far; dfree(p);
    p = k->ubuf; dfree(p);
    p = k->gs; dfree(p);
    p = k->tmp; dfree(p);
    p = k->qpart; dfree(p);
    p = k->qout; dfree(p);
    delete k;
    c->coarse = nullptr;
}

}  // namespace fdirw

extern "C" {

int fdirw_create_coarse(const fdirw_grid* grid, const double* D_map, const uint8_t* liquid, int32_t block,
                        double dt_macro, int32_t window_R, int32_t n_sub, const fdirw_opts* opts, fdirw_ctx** out) {
    if (!out) return fail(nullptr, FDIRW_ERR_ARG, "NULL out");
    *out = nullptr;
    if (!grid_ok(grid)) return fail(nullptr, FDIRW_ERR_ARG, "invalid grid (dimensions >= 1, finite h > 0)");
    if (!D_map) return fail(nullptr, FDIRW_ERR_ARG, "NULL D_map");
    if (block < 1 || block % 2 == 0) return fail(nullptr, FDIRW_ERR_ARG, "block must be odd and >= 1");
    if (window_R < 0 || window_R + (block - 1) / 2 > fdirw::kMaxR)
        return fail(nullptr, FDIRW_ERR_ARG, "need 0 <= window_R and window_R + (block - 1) / 2 <= " + std::to_string(fdirw::kMaxR));
    if (window_R + (block - 1) / 2 < 1) return fail(nullptr, FDIRW_ERR_ARG, "window_R + (block - 1) / 2 must be >= 1");
    fdirw_opts o{FDIRW_FP32, -1, nullptr, 0, 0, 0};
    if (opts) o = *opts;
    if (o.prec < FDIRW_FP32 || o.prec > FDIRW_FP32_STORE_BF16)
        return fail(nullptr, FDIRW_ERR_ARG, "the coarse path marches in FP32 (prec FP32, FP16 or BF16; P is FP64)");
    if (o.accum != FDIRW_ACCUM_FF) return fail(nullptr, FDIRW_ERR_ARG, "coarse contexts take FDIRW_ACCUM_FF only");
    // fdirw_create validates D, dt_macro, n_sub and stability and builds the face coefficients; the
    // coarse path then masks them and replaces the kernel cache with the coarse matrix.
    fdirw_opts o2 = o;
    o2.prec = FDIRW_FP32;
    fdirw_ctx* c = nullptr;
    int rc = fdirw_create(grid, D_map, dt_macro, 0, n_sub, &o2, &c);
    if (rc != FDIRW_OK) return rc;
    DeviceGuard dg(c->device);
    c->coarse = new fdirw::Coarse();
    fdirw::Coarse& k = *c->coarse;
    c->R = window_R;
    c->prec = o.prec;
    k.B = block;
    k.Rc = (window_R + block - 1) / block;
    k.Rw = window_R + (block - 1) / 2;
    k.ncx = (grid->nx + block - 1) / block;
    k.ncy = (grid->ny + block - 1) / block;
    k.ncz = (grid->nz + block - 1) / block;
    k.nc = (int64_t)k.ncx * k.ncy * k.ncz;
    const uint64_t n = (uint64_t)c->g.n;
    auto bail = [&](int code) {
        std::string msg = c->err;
        fdirw_destroy(c);
        return fail(nullptr, code, msg);
    };
    if ((rc = dalloc(c, reinterpret_cast<void**>(&k.liquid), n, "liquid mask")) != FDIRW_OK) return bail(rc);
    cudaError_t e = cudaSuccess;
    if (liquid) {
        if (classify(liquid, c->device) == Kind::Foreign) { c->err = "liquid is device memory of another device"; return bail(FDIRW_ERR_ARG); }
        e = cudaMemcpyAsync(k.liquid, liquid, n, cudaMemcpyDefault, c->stream);
    } else {
        e = cudaMemsetAsync(k.liquid, 1, n, c->stream);
    }
    if (e != cudaSuccess) { c->err = cuda_msg("copy liquid mask", e); return bail(FDIRW_ERR_CUDA); }
    if ((rc = dalloc(c, reinterpret_cast<void**>(&k.count), (uint64_t)k.nc * 4, "block counts")) != FDIRW_OK) return bail(rc);
    const uint64_t W3 = (uint64_t)(2 * k.Rc + 1) * (2 * k.Rc + 1) * (2 * k.Rc + 1);
    if ((rc = dalloc(c, reinterpret_cast<void**>(&k.Qc), W3 * (uint64_t)k.nc * 8, "coarse matrix")) != FDIRW_OK) return bail(rc);
    if ((rc = dalloc(c, reinterpret_cast<void**>(&k.C), (uint64_t)k.nc * 8, "coarse field")) != FDIRW_OK) return bail(rc);
    if ((rc = dalloc(c, reinterpret_cast<void**>(&k.Cn), (uint64_t)k.nc * 8, "coarse field")) != FDIRW_OK) return bail(rc);
    fdirw::mask_faces_kernel<<<fdirw::grid_blocks(c->g.n, 256), 256, 0, c->stream>>>(
        c->g, k.liquid, reinterpret_cast<float*>(c->coef[0]), reinterpret_cast<float*>(c->coef[1]),
        reinterpret_cast<float*>(c->coef[2]));
    fdirw::count_kernel<<<fdirw::grid_blocks(k.nc, 128), 128, 0, c->stream>>>(c->g, k.liquid, k.B, k.ncx, k.ncy, k.nc, k.count);
    if ((e = cudaGetLastError()) != cudaSuccess) { c->err = cuda_msg("coarse setup", e); return bail(FDIRW_ERR_CUDA); }
    // Blocks with liquid, ascending (host pass over the counts).
    std::vector<int32_t> cnt((size_t)k.nc);
    if ((e = cudaMemcpyAsync(cnt.data(), k.count, (size_t)k.nc * 4, cudaMemcpyDeviceToHost, c->stream)) != cudaSuccess ||
        (e = cudaStreamSynchronize(c->stream)) != cudaSuccess) {
        c->err = cuda_msg("coarse setup", e);
        return bail(FDIRW_ERR_CUDA);
    }
    std::vector<int64_t> list;
    for (int64_t I = 0; I < k.nc; I++) if (cnt[(size_t)I] > 0) list.push_back(I);
    k.nodes = (int64_t)list.size();
    if (k.nodes > 0) {
        if ((rc = dalloc(c, reinterpret_cast<void**>(&k.list), (uint64_t)k.nodes * 8, "node list")) != FDIRW_OK) return bail(rc);
        if ((e = cudaMemcpy(k.list, list.data(), (size_t)k.nodes * 8, cudaMemcpyHostToDevice)) != cudaSuccess) {
            c->err = cuda_msg("copy node list", e);
            return bail(FDIRW_ERR_CUDA);
        }
    }
    c->kernels_ready = false;
    // Sum over the nodes of their clipped march windows (cells), for the roofline's work count.
    double wc = 0.0;
    for (int64_t I : list) {
        const int bx = (int)(I % k.ncx), by = (int)((I / k.ncx) % k.ncy), bz = (int)(I / ((int64_t)k.ncx * k.ncy));
        auto ext = [&](int b, int n) {
            return (double)(std::min(b * block + block - 1 + window_R, n - 1) - std::max(b * block - window_R, 0) + 1);
        };
        wc += ext(bx, grid->nx) * ext(by, grid->ny) * ext(bz, grid->nz);
    }
    c->window_cells = wc;
    *out = c;
    return FDIRW_OK;
}

int fdirw_coarse_far_field(fdirw_ctx* c, double V_far, double c_far) {
    if (!c) return fail(nullptr, FDIRW_ERR_ARG, "NULL context");
    if (!c->coarse) return fail(c, FDIRW_ERR_ARG, "not a coarse-mesh context");
    if (!(std::isfinite(V_far) && V_far > 0.0) || !std::isfinite(c_far))
        return fail(c, FDIRW_ERR_ARG, "V_far must be finite and > 0, c_far finite");
    DeviceGuard dg(c->device);
    fdirw::Coarse& k = *c->coarse;
    if (c->flow && !k.abnd)
        return fail(c, FDIRW_ERR_STATE, "open the far field before setting a velocity (its stability check includes the flow)");
    const uint64_t n = (uint64_t)c->g.n;
    int rc;
    if (!k.abnd) {
        if ((rc = dalloc(c, reinterpret_cast<void**>(&k.abnd), n * 4, "open-face coefficients")) != FDIRW_OK) return rc;
        if ((rc = dalloc(c, reinterpret_cast<void**>(&k.pbc), (uint64_t)k.nc * 8, "P_BC")) != FDIRW_OK) return rc;
        if ((rc = dalloc(c, reinterpret_cast<void**>(&k.far), 3 * 8, "far field")) != FDIRW_OK) return rc;
        if ((rc = dalloc(c, reinterpret_cast<void**>(&k.ubuf), 2 * n * 4, "P_BC march")) != FDIRW_OK) return rc;
        unsigned long long* mx = nullptr;
        if ((rc = dalloc(c, reinterpret_cast<void**>(&mx), 8, "flags")) != FDIRW_OK) return rc;
        unsigned long long h = 0;
        cudaError_t e = cudaMemsetAsync(mx, 0, 8, c->stream);
        if (e == cudaSuccess) {
            fdirw::open_faces_kernel<<<fdirw::grid_blocks(c->g.n, 256), 256, 0, c->stream>>>(c->g, c->Dd, k.liquid, c->lam,
                                                                                           k.abnd, mx);
            e = cudaGetLastError();
        }
        if (e == cudaSuccess) e = cudaMemcpyAsync(&h, mx, 8, cudaMemcpyDeviceToHost, c->stream);
        const cudaError_t w = cudaStreamSynchronize(c->stream);      // also after a failure: the blocks go to other contexts
        if (e == cudaSuccess) e = w;
        drelease(mx);
        c->allocated -= 8;
        if (e != cudaSuccess) { cudaGetLastError(); return fail(c, FDIRW_ERR_CUDA, cuda_msg("open faces", e)); }
        double m;
        std::memcpy(&m, &h, 8);
        if (c->lam * m > 1.0 + 1e-12) {
            char buf[200];
            std::snprintf(buf, sizeof buf, "unstable with open faces: dt_sub*max(sum g)/h^2 = %.17g > 1", c->lam * m);
            return fail(c, FDIRW_ERR_UNSTABLE, buf);
        }
    }
    const double h3[3] = {c_far, 0.0, 0.0};
    FDIRW_CUDA(c, cudaMemcpyAsync(k.far, h3, 24, cudaMemcpyHostToDevice, c->stream));
    FDIRW_CUDA(c, cudaStreamSynchronize(c->stream));
    k.V_far = V_far;
    if (!k.open) {
        k.open = true;
        k.built = false;                 // the coarse matrix changes with open faces
        c->kernels_ready = false;
    }
    return FDIRW_OK;
}

int fdirw_coarse_get_far_field(fdirw_ctx* c, double* c_far) {
    if (!c || !c_far) return fail(c, FDIRW_ERR_ARG, "NULL context or c_far");
    if (!c->coarse || !c->coarse->open) return fail(c, FDIRW_ERR_STATE, "no far field set (fdirw_coarse_far_field)");
    DeviceGuard dg(c->device);
    FDIRW_CUDA(c, cudaMemcpyAsync(c_far, c->coarse->far, 8, cudaMemcpyDeviceToHost, c->stream));
    FDIRW_CUDA(c, cudaStreamSynchronize(c->stream));
    return FDIRW_OK;
}

int fdirw_read_coarse_pbc(fdirw_ctx* c, double* out) {
    if (!c || !out) return fail(c, FDIRW_ERR_ARG, "NULL context or out");
    if (!c->coarse || !c->coarse->open) return fail(c, FDIRW_ERR_STATE, "no far field set (fdirw_coarse_far_field)");
    if (!c->coarse->built) return fail(c, FDIRW_ERR_STATE, "coarse matrix not built (call fdirw_kernels)");
    DeviceGuard dg(c->device);
    FDIRW_CUDA(c, cudaMemcpyAsync(out, c->coarse->pbc, (size_t)c->coarse->nc * 8, cudaMemcpyDeviceToHost, c->stream));
    FDIRW_CUDA(c, cudaStreamSynchronize(c->stream));
    return FDIRW_OK;
}

int fdirw_coupled_step(fdirw_ctx* c, const fdirw_coupled_params* p, double* field, int32_t n_steps, double* QL,
                       double* QS, double* c_far) {
    if (!c || !p || !field) return fail(c, FDIRW_ERR_ARG, "NULL context, params or field");
    if (!c->coarse || !c->coarse->open)
        return fail(c, FDIRW_ERR_STATE, "the coupled step needs a coarse-mesh context with a far field");
    if (n_steps < 0) return fail(c, FDIRW_ERR_ARG, "n_steps must be >= 0");
    if (!(std::isfinite(p->k) && p->k >= 0.0) || !(std::isfinite(p->cS_eq) && p->cS_eq > 0.0) ||
        !(std::isfinite(p->cL_eq) && p->cL_eq > 0.0) || !(std::isfinite(p->dt) && p->dt >= 0.0) || p->n_sub_solid < 0)
        return fail(c, FDIRW_ERR_ARG, "need k >= 0, cS_eq > 0, cL_eq > 0, dt >= 0, n_sub_solid >= 0");
    if ((reinterpret_cast<uintptr_t>(field) & 7u) != 0) return fail(c, FDIRW_ERR_ARG, "field must be 8-byte aligned");
    DeviceGuard dg(c->device);
    fdirw::Coarse& k = *c->coarse;
    const Kind kf = classify(field, c->device);
    if (kf == Kind::Foreign) return fail(c, FDIRW_ERR_ARG, "field is device memory of another device");
    const uint64_t n = (uint64_t)c->g.n;
    int rc;
    const double lam_s = p->n_sub_solid > 0 ? (p->dt / p->n_sub_solid) / (c->h * c->h) : 0.0;
    if (!k.gs_ready) {
        if (!k.tmp && (rc = dalloc(c, reinterpret_cast<void**>(&k.tmp), 2 * n * 8, "coupled scratch")) != FDIRW_OK) return rc;
        if (!k.qpart && (rc = dalloc(c, reinterpret_cast<void**>(&k.qpart), fdirw::kMassBlocks * 8, "phase partials")) != FDIRW_OK)
            return rc;
        if (!k.gs && (rc = dalloc(c, reinterpret_cast<void**>(&k.gs), 3 * n * 8, "solid faces")) != FDIRW_OK) return rc;
        fdirw::solid_faces_kernel<<<fdirw::grid_blocks(c->g.n, 256), 256, 0, c->stream>>>(c->g, c->Dd, k.liquid, k.gs,
                                                                                        k.gs + n, k.gs + 2 * n);
        FDIRW_CUDA(c, cudaGetLastError());
        k.gs_ready = true;
    }
    if (lam_s > 0.0 && k.gs_max < 0.0) {
        // The largest sum of a cell's solid faces, for the stability check of every call (on the device: copying the
        // 3 N conductances out for a host loop took 8 of a 30 ms call at 96^3).
        unsigned long long h = 0, *mx = reinterpret_cast<unsigned long long*>(k.tmp);
        FDIRW_CUDA(c, cudaMemsetAsync(mx, 0, 8, c->stream));
        fdirw::solid_max_kernel<<<fdirw::grid_blocks(c->g.n, 256), 256, 0, c->stream>>>(c->g, k.gs, k.gs + n, k.gs + 2 * n, mx);
        FDIRW_CUDA(c, cudaGetLastError());
        FDIRW_CUDA(c, cudaMemcpyAsync(&h, mx, 8, cudaMemcpyDeviceToHost, c->stream));
        FDIRW_CUDA(c, cudaStreamSynchronize(c->stream));
        std::memcpy(&k.gs_max, &h, 8);
    }
    if (lam_s > 0.0 && lam_s * k.gs_max > 1.0 + 1e-12)
        return fail(c, FDIRW_ERR_UNSTABLE, "solid march unstable: raise n_sub_solid");
    if ((QL || QS) && n_steps > k.qcap) {
        retire(c, k.qout);
        c->allocated -= (uint64_t)k.qcap * 16;
        k.qcap = 0;
        if ((rc = dalloc(c, reinterpret_cast<void**>(&k.qout), (uint64_t)n_steps * 16, "phase masses")) != FDIRW_OK) return rc;
        k.qcap = n_steps;
    }
    if (!k.built) {
        if ((rc = fdirw::coarse_kernels(c)) != FDIRW_OK) return rc;
    }
    double* cur = field;
    if (kf == Kind::Host) {
        FDIRW_CUDA(c, cudaMemcpyAsync(c->cbuf, field, n * 8, cudaMemcpyHostToDevice, c->stream));
        cur = c->cbuf;
    }
    const int gb = fdirw::grid_blocks(c->g.n, 256);
    for (int t = 0; t < n_steps; t++) {
        fdirw::rate_kernel<<<gb, 256, 0, c->stream>>>(c->g, k.liquid, p->k, p->cS_eq, p->cL_eq, cur, k.tmp + n);
        fdirw::absorb_kernel<<<gb, 256, 0, c->stream>>>(c->g, k.liquid, p->dt, k.tmp + n, cur, k.tmp);
        FDIRW_CUDA(c, cudaGetLastError());
        double* a = k.tmp;
        double* b = k.tmp + n;
        for (int s = 0; s < p->n_sub_solid; s++) {
            fdirw::solid_substep_kernel<<<gb, 256, 0, c->stream>>>(c->g, k.gs, k.gs + n, k.gs + 2 * n, lam_s, a, b);
            FDIRW_CUDA(c, cudaGetLastError());
            std::swap(a, b);
        }
        if ((rc = fdirw::coarse_coupled(c, a, cur, (QL || QS) ? k.qout + 2 * t : nullptr)) != FDIRW_OK) return rc;
    }
    if (kf == Kind::Host) FDIRW_CUDA(c, cudaMemcpyAsync(field, cur, n * 8, cudaMemcpyDeviceToHost, c->stream));
    if ((QL || QS) && n_steps > 0) {
        std::vector<double> q((size_t)n_steps * 2);
        FDIRW_CUDA(c, cudaMemcpyAsync(q.data(), k.qout, (size_t)n_steps * 16, cudaMemcpyDeviceToHost, c->stream));
        FDIRW_CUDA(c, cudaStreamSynchronize(c->stream));
        for (int t = 0; t < n_steps; t++) {
            if (QL) QL[t] = q[2 * t];
            if (QS) QS[t] = q[2 * t + 1];
        }
    }
    if (c_far) FDIRW_CUDA(c, cudaMemcpyAsync(c_far, k.far, 8, cudaMemcpyDeviceToHost, c->stream));
    if (c_far || kf == Kind::Host) FDIRW_CUDA(c, cudaStreamSynchronize(c->stream));
    return FDIRW_OK;
}

int fdirw_read_coarse(fdirw_ctx* c, const int64_t* blocks, int64_t n, double* out) {
    if (!c) return fail(nullptr, FDIRW_ERR_ARG, "NULL context");
    if (!c->coarse) return fail(c, FDIRW_ERR_ARG, "not a coarse-mesh context");
    if (n < 0 || (n > 0 && (!blocks || !out))) return fail(c, FDIRW_ERR_ARG, "bad blocks/out");
    fdirw::Coarse& k = *c->coarse;
    for (int64_t q = 0; q < n; q++)
        if (blocks[q] < 0 || blocks[q] >= k.nc) return fail(c, FDIRW_ERR_ARG, "block index out of range");
    if (!k.built) return fail(c, FDIRW_ERR_STATE, "coarse matrix not built (call fdirw_kernels)");
    if (n == 0) return FDIRW_OK;
    DeviceGuard dg(c->device);
    const int64_t W3 = (int64_t)(2 * k.Rc + 1) * (2 * k.Rc + 1) * (2 * k.Rc + 1);
    int64_t* db = nullptr;
    double* dout = nullptr;
    int rc = dalloc(c, reinterpret_cast<void**>(&db), (uint64_t)n * 8, "block list");
    if (rc != FDIRW_OK) return rc;
    rc = dalloc(c, reinterpret_cast<void**>(&dout), (uint64_t)(n * W3) * 8, "coarse readback");
    if (rc != FDIRW_OK) { drelease(db); c->allocated -= (uint64_t)n * 8; return rc; }
    cudaError_t e = cudaMemcpyAsync(db, blocks, (size_t)n * 8, cudaMemcpyHostToDevice, c->stream);
    if (e == cudaSuccess) {
        fdirw::read_coarse_kernel<<<fdirw::grid_blocks(n * W3, 256), 256, 0, c->stream>>>(k.Qc, k.ncx, k.ncy, k.ncz, k.Rc,
                                                                                         db, n, dout);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(out, dout, (size_t)(n * W3) * 8, cudaMemcpyDeviceToHost, c->stream);
    const cudaError_t w = cudaStreamSynchronize(c->stream);      // also after a failure: the blocks go to other contexts
    if (e == cudaSuccess) e = w;
    drelease(db);
    drelease(dout);
    c->allocated -= (uint64_t)n * 8 + (uint64_t)(n * W3) * 8;
    if (e != cudaSuccess) { cudaGetLastError(); return fail(c, FDIRW_ERR_CUDA, cuda_msg("read coarse matrix", e)); }
    return FDIRW_OK;
}

}  // extern "C"
