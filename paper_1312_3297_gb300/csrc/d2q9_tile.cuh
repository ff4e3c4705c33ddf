// D2Q9: several time steps per launch on a tile held in shared memory, for lattices whose
// states stay in L2 and for rows that no vector pack divides.
//
// What bounds it: on small lattices a launch (2.1 us) and the latency of a step (0.46 us: shared
// loads, a chain of some 40 dependent FP32 instructions, a barrier); on larger ones the FP32
// pipe and the issue slots (a warp's two rows of 32 nodes take 54 ns of an SM, 48 % of issue
// slots busy at 1024^2). Two nodes per thread in one column, because neighbouring lanes then
// read and write neighbouring words whatever the row's alignment.
#pragma once

#include <cuda_runtime.h>

#include <atomic>

#include "d2q9.cuh"
#include "launch.h"
#include "occupancy.cuh"
#include "pdl.cuh"
#include "pull.cuh"

namespace lbmrv {
namespace {

constexpr int kTileThreads = 32 * kTileWarps;  // most per block (80 registers, no spills)

// Which relaxation the one-step kernel of the same rows uses, so that both give the same bits:
// node pairs with one of the forms of 1/rho (FORM_ROW added: relax_node's ROW), or Geier's
// basis node by node.
enum { FORM_NODES = 3, FORM_ROW = 4 };  // else RCP_*: pairs

template <typename T, int UM, int BASIS, int FORM>
__device__ __forceinline__ void relax_two(float p[9], float q[9], float ux0, float uy0, float ux1,
                                          float uy1, const StepArgs& a) {
    if constexpr (FORM == FORM_NODES) {
        if constexpr (UM == UM_FLUID) {
            relative_velocity<UM_FLUID>(p, a.ref, 0, 0, 0, a, ux0, uy0);
            relative_velocity<UM_FLUID>(q, a.ref, 0, 0, 0, a, ux1, uy1);
        }
        relax_node_geier(p, ux0, uy0, a.s, a.ref);
        relax_node_geier(q, ux1, uy1, a.s, a.ref);
    } else {
        F2 h[9];
#pragma unroll
        for (int j = 0; j < 9; ++j) h[j] = pack2(p[j], q[j]);
        F2 ux = pack2(ux0, ux1), uy = pack2(uy0, uy1);
        if constexpr (BASIS == 0)
            relax_node<UM, FORM & 3, (FORM & FORM_ROW) != 0>(h, ux, uy, a.s, a.ref);
        else
            relax_node_geier_r<UM, FORM & 3>(h, ux, uy, a.s, a.ref);
#pragma unroll
        for (int j = 0; j < 9; ++j) unpack2(h[j], p[j], q[j]);
    }
}

__device__ __forceinline__ int wrap(int v, int n) {
    v %= n;
    return v < 0 ? v + n : v;
}

// One block: `steps` steps of a tile of (RX - 2 h) x (ry - 2 h) nodes, h = steps - 1. Step s
// relaxes the tile and steps - s nodes around it (what the later steps pull from); step 1
// pulls from src, the last step stores to dst. In between the populations stay in one shared
// array of RX x ry nodes, which every node reads and writes in the same places: odd steps read
// population j at slot j of the node and leave the result in slot opp(j) of the node; even
// steps read population j from slot opp(j) of node x - c_j and leave the result in slot j of
// node x + c_j. So one barrier per step is enough and no second array is needed. (The "AA" access
// pattern of P. Bailey et al., Accelerating lattice Boltzmann fluid flow simulations using
// graphics processors, ICPP 2009, here within a block.)
// A thread has one column and relaxes two nodes, (x, y) and (x, y + 1), at a time. Rows of
// the array are RX values per population, populations side by side, so that every shared
// address is one register plus a constant. Rows -1, ry and ry + 1 of the array are only read for
// nodes that are not kept; then comes the prescribed field (the analytic one's cos per row, or
// a stored one's two components per node).
template <typename T, int UM, int BASIS, int FORM, int RX>
__global__ void __launch_bounds__(kTileThreads, 1)
    k_tile(const T* __restrict__ src, T* __restrict__ dst, StepArgs a, TileAmps amps, int steps,
           int ry, int tiles_x) {
    extern __shared__ __align__(16) char smem[];
    constexpr int kRowWarps = RX / 32;
    constexpr int opp[9] = {0, 3, 4, 1, 2, 7, 8, 5, 6};
    constexpr int cx[9] = {0, 1, 0, -1, 0, 1, -1, -1, 1};
    constexpr int cy[9] = {0, 0, 1, 0, -1, 1, 1, -1, -1};
    const int nx = a.nx, ny = a.ny;
    const int64_t n = (int64_t)nx * ny;
    const int groups = (int)blockDim.x / RX;
    const int halo = steps - 1;
    const int ox = (blockIdx.x % tiles_x) * (RX - 2 * halo) - halo;  // array origin
    const int oy = (blockIdx.x / tiles_x) * (ry - 2 * halo) - halo;
    const int warp = threadIdx.x >> 5;
    const int x = (warp % kRowWarps) * 32 + (threadIdx.x & 31), grp = warp / kRowWarps;
    T* const f = reinterpret_cast<T*>(smem) + 9 * RX + x;  // row 0 of this column
    float* const field = reinterpret_cast<float*>(smem + 9LL * RX * (ry + 3) * sizeof(T));
    const int gx = wrap(ox + x, nx);
    const int xs[3] = {gx == nx - 1 ? 0 : gx + 1, gx, gx == 0 ? nx - 1 : gx - 1};
    float sx = 0.0f;
    if constexpr (UM == UM_ANALYTIC) {  // the handle's own constant table: no need to wait for it
        sx = __ldg(a.sin_x + gx);
        for (int i = threadIdx.x; i <= ry; i += (int)blockDim.x)
            field[i] = cospif(a.two_over_ny * (float)(wrap(oy + i, ny) + a.y_off));
        __syncthreads();
    }
    pdl_wait_prior();
    pdl_allow_next();
    if constexpr (UM == UM_FIELD) {  // a thread reads back what it writes
        for (int r = grp; 2 * r < ry; r += groups) {
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                const int64_t at = (int64_t)wrap(oy + 2 * r + k, ny) * nx + gx;
                field[(2 * r + k) * RX + x] = __ldg(a.ut0 + at);
                field[(ry + 1 + 2 * r + k) * RX + x] = __ldg(a.ut0 + n + at);
            }
        }
    }
    for (int s = 1; s <= steps; ++s) {
        const bool in_x = x >= s - 1 && x <= RX - s;
        const float amp = amps.v[s - 1];
        for (int r = grp; 2 * r < ry; r += groups) {
            const int y = 2 * r;
            const bool k0 = in_x && y >= s - 1 && y <= ry - s;  // the nodes to keep
            const bool k1 = in_x && y + 1 >= s - 1 && y + 1 <= ry - s;
            if (!(k0 || k1)) continue;
            T* const c = f + y * 9 * RX;
            float p[9], q[9];
            if (s == 1) {
                const int g1 = wrap(oy + y, ny);
                const int g0 = g1 == 0 ? ny - 1 : g1 - 1;
                const int g2 = g1 == ny - 1 ? 0 : g1 + 1;
                const int g3 = g2 == ny - 1 ? 0 : g2 + 1;
                const int row[4] = {g0 * nx, g1 * nx, g2 * nx, g3 * nx};
#pragma unroll
                for (int j = 0; j < 9; ++j) {
                    const T* const sj = src + j * n;
                    p[j] = to_f(sj[row[1 - cy[j]] + xs[1 + cx[j]]]);
                    q[j] = to_f(sj[row[2 - cy[j]] + xs[1 + cx[j]]]);
                }
            } else if (s & 1) {
#pragma unroll
                for (int j = 0; j < 9; ++j) {
                    p[j] = to_f(c[j * RX]);
                    q[j] = to_f(c[(9 + j) * RX]);
                }
            } else {
#pragma unroll
                for (int j = 0; j < 9; ++j) {
                    p[j] = to_f(c[(opp[j] - 9 * cy[j]) * RX - cx[j]]);
                    q[j] = to_f(c[(9 + opp[j] - 9 * cy[j]) * RX - cx[j]]);
                }
            }
            float ux0 = 0.0f, uy0 = 0.0f, ux1 = 0.0f, uy1 = 0.0f;
            if constexpr (UM == UM_ANALYTIC) {
                ux0 = amp * field[y];
                ux1 = amp * field[y + 1];
                uy0 = uy1 = amp * sx;
            } else if constexpr (UM == UM_FIELD) {
                ux0 = amp * field[y * RX + x];
                ux1 = amp * field[(y + 1) * RX + x];
                uy0 = amp * field[(ry + 1 + y) * RX + x];
                uy1 = amp * field[(ry + 2 + y) * RX + x];
            }
            relax_two<T, UM, BASIS, FORM>(p, q, ux0, uy0, ux1, uy1, a);
            if (s == steps) {
                const int X = ox + x, Y = oy + y;
                if (X < nx) {
                    T* const d = dst + (int64_t)Y * nx + X;
                    if (k0 && Y < ny) {
#pragma unroll
                        for (int j = 0; j < 9; ++j) d[j * n] = from_f<T>(p[j]);
                    }
                    if (k1 && Y + 1 < ny) {
#pragma unroll
                        for (int j = 0; j < 9; ++j) d[j * n + nx] = from_f<T>(q[j]);
                    }
                }
            } else if (s & 1) {
                if (k0) {
#pragma unroll
                    for (int j = 0; j < 9; ++j) c[opp[j] * RX] = from_f<T>(p[j]);
                }
                if (k1) {
#pragma unroll
                    for (int j = 0; j < 9; ++j) c[(9 + opp[j]) * RX] = from_f<T>(q[j]);
                }
            } else {
                if (k0) {
#pragma unroll
                    for (int j = 0; j < 9; ++j) c[(j + 9 * cy[j]) * RX + cx[j]] = from_f<T>(p[j]);
                }
                if (k1) {
#pragma unroll
                    for (int j = 0; j < 9; ++j)
                        c[(9 + j + 9 * cy[j]) * RX + cx[j]] = from_f<T>(q[j]);
                }
            }
        }
        if (s < steps) __syncthreads();
    }
}

template <typename T, int UM, int BASIS, int FORM, int RX>
cudaError_t tile_launch_rx(const void* src, void* dst, const StepArgs& a, const TileAmps& amps,
                           const TilePlan& p, cudaStream_t st) {
    auto kernel = k_tile<T, UM, BASIS, FORM, RX>;
    // sets the shared memory of the largest tile of any plan, once per device
    static std::atomic<int> resident[kMaxDevicesOcc];
    int full = 0;
    cudaError_t e = resident_blocks(kernel, resident, 32, kTileMaxSmem, 32, &full);
    if (e != cudaSuccess) return e;
    const int tx = RX - 2 * (p.steps - 1), ty = p.ry - 2 * (p.steps - 1);
    const int tiles_x = (a.nx + tx - 1) / tx, tiles_y = (a.ny + ty - 1) / ty;
    // Blocks of a dependent launch start on whatever SM its predecessor has left, several on
    // one and none on another. Where one wave is planned, ask for so much shared memory that no
    // more than the planned number fit (FP16 700^2, 286 blocks: 6.9 -> 5.0 us a step).
    int64_t smem = tile_bytes(RX, p.ry, (int)sizeof(T), UM);
    const int64_t alone = p.per_sm > 0 ? 228 * 1024 / (p.per_sm + 1) : 0;
    if (smem < alone) smem = alone;
    e = launch_pdl_smem(kernel, dim3((unsigned)((int64_t)tiles_x * tiles_y)),
                        dim3((unsigned)(32 * p.warps)), (size_t)smem, st,
                        static_cast<const T*>(src), static_cast<T*>(dst), a, amps, p.steps, p.ry,
                        tiles_x);
    return e != cudaSuccess ? e : cudaGetLastError();
}

template <typename T, int UM, int BASIS, int FORM>
cudaError_t tile_launch(const void* src, void* dst, const StepArgs& a, const TileAmps& amps,
                        const TilePlan& p, cudaStream_t st) {
    return p.rx == 32 ? tile_launch_rx<T, UM, BASIS, FORM, 32>(src, dst, a, amps, p, st)
                      : tile_launch_rx<T, UM, BASIS, FORM, 64>(src, dst, a, amps, p, st);
}

// nv: the pack width of the one-step kernel for these rows, which decides its relaxation.
template <typename T, int UM, int BASIS>
cudaError_t tile_form(int nv, const void* s, void* d, const StepArgs& a, const TileAmps& amps,
                      const TilePlan& p, cudaStream_t st) {
    if constexpr (BASIS == 1) {
        if constexpr (sizeof(T) == 4) {
            return tile_launch<T, UM, BASIS, RCP_RN>(s, d, a, amps, p, st);
        } else {
            if (nv == 8 || (nv == 4 && UM != UM_FIELD))
                return tile_launch<T, UM, BASIS, UM == UM_ZERO ? RCP_RN : RCP_DIV>(s, d, a, amps,
                                                                                   p, st);
            return tile_launch<T, UM, BASIS, FORM_NODES>(s, d, a, amps, p, st);
        }
    } else {
        constexpr int rcp = sizeof(T) == 4 ? RCP_APPROX : RCP_RN;
        constexpr int row = UM == UM_ANALYTIC ? FORM_ROW : 0;
        if constexpr (sizeof(T) == 2 && UM != UM_ZERO) {
            if (nv == 8) return tile_launch<T, UM, BASIS, RCP_DIV | row>(s, d, a, amps, p, st);
        }
        if (nv > 1) return tile_launch<T, UM, BASIS, rcp | row>(s, d, a, amps, p, st);
        return tile_launch<T, UM, BASIS, rcp>(s, d, a, amps, p, st);
    }
}

template <typename T, int BASIS>
cudaError_t tile_um(int um, int nv, const void* s, void* d, const StepArgs& a,
                    const TileAmps& amps, const TilePlan& p, cudaStream_t st) {
    switch (um) {
        case UM_ZERO: return tile_form<T, UM_ZERO, BASIS>(nv, s, d, a, amps, p, st);
        case UM_FLUID: return tile_form<T, UM_FLUID, BASIS>(nv, s, d, a, amps, p, st);
        case UM_ANALYTIC: return tile_form<T, UM_ANALYTIC, BASIS>(nv, s, d, a, amps, p, st);
        case UM_FIELD: return tile_form<T, UM_FIELD, BASIS>(nv, s, d, a, amps, p, st);
        default: return cudaErrorInvalidValue;
    }
}

template <typename T>
cudaError_t tile_basis(int um, int basis, int nv, const void* s, void* d, const StepArgs& a,
                       const TileAmps& amps, const TilePlan& p, cudaStream_t st) {
    return basis == 0 ? tile_um<T, 0>(um, nv, s, d, a, amps, p, st)
                      : tile_um<T, 1>(um, nv, s, d, a, amps, p, st);
}

}  // namespace
}  // namespace lbmrv
