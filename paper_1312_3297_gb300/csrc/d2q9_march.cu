// D2Q9: three time steps per pass over memory (temporal blocking in the row direction).
//
// One step reads and writes every population once and runs at the copy bandwidth, so a run of
// n steps costs n times the state's traffic although only the first and the last state are
// wanted. k_march3 carries each row of a strip through three relaxations before it is stored:
// a warp marches up a strip of 32 packs (4 nodes each); when level 1 has relaxed row r, level
// 2 can relax row r - 1 and level 3 row r - 2, from the populations the level below left one
// and two rows ago (a delay line in shared memory) and just now (registers). The arithmetic of
// a node is that of the one-step kernels, in storage precision between the levels, so the
// states are theirs bit for bit.
//
// What bounds it: the FP32 pipe, 68 % busy at 4096^2 (ncu; 55 % of issue slots, DRAM at 5 TB/s).
// A packed multiply-add of three distinct register pairs takes it 3 cycles instead of 2 (24.7
// against 36.6 T lane operations/s measured), and 1.06 - 1.16 relaxations are done per stored
// one (lanes 0 and 31, the rows below a segment). Scalar multiply-adds in place of the packed
// ones, three warps per scheduler instead of four, and two or four levels were slower (FP32
// 4096^2: 150 k MLUPS with two levels, 203 k with four). Steps per pass are odd so that every
// state lands in the buffer in which as many single steps would leave it.
// Measured, MLUPS, u~ = q/rho, one step per launch -> here: FP32 3072^2 96 k -> 203 k, 2048^2
// 91 k -> 176 k; FP16 8192^2 184 k -> 216 k, 2048^2 166 k -> 172 k; BF16 8192^2 185 k -> 228 k.
#include <cuda_runtime.h>

#include <atomic>
#include <cmath>

#include "async_copy.cuh"
#include "d2q9.cuh"
#include "launch.h"
#include "occupancy.cuh"
#include "pdl.cuh"
#include "pull.cuh"

namespace lbmrv {
namespace {

constexpr int kLevels = kMarchSteps;
constexpr int kNV = 4;  // nodes per pack
// Packs of a strip that are stored: each level, the first too, leaves one wrong node more at
// both ends of a strip, whose neighbours belong to the next strips, so lanes 0 and 31 are
// recomputed there. The last level must still find a right node in them.
constexpr int kUse = 30;
static_assert(kLevels <= kNV, "wrong nodes would reach the lanes that are stored");
static_assert(kLevels % 2 == 1, "the state would land in the other buffer");

// A pack in storage form: NV consecutive nodes in W 32-bit words.
template <typename T>
constexpr int kW = kNV * (int)sizeof(T) / 4;

template <typename T>
__device__ __forceinline__ F2 get_pair(const uint32_t* w, int k) {
    if constexpr (sizeof(T) == 4) {
        return pack2(__uint_as_float(w[2 * k]), __uint_as_float(w[2 * k + 1]));
    } else {
        const float2 f = Cvt16<T>::unpack(w[k]);
        return pack2(f.x, f.y);
    }
}

template <typename T>
__device__ __forceinline__ void put_pair(uint32_t* w, int k, F2 v) {
    float a, b;
    unpack2(v, a, b);
    if constexpr (sizeof(T) == 4) {
        w[2 * k] = __float_as_uint(a);
        w[2 * k + 1] = __float_as_uint(b);
    } else {
        w[k] = Cvt16<T>::pack(a, b);
    }
}

// (prev, v0, ..., v_{NV-2}), prev from the left lane.
template <typename T>
__device__ __forceinline__ void from_left(uint32_t v[kW<T>], int left) {
    constexpr int W = kW<T>;
    const uint32_t p = __shfl_sync(kFullMask, v[W - 1], left);
#pragma unroll
    for (int i = W - 1; i >= 0; --i) {
        const uint32_t l = i ? v[i - 1] : p;
        v[i] = sizeof(T) == 4 ? l : __byte_perm(l, v[i], 0x5432);
    }
}
// (v1, ..., v_{NV-1}, next), next from the right lane.
template <typename T>
__device__ __forceinline__ void from_right(uint32_t v[kW<T>], int right) {
    constexpr int W = kW<T>;
    const uint32_t p = __shfl_sync(kFullMask, v[0], right);
#pragma unroll
    for (int i = 0; i < W; ++i) {
        const uint32_t r = i < W - 1 ? v[i + 1] : p;
        v[i] = sizeof(T) == 4 ? r : __byte_perm(v[i], r, 0x5432);
    }
}

template <typename T>
__device__ __forceinline__ void shift_x(uint32_t g[9][kW<T>], int left, int right) {
    from_left<T>(g[1], left);
    from_right<T>(g[3], right);
    from_left<T>(g[5], left);
    from_right<T>(g[6], right);
    from_right<T>(g[7], right);
    from_left<T>(g[8], left);
}

template <int W>
struct alignas(4 * W) Words {
    uint32_t w[W];
};
template <int W>
__device__ __forceinline__ void ldw(const void* p, uint32_t w[W]) {
    const Words<W> v = *reinterpret_cast<const Words<W>*>(p);
#pragma unroll
    for (int i = 0; i < W; ++i) w[i] = v.w[i];
}
template <int W>
__device__ __forceinline__ void stw(void* p, const uint32_t w[W]) {
    Words<W> v;
#pragma unroll
    for (int i = 0; i < W; ++i) v.w[i] = w[i];
    *reinterpret_cast<Words<W>*>(p) = v;
}

// The relaxation of one pack held in storage form, two nodes per packed FP32 instruction.
// amp: the prescribed field's factor; cx, cy: its base field on the pack (analytic: cx[0] for
// the whole row).
template <typename T, int UM, int BASIS, int RCP>
__device__ __forceinline__ void relax_pack(uint32_t g[9][kW<T>], float amp, const float* cx,
                                           const float* cy, const StepArgs& a) {
#pragma unroll
    for (int k = 0; k < kNV / 2; ++k) {
        F2 h[9];
#pragma unroll
        for (int j = 0; j < 9; ++j) h[j] = get_pair<T>(g[j], k);
        F2 ux(0.0f), uy(0.0f);
        if constexpr (UM == UM_ANALYTIC) {
            ux = F2(amp * cx[0]);
            uy = F2(amp) * pack2(cy[2 * k], cy[2 * k + 1]);
        } else if constexpr (UM == UM_FIELD) {
            ux = F2(amp) * pack2(cx[2 * k], cx[2 * k + 1]);
            uy = F2(amp) * pack2(cy[2 * k], cy[2 * k + 1]);
        }
        if constexpr (BASIS == 0)
            relax_node<UM, RCP>(h, ux, uy, a.s, a.ref);
        else
            relax_node_geier_r<UM, RCP>(h, ux, uy, a.s, a.ref);
#pragma unroll
        for (int j = 0; j < 9; ++j) put_pair<T>(g[j], k, h[j]);
    }
}

// Shared memory, private to each thread: the next row's nine packs, and nine packs of delay
// line per level but the last; a stored field adds its next row's two packs.
template <typename T, int WPB>
constexpr int kSlot = 32 * WPB * 4 * kW<T>;
template <typename T, int UM, int WPB>
constexpr int kSmem = kSlot<T, WPB> * 9 * kLevels + (UM == UM_FIELD ? 2 * 32 * WPB * 16 : 0);
// 16 warps per SM (128 registers, no spills); 12 with a stored field, whose rows of the three
// levels stay in registers.
template <int UM>
constexpr int kSmWarps = UM == UM_FIELD ? 12 : 16;

// Warps that an SM holds in blocks of `warps` warps: by its registers, and by its 228 KB of
// shared memory, of which every block takes 1 KB more than it asks for (FP32 blocks of one warp:
// 15). Sized for 16, the grid left a last wave, or, at half of it, blocks that did not fit beside
// those of the launch before (u~ = q/rho, us a step, sized for 16 -> 15: 600 x 4000 17.5 -> 15.1,
// 800 x 1000 10.9 -> 7.1, 64 x 9000 12.8 -> 7.4).
constexpr int kSmSmem = 228 * 1024, kSmemMost = 227 * 1024;
int sm_warps(int storage, int um, int warps) {
    const int slot = 32 * warps * kNV * (storage == kStoreF32 ? 4 : 2);
    const int smem = slot * 9 * kLevels + (um == UM_FIELD ? 2 * 32 * warps * 16 : 0);
    const int by_regs = (um == UM_FIELD ? kSmWarps<UM_FIELD> : kSmWarps<UM_ZERO>) / warps;
    const int by_smem = kSmSmem / (smem + 1024);
    return (by_regs < by_smem ? by_regs : by_smem) * warps;
}

// Strips of a row: one if the row has no more packs than a warp has lanes (its lanes are then
// each other's periodic neighbours and nothing is recomputed), else of kUse packs. Warps per
// block, on neighbouring strips of the same rows: two in FP32 unless that leaves a good part of
// them idle (4096^2 204 k MLUPS with two, 201 k with one), one in 16-bit storage (8192^2 227 k
// with one, 221 k with two).
struct Strips {
    int packs, warps, groups, segs;
    Strips(int storage, int um, int nx, int ny) {
        packs = nx / kNV;
        const int strips = packs <= 32 ? 1 : (packs + kUse - 1) / kUse;
        warps = storage == kStoreF32 && (strips % 2 == 0 || strips > 8) ? 2 : 1;
        groups = (strips + warps - 1) / warps;
        const int64_t resident_warps = (int64_t)sm_warps(storage, um, warps) * sm_count();
        // One segment of rows per resident block and strip group. Segments under 8 rows repeat
        // too many relaxations (2 (kLevels - 1) rows each): half as many then (FP32 1536 x 1000
        // 145 k MLUPS against 138 k). Long 16-bit segments are halved, so that blocks that end
        // early leave work to take (8192^2 227 k against 224 k; no gain in FP32).
        int64_t s = resident_warps / warps / groups;
        if (s * 8 > ny) s = resident_warps / 2 / warps / groups;
        if (storage != kStoreF32 && s * 64 < ny) s = 2 * s;
        if (s > ny) s = ny;
        segs = (int)(s < 1 ? 1 : s);
    }
};

template <typename T, int UM, int BASIS, int RCP, int WPB>
__global__ void __launch_bounds__(32 * WPB, kSmWarps<UM> / WPB)
    k_march3(const T* __restrict__ src, T* __restrict__ dst, StepArgs a, MarchAmps amps,
             int groups, int segs) {
    extern __shared__ __align__(16) char smem[];
    pdl_wait_prior();
    pdl_allow_next();
    constexpr int W = kW<T>, SB = kSlot<T, WPB>, NT = 32 * WPB;
    const int nx = a.nx, ny = a.ny;
    const int64_t n = (int64_t)nx * ny;
    const int lane = threadIdx.x & 31;
    const int grp = blockIdx.x % groups, seg = blockIdx.x / groups;
    const int packs = nx / kNV;
    int pk, left = lane - 1, right = lane + 1;  // this lane's pack, the neighbours' lanes
    bool act;
    if (packs <= 32) {
        pk = lane;
        act = lane < packs;
        if (lane == 0) left = packs - 1;
        if (lane == packs - 1) right = 0;
    } else {
        pk = (grp * WPB + (threadIdx.x >> 5)) * kUse + lane - 1;
        act = lane >= 1 && lane <= kUse && pk < packs;
    }
    int pw = pk % packs;  // lanes past the row's ends take its periodic continuation
    if (pw < 0) pw += packs;
    const int x0 = pw * kNV;
    const int y0 = (int)((int64_t)seg * ny / segs), y1 = (int)((int64_t)(seg + 1) * ny / segs);
    char* const mine = smem + threadIdx.x * (4 * W);
    char* const field = smem + 9 * kLevels * SB + threadIdx.x * 16;
    const T* const s0 = src + x0;
    auto load_row = [&](int64_t om, int64_t o0, int64_t op) {
        const int64_t row[3] = {om, o0, op};
        constexpr int dy[9] = {1, 1, 0, 1, 2, 0, 0, 2, 2};  // row[1 - c_y]
#pragma unroll
        for (int j = 0; j < 9; ++j) {
            if constexpr (W == 4)
                cp_async16(mine + j * SB, s0 + j * n + row[dy[j]]);
            else
                cp_async8(mine + j * SB, s0 + j * n + row[dy[j]]);
        }
        if constexpr (UM == UM_FIELD) {
            cp_async16(field, a.ut0 + o0 + x0);
            cp_async16(field + NT * 16, a.ut0 + n + o0 + x0);
        }
        cp_async_commit();
    };
    auto up = [&](int y) { return y == ny - 1 ? 0 : y + 1; };
    // u~0 on the rows of the three levels: the analytic field's cos 2 pi y/ny per row and sin
    // 2 pi x/nx per column, or a stored field's packs
    float bx[kLevels][UM == UM_FIELD ? kNV : 1], by[UM == UM_FIELD ? kLevels : 1][kNV];
    if constexpr (UM == UM_ANALYTIC) {
#pragma unroll
        for (int k = 0; k < kNV; ++k) by[0][k] = __ldg(a.sin_x + x0 + k);
    }
    // rows r - 1, r, r + 1 of the row that level 1 relaxes next
    int r = y0 - (kLevels - 1);
    while (r < 0) r += ny;
    int rm = r == 0 ? ny - 1 : r - 1, rp = up(r);
    int out = y0;
    const int rows = y1 - y0 + 2 * (kLevels - 1);
    load_row((int64_t)rm * nx, (int64_t)r * nx, (int64_t)rp * nx);
    for (int i = 0; i < rows; ++i) {
        const int rq = up(rp);
        cp_async_wait_all_but<0>();
        uint32_t g[9][W];
#pragma unroll
        for (int j = 0; j < 9; ++j) ldw<W>(mine + j * SB, g[j]);
        if constexpr (UM == UM_ANALYTIC) {
#pragma unroll
            for (int l = kLevels - 1; l > 0; --l) bx[l][0] = bx[l - 1][0];
            bx[0][0] = cospif(a.two_over_ny * (float)(r + a.y_off));
        } else if constexpr (UM == UM_FIELD) {
#pragma unroll
            for (int k = 0; k < kNV; ++k) {
#pragma unroll
                for (int l = kLevels - 1; l > 0; --l) {
                    bx[l][k] = bx[l - 1][k];
                    by[l][k] = by[l - 1][k];
                }
            }
            ldw<kNV>(field, reinterpret_cast<uint32_t*>(bx[0]));
            ldw<kNV>(field + NT * 16, reinterpret_cast<uint32_t*>(by[0]));
        }
        shift_x<T>(g, left, right);
        relax_pack<T, UM, BASIS, RCP>(g, amps.v[0], bx[0], by[0], a);
        // the slots have been read: fetch the next row behind levels 2 and 3
        if (i + 1 < rows) load_row((int64_t)r * nx, (int64_t)rp * nx, (int64_t)rq * nx);
#pragma unroll
        for (int l = 1; l < kLevels; ++l) {
            if (i < 2 * (l - 1)) continue;
            // the row below: {0,1,3} as level l left them one row ago, {2,5,6} two rows ago
            // (a ring of two), {4,7,8} now
            shift_x<T>(g, left, right);
            char* const d = mine + 9 * l * SB;
            char* const e = d + (3 + 3 * (i & 1)) * SB;
            constexpr int c0[3] = {0, 1, 3}, cp[3] = {2, 5, 6};
            uint32_t q[6][W];
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                ldw<W>(d + c * SB, q[c]);
                ldw<W>(e + c * SB, q[3 + c]);
            }
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                stw<W>(d + c * SB, g[c0[c]]);
                stw<W>(e + c * SB, g[cp[c]]);
            }
            if (i < 2 * l) continue;  // the delay line is not yet full
#pragma unroll
            for (int c = 0; c < 3; ++c) {
#pragma unroll
                for (int w = 0; w < W; ++w) {
                    g[c0[c]][w] = q[c][w];
                    g[cp[c]][w] = q[3 + c][w];
                }
            }
            relax_pack<T, UM, BASIS, RCP>(g, amps.v[l], bx[l], by[UM == UM_FIELD ? l : 0], a);
        }
        if (i >= 2 * (kLevels - 1)) {
            if (act) {
                T* const d = dst + (int64_t)out * nx + x0;
#pragma unroll
                for (int j = 0; j < 9; ++j) stw<W>(d + j * n, g[j]);
            }
            ++out;
        }
        rm = r;
        r = rp;
        rp = rq;
    }
}

template <typename T, int UM, int BASIS, int RCP, int WPB>
cudaError_t launch_w(const void* src, void* dst, const StepArgs& a, const MarchAmps& amps,
                     const Strips& p, cudaStream_t st, MarchStart start) {
    auto kernel = k_march3<T, UM, BASIS, RCP, WPB>;
    static std::atomic<int> resident[kMaxDevicesOcc];  // sets the kernel's shared memory, once
    int full = 0;
    cudaError_t e = resident_blocks(kernel, resident, 32 * WPB, kSmemMost, 32, &full);
    if (e != cudaSuccess) return e;
    // Blocks of a dependent launch start on whatever SM its predecessor has left, several on
    // one and none on another, and the launch after that fills the gaps they leave: with single
    // steps before them, the passes of a whole call ran up to 1.4 times longer. So of a few
    // passes each asks for as much shared memory as lets an SM hold its share of the blocks and
    // no more (BF16 816 x 2096, calls of 10 steps, us a step, 14.6 -> 10.9), and of many the first
    // starts alone, which spreads the blocks evenly, and the others follow freely (stored field,
    // FP32 1536 x 1000, 50 steps: 1.4 % faster than each with its share). Grids that fill the SMs
    // need neither (4096^2, calls of 24 steps, the first alone: 0.7 % slower).
    const int64_t blocks = (int64_t)p.groups * p.segs;
    const int64_t share = (blocks + sm_count() - 1) / sm_count();
    const bool fills =
        share * WPB >= sm_warps(sizeof(T) == 4 ? kStoreF32 : kStoreF16, UM, WPB);
    int smem = kSmem<T, UM, WPB>;
    if (start == MarchStart::kShare && !fills) {
        const int only = ((int)(kSmSmem / share) - 1024) / 128 * 128;  // allocated by 128 bytes
        if (smem < only) smem = only;
        if (smem > kSmemMost) smem = kSmemMost;
    }
    const T* const from = static_cast<const T*>(src);
    T* const to = static_cast<T*>(dst);
    const dim3 grid((unsigned)blocks);
    if (start == MarchStart::kAlone && !fills)
        kernel<<<grid, 32 * WPB, smem, st>>>(from, to, a, amps, p.groups, p.segs);
    else
        e = launch_pdl_smem(kernel, grid, dim3(32 * WPB), smem, st, from, to, a, amps, p.groups,
                            p.segs);
    return e != cudaSuccess ? e : cudaGetLastError();
}

template <typename T, int UM, int BASIS, int RCP>
cudaError_t launch_t(const void* src, void* dst, const StepArgs& a, const MarchAmps& amps,
                     cudaStream_t st, MarchStart start) {
    const Strips p(sizeof(T) == 4 ? kStoreF32 : kStoreF16, UM, a.nx, a.ny);
    if constexpr (sizeof(T) == 4) {
        if (p.warps == 2) return launch_w<T, UM, BASIS, RCP, 2>(src, dst, a, amps, p, st, start);
    }
    return launch_w<T, UM, BASIS, RCP, 1>(src, dst, a, amps, p, st, start);
}

// 1/rho in the form that the one-step kernel of the same rows uses (d2q9_kernels.cu), so that
// both give the same bits: FP32 the approximation (Geier's basis: correctly rounded); 16-bit
// rows of 8-node packs, and Geier's 4-node packs, the paired form; other 16-bit rows the
// correctly rounded one.
template <typename T, int BASIS, int UM>
cudaError_t launch_rcp(const void* s, void* d, const StepArgs& a, const MarchAmps& amps,
                       cudaStream_t st, MarchStart start) {
    if constexpr (sizeof(T) == 4) {
        return launch_t<T, UM, BASIS, BASIS == 0 ? RCP_APPROX : RCP_RN>(s, d, a, amps, st, start);
    } else if constexpr (UM == UM_ZERO) {
        return launch_t<T, UM, BASIS, RCP_RN>(s, d, a, amps, st, start);
    } else {
        if constexpr (BASIS == 0) {
            if (a.nx % 8 != 0) return launch_t<T, UM, BASIS, RCP_RN>(s, d, a, amps, st, start);
        }
        return launch_t<T, UM, BASIS, RCP_DIV>(s, d, a, amps, st, start);
    }
}

template <typename T, int BASIS>
cudaError_t launch_um(int um, const void* s, void* d, const StepArgs& a, const MarchAmps& amps,
                      cudaStream_t st, MarchStart start) {
    switch (um) {
        case UM_ZERO: return launch_rcp<T, BASIS, UM_ZERO>(s, d, a, amps, st, start);
        case UM_FLUID: return launch_rcp<T, BASIS, UM_FLUID>(s, d, a, amps, st, start);
        case UM_ANALYTIC: return launch_rcp<T, BASIS, UM_ANALYTIC>(s, d, a, amps, st, start);
        case UM_FIELD: return launch_rcp<T, BASIS, UM_FIELD>(s, d, a, amps, st, start);
        default: return cudaErrorInvalidValue;
    }
}

template <typename T>
cudaError_t launch_basis(int um, const void* s, void* d, const StepArgs& a,
                         const MarchAmps& amps, cudaStream_t st, int basis, MarchStart start) {
    return basis == 0 ? launch_um<T, 0>(um, s, d, a, amps, st, start)
                      : launch_um<T, 1>(um, s, d, a, amps, st, start);
}

}  // namespace

double march_step_us(int storage, int um, int basis, int nx, int ny, const void* a,
                     const void* b, const float* ut0) {
    const int bytes = storage == kStoreF32 ? 16 : 8;
    if (nx % kNV != 0 || reinterpret_cast<uintptr_t>(a) % bytes != 0 ||
        reinterpret_cast<uintptr_t>(b) % bytes != 0)
        return kNoForm;
    if (um == UM_FIELD && (reinterpret_cast<uintptr_t>(ut0) % 16 != 0 ||
                           (storage != kStoreF32 && basis == 1 && nx % 8 != 0)))
        return kNoForm;
    // Fitted as single_step_us is: a launch; the rows that a warp marches through, with a latency
    // of their own or, beside enough other warps, the SM's share; the memory beyond L2.
    const Strips p(storage, um, nx, ny);
    const bool f32 = storage == kStoreF32, field = um == UM_FIELD;
    const double rows = (ny + p.segs - 1) / p.segs + 2 * (kLevels - 1);
    const double warps = (double)p.groups * p.warps * p.segs / sm_count();  // per SM
    const int most = sm_warps(storage, um, p.warps);
    const double busy = std::ceil(warps < most ? warps : most);
    const double latency = f32 ? (field ? 0.954 : 0.786) : (field ? 0.917 : 0.953);
    const double share = (f32 ? (field ? 0.256 : 0.170) : (field ? 0.253 : 0.196)) * busy;
    constexpr double modes[2][2][4] = {{{1.0, 1.21, 1.22, 1.0}, {1.28, 1.46, 1.52, 1.24}},
                                       {{1.0, 0.97, 1.0, 1.0}, {1.04, 0.98, 1.01, 1.01}}};
    const double l2 = latency * latency, s2 = share * share;
    double row = modes[!f32][basis][um] * std::sqrt(std::sqrt(l2 * l2 + s2 * s2));
    if (!f32 && basis == 0 && um != UM_ZERO && nx % 8 != 0) row *= 1.24;  // 1/rho correctly rounded
    const double us = 1.2 + rows * row * (warps > most ? warps / most : 1.0) +
                      (field ? 0.0 : f32 ? 1.12 : 2.2) * 1e-6 * ((double)nx * ny) *
                          beyond_l2(storage, um, nx, ny, 40e6, 130e6);
    return us / kLevels * (beyond_l2(storage, um, nx, ny, 125e6, 125e6) > 0.0 ? 0.9 : 1.0);
}

cudaError_t launch_march(int storage, int um, const void* src, void* dst, const StepArgs& a,
                         const MarchAmps& amps, cudaStream_t st, int basis, MarchStart start) {
    switch (storage) {
        case kStoreF32: return launch_basis<float>(um, src, dst, a, amps, st, basis, start);
        case kStoreF16: return launch_basis<__half>(um, src, dst, a, amps, st, basis, start);
        case kStoreBF16:
            return launch_basis<__nv_bfloat16>(um, src, dst, a, amps, st, basis, start);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace lbmrv
