// The tile kernel's plan and its FP32 instances (d2q9_tile.cuh).
#include "d2q9_tile.cuh"

namespace lbmrv {

namespace {

// Times in microseconds measured on GB300, for the choice of a plan only (any plan gives the
// same states).
constexpr double kLaunch = 2.1;      // a pass: launch, first loads, last stores
constexpr double kStepFloor = 0.46;  // a step of a block that fills no pipe
constexpr double kItem = 0.0545;     // a warp's two rows of 32 nodes on a busy SM, per SM
constexpr double kSerial = 2.0;      // loads and stores of a tile that nothing else overlaps

bool fits_l2(double nodes, int node_bytes) { return 2.0 * node_bytes * nodes < 128e6; }

// the correctly rounded 1/rho of 16-bit storage, and the conversions, take a little longer
double tile_item_us(int elem, int um, int nv) {
    return kItem * (elem == 2 && um != UM_ZERO ? (nv == 8 ? 1.03 : 1.1) : 1.0);
}

}  // namespace

int sm_count() {
    static std::atomic<int> sms_of[kMaxDevicesOcc];
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev >= kMaxDevicesOcc) return 152;
    sms = sms_of[dev].load(std::memory_order_relaxed);
    if (sms == 0) {
        if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
            sms < 1)
            return 152;
        sms_of[dev].store(sms, std::memory_order_relaxed);
    }
    return sms;
}

// The launch, and the time per million nodes at the pack width nv: with the states in L2, too
// large for it, or between; more where a row leaves many of a block's 128 threads without a
// pack.
double single_step_us(int storage, int um, int nv, int nx, int ny) {
    const double nodes = (double)nx * ny;
    const bool f32 = storage == kStoreF32;
    const double field = um == UM_FIELD ? 8.0 : 0.0;
    const double both = (2.0 * 9.0 * (f32 ? 4 : 2) + field) * nodes;
    const bool l2 = both < 78e6, dram = both > 128e6;
    double per_m;
    if (f32)
        per_m = nv == 4 ? (l2 ? 6.4 : dram ? 10.5 : 7.8)
              : nv == 2 ? (dram ? 10.9 : 8.2)
                        : (dram ? 11.2 : 7.7);
    else
        per_m = nv == 8 ? (dram ? 5.8 : 4.4) : nv == 4 ? 5.4 : nv == 2 ? 7.7 : 9.5;
    if (nv >= 4) {
        const int span = 128 * nv;
        const double used = (double)nx / (span * ((nx + span - 1) / span));
        if (f32)
            per_m *= used < 0.1 ? 0.3 / used : 1.0 + 0.2 * (1.0 - used);
        else
            per_m *= used < 0.4 ? 0.5 / used : 1.0 + 0.8 * (1.0 - used);
    }
    if (um == UM_ZERO && !f32 && !dram) per_m *= 0.87;
    if (um == UM_FIELD) per_m *= !dram || f32 ? 1.07 : 1.22;
    return 1.9 + per_m * 1e-6 * nodes;
}

namespace {

// The array and warps per block that take a launch of s steps in the least modelled time
// (steps = 1 if that is `least` or more).
TilePlan tile_pass(int storage, int um, int nv, int nx, int ny, int s, double least) {
    TilePlan best;
    best.us = least;
    const int elem = storage == kStoreF32 ? 4 : 2, sms = sm_count();
    const bool in_l2 = fits_l2((double)nx * ny, 9 * elem);
    const double item_us = tile_item_us(elem, um, nv);
    const double per_sm = item_us / sms;
    // the first step's loads: latency that few later steps leave exposed
    const double first = (s == 2 ? (in_l2 ? 1.5 : 2.0) : s == 3 ? 1.2 : 1.0) +
                         (um == UM_FIELD ? 0.8 : 0.0);
    constexpr int heights[] = {12, 16, 20, 22, 24, 26, 28, 32, 36, 38, 40, 44, 46, 48, 56, 62};
    for (int rx = 32; rx <= 64; rx += 32) {
        const int tx = rx - 2 * (s - 1);
        if (tx < 4) continue;
        const int tiles_x = (nx + tx - 1) / tx;
        for (int ry : heights) {
            const int ty = ry - 2 * (s - 1);
            if (ty < 4) continue;
            const int bytes = (int)tile_bytes(rx, ry, elem, um);
            if (bytes > kTileMaxSmem || ty > ny + 8) break;
            const int tiles = tiles_x * ((ny + ty - 1) / ty);
            // the pipes' share, were the tiles spread evenly: usually enough to drop it
            const double even = per_sm * s * (rx / 32) * ((ry + ty) / 4) * tiles;
            const double steps_alone = kStepFloor * s;
            if (kLaunch + (even > steps_alone ? even : steps_alone) >= best.us) continue;
            const int items = rx / 32 * (ry / 2);
            const int rounds = (items + kTileWarps - 1) / kTileWarps;
            const int whole = (items + rounds - 1) / rounds;
            // one block per SM with a warp for every item, or several with half as many
            for (int half = 1; half <= 2; ++half) {
                int warps = (whole + half - 1) / half;
                warps = (warps + rx / 32 - 1) / (rx / 32) * (rx / 32);
                int fit = (227 * 1024) / (bytes + 1024);
                if (fit > kTileWarps / warps) fit = kTileWarps / warps;
                if (fit < 1) continue;
                // `resident` tiles at a time on an SM
                auto wave = [&](int resident) {
                    const double busy = (double)resident * warps;
                    const double item =
                        item_us * (busy < 20.0 ? 1.0 + 0.03 * (20.0 - busy) : 1.0);
                    double us = 0.0;
                    for (int k = 0; k < s; ++k) {
                        const int pairs = rx / 32 * ((ry - k - 1) / 2 - k / 2 + 1);
                        const double pipes = (k ? 1.0 : first) * item * pairs * resident;
                        const double alone =
                            pairs <= warps ? kStepFloor
                                           : kStepFloor * ((pairs + warps - 1) / warps);
                        us += pipes > alone ? pipes : alone;
                    }
                    return us;
                };
                const int full = tiles / (sms * fit), rest = tiles - full * sms * fit;
                double us = full * wave(fit) + (rest ? wave((rest + sms - 1) / sms) : 0.0);
                if (fit == 1 && tiles > sms) us += kSerial * (tiles - sms) / sms;
                if (kLaunch + us < best.us) {
                    best.us = kLaunch + us;
                    best.steps = s;
                    best.rx = rx;
                    best.ry = ry;
                    best.warps = warps;
                    best.per_sm =
                        full == 0 || (rest == 0 && full == 1) ? (tiles + sms - 1) / sms : 0;
                }
            }
        }
    }
    return best;
}

}  // namespace

// The plan with the least modelled time for n steps: steps per pass, array size and warps per
// block. Small lattices take many steps per pass (64^2: 10, over 32 x 22 arrays), since a launch
// costs as much as four steps; larger ones the array whose tiles just fill the SMs (512^2: 4 over
// 64 x 38). Aligned rows of larger L2-resident lattices stay with single steps, which the
// repeated relaxations of the halos would not beat (FP32 1024^2 8.5 us a step against 9.4,
// 16-bit 768^2 5.0 against 5.6); there is no such limit for rows without vector packs.
// Measured, single steps -> here, us a step (u~ = q/rho): FP32 64^2 2.05 -> 0.82, 256^2 2.3 ->
// 1.22, 512^2 3.9 -> 2.73, 1023^2 10.1 -> 8.3, 4097 x 1999 94 -> 60; FP16 64^2 2.1 -> 0.87,
// 512^2 3.0 -> 2.9, 513 x 511 4.5 -> 2.9, 4097 x 1999 82 -> 60.
TilePlan tile_plan(TileTable& table, int storage, int um, int nv, int nx, int ny, int64_t n,
                   double least) {
    TilePlan best;
    best.us = least;
    // What a launch of s steps takes at least: the launch, and each step's latency or the pipes'
    // share of the lattice.
    const double share = tile_item_us(storage == kStoreF32 ? 4 : 2, um, nv) * (double)nx * ny /
                         (64.0 * sm_count());
    const double step = share > kStepFloor ? share : kStepFloor;
    // likely lengths first: a good plan early drops most of the others unsearched
    constexpr int lengths[] = {5, 10, 4, 3, 8, 6, 12, 2};
    for (int want : lengths) {
        // an odd number of passes for an odd number of steps, an even one for an even number:
        // the state ends in the buffer in which single steps would leave it
        int64_t m = (n + want - 1) / want;
        m += (m ^ n) & 1;
        const int s = (int)((n + m - 1) / m);
        if (s < 2 || m * (kLaunch + step * s) >= best.us) continue;
        TilePlan& pass = table.best[s];
        const double least = best.us / m;
        if (pass.steps == 1 && pass.us < least)
            pass = tile_pass(storage, um, nv, nx, ny, s, least);
        if (pass.steps > 1 && pass.us < least) {
            best = pass;
            best.us = m * pass.us;
            best.launches = m;
        }
    }
    return best;
}

cudaError_t launch_tile(int storage, int um, int basis, int nv, const void* src, void* dst,
                        const StepArgs& a, const TileAmps& amps, const TilePlan& p,
                        cudaStream_t st) {
    if (storage == kStoreF32) return tile_basis<float>(um, basis, nv, src, dst, a, amps, p, st);
    return launch_tile16(storage, um, basis, nv, src, dst, a, amps, p, st);
}

}  // namespace lbmrv
