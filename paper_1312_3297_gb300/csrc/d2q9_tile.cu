// The tile kernel's plan and its FP32 instances (d2q9_tile.cuh).
#include "d2q9_tile.cuh"

namespace lbmrv {

namespace {

// The models below choose between forms and plans only (any choice gives the same states). Their
// numbers are fitted to single steps, three-step passes and tile launches of 10,500 random
// lattices of 8 - 4300 nodes a side, all storages, modes and bases, timed on GB300 (microseconds);
// each predicts these to 7 % (standard deviation).
constexpr double kStepFloor = 0.46;  // a step of a block that fills no pipe
constexpr double kItem = 0.0545;     // a warp's two rows of 32 nodes on a busy SM, per SM
constexpr double kSerial = 2.0;      // loads and stores of a tile that nothing else overlaps

bool fits_l2(double nodes, int node_bytes) { return 2.0 * node_bytes * nodes < 128e6; }

// A pass's fixed part and, relative to the numbers above, its steps: by storage, basis and mode,
// and by the relaxation that the pack width decides (node by node, or with the correctly rounded
// 1/rho).
struct TileCost {
    double launch, scale;
    TileCost(int storage, int um, int basis, int nv) {
        constexpr double fixed[4] = {1.85, 1.8, 2.1, 2.35};
        constexpr double steps[2][2][4] = {{{0.86, 1.04, 1.15, 1.05}, {1.00, 1.16, 1.24, 1.13}},
                                           {{0.97, 1.11, 1.23, 1.09}, {1.03, 1.12, 1.21, 1.10}}};
        const bool half = storage != kStoreF32;
        launch = fixed[um];
        scale = steps[half][basis][um];
        if (half && basis == 1 && (nv <= 2 || (nv == 4 && um == UM_FIELD))) {
            launch += 0.2;
            scale *= 1.12;
        } else if (half && basis == 0 && um != UM_ZERO && nv < 8) {
            scale *= 1.02;
        }
    }
};

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

// A launch; its blocks, warps and nodes (in L2, and beyond it); and, for blocks between half and
// all of those resident at once, the blocks of the next launch, which start early, leaving some
// SMs with more of them than others (FP32 1016 x 352, 704 blocks: 6.8 us where 528 take 3).
double single_step_us(int storage, int um, int basis, int nv, int nx, int ny) {
    struct Row {
        double launch, block, warp, l2, dram, pile;
        double mode[8];  // u~ = 0, 0 in Geier's basis, q/rho, ...
    };
    constexpr Row f32[3] = {
        {1.52, 0.34, 0.07, 3.74, 7.25, 1.23, {1.0, 1.07, 1.11, 1.17, 1.28, 1.27, 1.27, 1.26}},
        {1.82, 0.60, 0.21, 1.05, 5.39, 1.96, {1.0, 0.92, 1.27, 1.08, 0.99, 1.13, 1.23, 1.14}},
        {1.94, 0.63, 0.24, 2.17, 6.77, 2.75, {1.0, 1.11, 1.16, 1.20, 1.19, 1.32, 1.21, 1.28}}};
    constexpr Row half[4] = {
        {1.53, 0.22, 0.12, 2.75, 3.91, 1.01, {1.0, 1.23, 1.25, 1.32, 1.44, 1.41, 1.34, 1.38}},
        {1.69, 0.60, 0.17, 1.01, 1.93, 1.73, {1.0, 1.07, 1.18, 1.17, 1.25, 1.26, 1.24, 1.25}},
        {1.93, 0.63, 0.30, 0.57, 2.16, 0.89, {1.0, 1.02, 1.22, 1.19, 1.31, 1.27, 1.42, 1.38}},
        {2.16, 1.22, 0.56, 0.72, 2.15, 0.93, {1.0, 1.03, 1.04, 1.09, 1.08, 1.20, 1.23, 1.29}}};
    const bool is_f32 = storage == kStoreF32;
    const int i = nv == 8 ? 3 : nv == 4 ? 2 : nv - 1;
    const Row& c = is_f32 ? f32[i] : half[i];
    const int threads = nv == 1 ? 256 : 128, packs = nx / nv;
    const double blocks = (double)((packs + threads - 1) / threads) * ny;
    const double warps = (double)((packs + 31) / 32) * ny;
    // blocks per SM, by the kernels' registers
    int per_sm;
    if (nv == 1)
        per_sm = 6;
    else if (nv == 2)
        per_sm = 8;
    else if (nv == 8)
        per_sm = basis ? (um == UM_FIELD ? 4 : 5) : um <= UM_FLUID ? 4 : 3;
    else if (is_f32)
        per_sm = um <= UM_FLUID ? 7 : 6;
    else
        per_sm = basis == 1 && um != UM_FIELD ? 8 : 6;
    const double share = blocks / (per_sm * sm_count());
    double pile = 1.0;
    if (share > 0.56 && share < 1.0) {
        const double busy = (warps / blocks - 1.0) / (threads / 32 - 1);  // warps of a block
        pile += c.pile * (1.0 - share) * (busy < 1.0 ? busy : 1.0);
    }
    const double m = (double)nx * ny * 1e-6, far = beyond_l2(storage, um, nx, ny, 78e6, 135e6);
    return c.launch + pile * (c.mode[2 * um + basis] * (c.block * blocks * 1e-3 +
                                                        c.warp * warps * 1e-3 +
                                                        c.l2 * m * (1.0 - far)) +
                              c.dram * m * far);
}

// 0 if both states and a stored field take less than lo bytes, 1 if more than hi.
double beyond_l2(int storage, int um, int nx, int ny, double lo, double hi) {
    const double bytes = ((storage == kStoreF32 ? 72.0 : 36.0) + (um == UM_FIELD ? 8.0 : 0.0)) *
                         ((double)nx * ny);
    return bytes <= lo ? 0.0 : bytes >= hi ? 1.0 : (bytes - lo) / (hi - lo);
}

namespace {

// The array and warps per block that take a launch of s steps in the least modelled time
// (steps = 1 if that is `least` or more).
TilePlan tile_pass(int storage, int um, int basis, int nv, int nx, int ny, int s,
                   double least) {
    TilePlan best;
    best.us = least;
    const int elem = storage == kStoreF32 ? 4 : 2, sms = sm_count();
    const bool in_l2 = fits_l2((double)nx * ny, 9 * elem);
    const TileCost cost(storage, um, basis, nv);
    const double item_us = kItem * cost.scale, floor_us = kStepFloor * cost.scale;
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
            const double steps_alone = floor_us * s;
            if (cost.launch + (even > steps_alone ? even : steps_alone) >= best.us) continue;
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
                            pairs <= warps ? floor_us : floor_us * ((pairs + warps - 1) / warps);
                        us += pipes > alone ? pipes : alone;
                    }
                    return us;
                };
                const int full = tiles / (sms * fit), rest = tiles - full * sms * fit;
                double us = full * wave(fit) + (rest ? wave((rest + sms - 1) / sms) : 0.0);
                if (fit == 1 && tiles > sms) us += kSerial * cost.scale * (tiles - sms) / sms;
                if (cost.launch + us < best.us) {
                    best.us = cost.launch + us;
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
// repeated relaxations of the halos do not beat (FP32 1024^2 8.5 us a step against 8.3, 16-bit
// 768^2 4.9 against 5.3, 1024^2 6.4 against 8.9); there is no such limit for rows without vector
// packs. Measured, single steps -> here, us a step (u~ = q/rho, calls of 24 steps): FP32 64^2
// 2.07 -> 0.81, 256^2 2.3 -> 1.24, 512^2 3.5 -> 2.68, 1023^2 10.0 -> 8.3, 4097 x 1999 93 -> 64;
// FP16 64^2 2.1 -> 0.87, 512^2 3.0 -> 2.9, 513 x 511 4.5 -> 2.9, 4097 x 1999 82 -> 60.
TilePlan tile_plan(TileTable& table, int storage, int um, int basis, int nv, int nx, int ny,
                   int64_t n, double least) {
    TilePlan best;
    best.us = least;
    // What a launch of s steps takes at least: the launch, and each step's latency or the pipes'
    // share of the lattice.
    const TileCost cost(storage, um, basis, nv);
    const double share = kItem * (double)nx * ny / (64.0 * sm_count());
    const double step = cost.scale * (share > kStepFloor ? share : kStepFloor);
    // likely lengths first: a good plan early drops most of the others unsearched
    constexpr int lengths[] = {5, 10, 4, 3, 8, 6, 12, 2};
    for (int want : lengths) {
        // an odd number of passes for an odd number of steps, an even one for an even number:
        // the state ends in the buffer in which single steps would leave it
        int64_t m = (n + want - 1) / want;
        m += (m ^ n) & 1;
        const int s = (int)((n + m - 1) / m);
        if (s < 2 || m * (cost.launch + step * s) >= best.us) continue;
        TilePlan& pass = table.best[s];
        const double least = best.us / m;
        if (pass.steps == 1 && pass.us < least)
            pass = tile_pass(storage, um, basis, nv, nx, ny, s, least);
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
