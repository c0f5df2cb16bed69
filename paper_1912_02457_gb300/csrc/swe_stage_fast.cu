// swe_stage_fast.cu -- the FP32 stage kernels of libswe (the fast path).
//
// Same scheme as the reference stage kernel (swe_device.cuh), organised for
// GB300:
//  * two warps march up a strip of 28 output columns (32 lanes: two halo
//    columns on each side), one row per iteration, the first a row ahead of
//    the second (swe_march.cuh): every cell's primitives, reconstructions and
//    face fluxes are computed once, and the x-neighbours come from warp
//    shuffles;
//  * a cell is one vector {eta, hu, hv, f}, so a row of a strip is one
//    asynchronous copy of 512 bytes per buffer;
//  * the CFL reduction is a warp/block max, and the last block of stage 2 to
//    finish advances the device clock (t, dt, forcing brackets), so a step
//    is two launches and needs no host round trip;
//  * ghosts of nested edges read an edge-state buffer that stage 1 fills for
//    the next time level; periodic ghosts read their periodic image;
//  * a pair of warps takes an item of the domain's work plan. A single domain's
//    arguments stay in the launch's parameter space (constant operands of
//    the march); a batch's come from a device tile table, through shared
//    memory. The march's arithmetic is spelled out, so both give a cell the
//    same bits;
//  * denormal results flush to zero (values below 1.2e-38, far below
//    anything the scheme resolves).
#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <cstring>
#include <queue>
#include <vector>

#include "swe_march.cuh"
#include "swe_kernels.h"

namespace swe {

namespace {

static_assert(kStrip == kStripColumns, "the planner's strips are the march's");
constexpr int kPairs = 4;            // items per block, two warps each
constexpr int kThreads = kPairs * 64;
// resident blocks per SM the register budgets target: 64 registers without a
// spill for a single domain and for stage 1 of a batch with uniform winds (with
// gridded ones that stage spills 8 bytes at 64 registers: a 12-domain ensemble with
// gridded winds takes 410 us a step, at 80 registers 428); stage 2 of a batch,
// whose arguments are in shared memory, needs 80 (at 64 it spills, and with the
// shared memory of the rings the L1 cache left over is too small for spills:
// 12.9 -> 22.2 ms on a 12-domain ensemble of 32 steps). Domains of a batch seldom
// leave an SM idle at a stage's end, so there a kernel per stage wins over one
// footprint for both: 12.0 -> 11.6 ms, and 11.2 with a march for each value of
// the Kahan flag, which is each domain's own.
constexpr int kMinBlocks = 4, kBatchMinBlocks = 3;
// The end of a step: every block leaves its CFL maximum and counts itself, the
// last one advances the device clock (clock_update in swe_device.cuh). Every
// other SM idles meanwhile, so the clock is worked out on a second warp while
// the first one's fence and count are in flight (0.7 and 0.5 us): from inputs
// that no kernel writes before it, loaded at the block's start, and the
// largest maximum seen so far, which nearly always is the final one (else it is
// worked out again). Blocks that cannot be among the last ones skip that, and so
// do batches (AHEAD false), whose domains end while others keep the SMs busy and
// whose kernel has no registers for it (260 bytes of spills, 12.0 -> 13.6 ms on
// the 12-domain ensemble). The end of a step took 5500 cycles without forcing and
// 6800 with it (fence 1550, count 1100, exchange 700, clock 2200 or 3500), now
// some 3500: 350 x 350 19.2 -> 18.1 us a step.
struct Finish {
    ClockIn in;
    unsigned int bits;
    int last;
};
constexpr int kNearLast = 2 * 152;

__device__ __forceinline__ void finish_load(const StageArgs<float> &a, const StepCtl *ctl, int mode, Finish &f) {
    ClockIn c;
    clock_load_state(ctl, c, mode);
    clock_load_forcing(a.clk, a.bnd, a.wind, c);
    f.in = c;
}

// Warps 0 and 1 of the block, after a barrier that follows finish_load.
template <bool AHEAD>
__device__ __forceinline__ void finish_step(const StageArgs<float> &a, float block_speed, int nblocks, int mode,
                                            int warp, int lane, Finish &f) {
    StepCtl *ctl = a.ctl;
    // a sub-domain leaves its maximum for the clock of all sub-domains
    if (mode == 5) {
        if (warp == 0 && lane == 0) atomicMax(&ctl->speed32, __float_as_uint(block_speed));
        return;
    }
    ClockOut o;
    unsigned int guess = 0u;
    bool have = false;
    if (lane == 0 && warp == 0) {
        atomicMax(&ctl->speed32, __float_as_uint(block_speed));
        __threadfence();                       // the block's maximum lands before its count
        const bool last = atomicAdd(&ctl->blocks_done, 1u) == (unsigned int)nblocks - 1u;
        f.last = last;
        if (last) {
            // atomics are performed at L2, so the exchange sees every block's
            // maximum; the next kernel sees the clock's writes (kernel boundary)
            f.bits = atomicExch(&ctl->speed32, 0u);
            ctl->blocks_done = 0u;
            if (!AHEAD) {
                clock_compute(a.clk, a.bnd, a.wind, (double)__uint_as_float(f.bits), mode, f.in, o);
                clock_store(ctl, o);
            }
        }
    } else if (AHEAD && lane == 0) {
        const unsigned int seen = *(volatile unsigned int *)&ctl->speed32;
        const unsigned int count = *(volatile unsigned int *)&ctl->blocks_done;
        if (count + kNearLast >= (unsigned int)nblocks) {
            guess = max(seen, __float_as_uint(block_speed));
            clock_compute(a.clk, a.bnd, a.wind, (double)__uint_as_float(guess), mode, f.in, o);
            have = true;
        }
    }
    if (!AHEAD) return;
    asm volatile("bar.sync %0, 64;" ::"n"(kPairs + 1) : "memory");
    if (warp == 0 || lane != 0 || !f.last) return;
    if (!have || guess != f.bits)
        clock_compute(a.clk, a.bnd, a.wind, (double)__uint_as_float(f.bits), mode, f.in, o);
    clock_store(ctl, o);
}

// One block of one domain: its kPairs pairs of warps take the items blk*kPairs
// .. blk*kPairs+kPairs-1 of the domain's plan, each a strip of 28 output
// columns by a run of rows. Numbering items linearly (instead of giving a
// block a 2-D tile) leaves no idle warps at the right edge and lets the item
// height be chosen to fill whole waves. `nblocks`: blocks of this domain in
// this launch (the last of them to finish stage 2 advances the domain's
// clock).
// MIXED: a batch.
template <int STAGE, bool GW, bool MIXED>
__device__ __forceinline__ void stage_tile(const StageArgs<float> &a, int blk, int nblocks, const bool KAHAN,
                                           Ring<float> *ring) {
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5, pair = warp & (kPairs - 1);
    const int item = blk * kPairs + pair;
    const bool live = item < a.n_items;
    int strip = 0, j0 = 0, j1 = 0;
    if (live && SWE_CHECK(a, item, a.n_items)) {
        const uint2 it = __ldg(a.items + item);
        strip = (int)it.x;
        j0 = (int)(it.y & 0xffffu);
        j1 = min(j0 + (int)(it.y >> 16), a.ny);
    }
    // everything above reads what no kernel writes (arguments, the plan). Stage 1
    // does not write the clock either: stage 2 reads it, and starts its march,
    // beside the end of stage 1
    if (STAGE != 2) previous_kernel_done();
    const StepCtl *ctl = a.ctl;
    if (STAGE == 2) {
        // from L2: the L1 may still hold the line of the step before. Once a
        // block: a read of that one line by each warp made the stage slower by
        // 1.3 us where blocks fill the GPU
        __shared__ StepCtl copy;
        constexpr int kCtlWords = sizeof(StepCtl) / 8;
        if (threadIdx.x < kCtlWords)
            reinterpret_cast<unsigned long long *>(&copy)[threadIdx.x] =
                __ldcg(reinterpret_cast<const unsigned long long *>(a.ctl) + threadIdx.x);
        __syncthreads();
        ctl = &copy;
    }
    const int done = ctl->done, par = ctl->parity;
    const double dt = ctl->dt;
    const float taux = STAGE == 0 ? 0.f : ctl->tau_f[STAGE - 1][0];
    const float tauy = STAGE == 0 ? 0.f : ctl->tau_f[STAGE - 1][1];
    if (done) {                                    // forecast horizon reached (block-uniform)
        if (STAGE == 2) previous_kernel_done();
        return;
    }
    // stage 1 also evaluates the external edge state of the next time level
    // (used by stage 2 and by stage 1 of the next step); the interior
    // blocks of the middle of the domain take it
    if (STAGE == 1) {
        const int b = blk + nblocks / 2 < nblocks ? blk + nblocks / 2 : blk + nblocks / 2 - nblocks;
        edge_fill(a, par ^ 1, 1, b * kThreads + threadIdx.x, nblocks * kThreads);
    }
    float speed = 0.f;
    const int mode = STAGE == 0 ? 3 : a.clk.split ? 5 : (a.clk.cfl_faces ? 4 : 1);
    __shared__ Finish fin;
    // (a consumer warp, which waits for its first row anyway)
    if (STAGE != 1 && threadIdx.x == kPairs * 32 && mode != 5) finish_load(a, ctl, mode, fin);
    if (live) {
        const StripCtx<float> k = strip_ctx<float, STAGE>(a, strip, j0, j1, par, dt, taux, tauy);
        if (warp < kPairs)
            speed = march_x<float, STAGE, GW, MIXED>(a, k, strip, ring[pair], 1 + pair) * a.inv_dx;
        else
            speed = march_y<float, STAGE, MIXED>(a, k, ring[pair], 1 + pair, KAHAN);
        // stage 2: the CFL maximum of the cells (eq:cfl with the cell
        // averages); the speed pass: the largest face speed over the cell
        // size (eq:cfl with the faces' one-sided speeds). A window of a
        // larger domain takes the maximum over its own cells: its halo rows
        // are not in its plan, and the lanes of its halo columns (written,
        // then overwritten by the halo exchange) drop out here, once, rather
        // than in every row
        if (STAGE == 2 && (unsigned)(k.i - a.own_x0) >= (unsigned)(a.own_x1 - a.own_x0)) speed = 0.f;
    }
    if (STAGE == 0 || STAGE == 2) {
        __shared__ float sh[2 * kPairs];
        for (int o = 16; o > 0; o >>= 1) speed = fmaxf(speed, __shfl_xor_sync(0xffffffffu, speed, o));
        if (lane == 0) sh[warp] = speed;
        __syncthreads();
        if (warp > 1) return;
        float bs = 0.f;
        for (int q = 0; q < 2 * kPairs; q++) bs = fmaxf(bs, sh[q]);
        finish_step<!MIXED>(a, bs, nblocks, mode, warp, lane, fin);
    }
}

}  // namespace

// A single domain: its arguments sit in the kernel's parameter space, where
// the march reads them as constant operands (no table lookups, no staging).
// GW: the kernel for domains with gridded wind; uniform-wind domains carry
// no code of the gridded path in their march. Both stages (and the speed
// pass) are one kernel: consecutive launches overlap at their ends, and an SM
// whose registers and shared memory are cut into blocks of one size has no
// holes that a block of the next launch does not fit into (with kernels of 56
// and 64 registers 2-5% of the stage-2 blocks had to wait for a second wave).
template <bool GW, bool KAHAN>
__global__ void __launch_bounds__(kThreads, kMinBlocks)
stage_kernel(const __grid_constant__ OneDomain one) {
    __shared__ Ring<float> ring[kPairs];
    // the next kernel may start while this one drains (stage 1 lets it later:
    // previous_kernel_done)
    if (one.stage != 1) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (one.stage == 2) stage_tile<2, GW, false>(one.args, blockIdx.x, one.tiles, KAHAN, ring);
    else if (one.stage == 1) stage_tile<1, GW, false>(one.args, blockIdx.x, one.tiles, KAHAN, ring);
    else stage_tile<0, GW, false>(one.args, blockIdx.x, one.tiles, KAHAN, ring);
}

// Batch kernel: block t takes tile t of the tile table of all domains
// (tile t belongs to the domain d = tile_dom[t], tile_start[d] <= t <
// tile_start[d+1]; a grid smaller than the table walks it with a stride).
// One block per tile lets the hardware scheduler balance uneven tiles (7%
// faster than a persistent grid on a 64-domain ensemble); the table lives
// in device memory, so a captured graph stays valid while domains come and
// go with an unchanged tile count. A batch with any gridded-wind domain
// launches the GW kernel for all of them.
template <int STAGE, bool GW>
__global__ void __launch_bounds__(kThreads, STAGE == 1 ? kMinBlocks : kBatchMinBlocks)
stage_batch_kernel(const BatchTable tab) {
    __shared__ Ring<float> ring[kPairs];
    // the domain's arguments, staged once per block in shared memory (they
    // are read uniformly by every thread)
    __shared__ StageArgs<float> sa;
    // (as in stage_kernel)
    if (STAGE != 1) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int n_dom = *tab.n_domains;
    const int total = n_dom > 0 ? tab.tile_start[n_dom] : 0;
    int have = -1;
    for (int t = blockIdx.x; t < total; t += gridDim.x) {
        const int d = tab.tile_dom[t];
        const int first = tab.tile_start[d];
        const int ntiles = tab.tile_start[d + 1] - first;
        if (d != have) {
            const int *src = reinterpret_cast<const int *>(tab.args + d);
            int *dst = reinterpret_cast<int *>(&sa);
            for (int k = threadIdx.x; k < (int)(sizeof(StageArgs<float>) / sizeof(int)); k += blockDim.x)
                dst[k] = src[k];
            __syncthreads();
            have = d;
        }
        if (STAGE == 2 && sa.comp[0] != nullptr) stage_tile<STAGE, GW, true>(sa, t - first, ntiles, true, ring);
        else stage_tile<STAGE, GW, true>(sa, t - first, ntiles, false, ring);
        __syncthreads();                        // shared scratch reused by the next tile
    }
}

// ---------------------------------------------------------------------------
// launch configuration

int fast_slots() {
    static int slots = 0;
    if (!slots) {
        int dev = 0, sms = 0, per_sm = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, stage_kernel<false, true>, kThreads, 0);
        slots = (sms > 0 ? sms : 152) * (per_sm > 0 ? per_sm : 4) * kPairs;
    }
    return slots;
}

// ---------------------------------------------------------------------------
// work planning: warp items of variable height
//
// A warp item is a strip of 28 output columns by a run of rows
// [j0, j0 + n), packed as {strip, j0 | n << 16}. A row costs about the same
// everywhere except where the march takes its slow path (a lane on land or a
// drying shelf: +40%), the general loads (the strips whose lanes reach past
// the west or east edge, and the items at the south and north edges: +30%),
// ghosts of a nested edge (another +10%) and, in stage 2, flow-relaxation
// zones (+40%). The weights come from per-item times of both stages on the
// coastal 1024 x 1024 step (a %globaltimer probe per warp in a scratch build:
// 0.53 us per plain row, +0.28 us per slow row; the start of an item and its
// four halo rows take as long as some eight plain rows). Without the slow-path
// term the slowest item of stage 1 ended 6.8 us after the median one, now 4.7 us.
// The halo weight decides how finely a domain is cut: 400 (four rows) measured
// 2-5% faster than the single row of before on the coastal domains of 1024 and
// 4096 cells a side, 200 to 800 within 1% of it. Rows without a wet cell in
// the strip are left out (land cells are never written and never enter the CFL
// maximum, and a march recomputes its own halo): each strip falls into
// segments of wet rows, split where a land run is longer than a halo. A
// budget (kPlanUnit per plain row) cuts a segment of cost C into
// ceil(C / budget) items of equal cost, so the item count follows the
// budget smoothly and fast_budget can fill the GPU's resident warp slots.

namespace {

constexpr int kNonIntCost = 30, kGhostCost = 10, kFrsCost = 40, kRoughCost = 40, kHaloCost = 400;
constexpr int kEdgeRows = 12;

struct PlanCtx {
    int nx, ny, strips, fw;
    bool nest[4];
    const unsigned char *wet;       // strips x ny, strip-major; NULL: all wet
    bool is_wet(int j, int s) const { return !wet || wet[(size_t)s * ny + j] != 0; }
    // the strips whose lanes reach past the west or east edge march on the
    // general load path (ghost handling on every row)
    bool cols_edge(int s) const { return s * kStrip - 2 < 0 || s * kStrip + 29 >= nx; }
    int strip_extra(int s) const {
        int c = cols_edge(s) ? kNonIntCost : 0;
        if ((s == 0 && nest[EDGE_W]) || (s == strips - 1 && nest[EDGE_E])) c += kGhostCost;
        const int c0 = s * kStrip, c1 = std::min(c0 + kStrip, nx);
        if ((nest[EDGE_W] && c0 < fw) || (nest[EDGE_E] && c1 > nx - fw)) c += kFrsCost;
        return c;
    }
    int row_cost(int j, int s, int xs) const {
        const bool frs = is_wet(j, s) && ((nest[EDGE_S] && j < fw) || (nest[EDGE_N] && j >= ny - fw));
        // the first and last item of a strip (about kEdgeRows rows) march on
        // the general load path too
        const bool edge = !cols_edge(s) && (j < kEdgeRows || j >= ny - kEdgeRows);
        const bool rough = wet && (wet[(size_t)s * ny + j] & kRough);
        return kPlanUnit + xs + (frs ? kFrsCost : 0) + (edge ? kNonIntCost : 0) + (rough ? kRoughCost : 0);
    }
};

struct Segment {
    int strip, start, rows;
    long long cost;
};

PlanCtx plan_ctx(int nx, int ny, const unsigned char *wet, const int bc[4], int frs_width) {
    PlanCtx p;
    p.nx = nx; p.ny = ny; p.strips = (nx + kStrip - 1) / kStrip; p.fw = frs_width; p.wet = wet;
    for (int e = 0; e < 4; e++) p.nest[e] = bc[e] == BC_NESTED;
    return p;
}

std::vector<Segment> plan_segments(const PlanCtx &p) {
    std::vector<Segment> seg;
    for (int s = 0; s < p.strips; s++) {
        const int xs = p.strip_extra(s);
        int j = 0;
        for (;;) {
            while (j < p.ny && !p.is_wet(j, s)) j++;
            if (j >= p.ny) break;
            const int start = j;
            int end = j;                // one past the last wet row
            while (j < p.ny) {
                if (p.is_wet(j, s)) { end = ++j; continue; }
                int L = 0;
                while (j + L < p.ny && !p.is_wet(j + L, s)) L++;
                if (j + L >= p.ny || L * kPlanUnit >= kHaloCost) break;
                j += L;
            }
            long long c = 0;
            for (int r = start; r < end; r++) c += p.row_cost(r, s, xs);
            seg.push_back({s, start, end - start, c});
            j = end;
        }
    }
    return seg;
}

// items of one segment under a budget
long long seg_items(const Segment &g, int budget) {
    return std::min<long long>(g.rows, std::max<long long>(1, (g.cost + budget - 1) / budget));
}

}  // namespace

int fast_strips(int nx) { return (nx + kStrip - 1) / kStrip; }

int fast_budget(int nx, int ny, const unsigned char *wet, const int bc[4], int frs_width, int n_slots) {
    const std::vector<Segment> seg = plan_segments(plan_ctx(nx, ny, wet, bc, frs_width));
    // Score: the fraction of the last wave filled (items / whole waves of
    // resident warps) times the share of the work that is not halo. Items
    // are kept to 32 rows or fewer: longer marches measured slower on every
    // domain that needs them (2048^2 to 8192^2 coastal: 6-12%), even where
    // they would fill the slots exactly. Small domains take items down to two
    // rows: a warp's march is a chain of dependent row iterations, so short
    // items on more warps finish sooner (350^2: 35%, 512^2: 20% faster than
    // items of eight rows or more).
    const double slots = n_slots;
    int best = 2 * kPlanUnit;
    double best_score = -1.0;
    for (int b = 2 * kPlanUnit; b <= 32 * kPlanUnit; b += kPlanUnit / 20) {
        long long n = 0, work = 0;
        for (const Segment &g : seg) {
            const long long k = seg_items(g, b);
            n += k;
            work += g.cost + k * kHaloCost;
        }
        if (n == 0) return 8 * kPlanUnit;      // all land: one no-op item whatever the budget
        const double waves = (double)n / slots;
        const double fill = waves / (waves <= 1.0 ? 1.0 : std::ceil(waves - 1e-9));
        const double useful = (double)(work - n * kHaloCost) / (double)work;
        const double score = fill * useful;
        if (score > best_score + 1e-12) { best_score = score; best = b; }
    }
    return best;
}

void fast_plan(int nx, int ny, const unsigned char *wet, const int bc[4], int frs_width, int budget,
               int per_block, int slots, std::vector<uint2> &items) {
    items.clear();
    const PlanCtx p = plan_ctx(nx, ny, wet, bc, frs_width);
    std::vector<long long> pref, cost;
    for (const Segment &g : plan_segments(p)) {
        const int xs = p.strip_extra(g.strip);
        pref.assign((size_t)g.rows + 1, 0);
        for (int r = 0; r < g.rows; r++) pref[r + 1] = pref[r] + p.row_cost(g.start + r, g.strip, xs);
        const int k = (int)seg_items(g, budget);
        // cut where the cost prefix is nearest to cost * q / k, each item
        // keeping at least one row
        int r0 = 0;
        for (int q = 1; q <= k; q++) {
            int r1 = g.rows;
            if (q < k) {
                const long long target = g.cost * q / k;
                r1 = r0 + 1;
                while (r1 < g.rows - (k - q) && pref[r1] < target) r1++;
                if (r1 - 1 > r0 && target - pref[r1 - 1] < pref[r1] - target) r1--;
            }
            items.push_back(make_uint2((unsigned)g.strip, (unsigned)(g.start + r0) | ((unsigned)(r1 - r0) << 16)));
            cost.push_back(pref[r1] - pref[r0] + kHaloCost);
            r0 = r1;
        }
    }
    if (items.empty()) { items.push_back(make_uint2(0u, 1u << 16)); cost.push_back(1); }
    const int n = (int)items.size(), nb = (n + per_block - 1) / per_block;
    const auto row_major = [&](int a, int c) {
        const unsigned ja = items[a].y & 0xffffu, jc = items[c].y & 0xffffu;
        return ja != jc ? ja < jc : items[a].x < items[c].x;
    };
    std::vector<int> order(n);
    for (int k = 0; k < n; k++) order[k] = k;
    std::vector<uint2> out;
    out.reserve(n);
    if (n > slots || budget < 8 * kPlanUnit) {
        // part of a batch, several waves, or short items: row-major order,
        // a block's warps taking neighbouring strips of the same rows (they
        // share halo lines in L1, which short items and later waves depend
        // on; measured 1-2% faster than balanced blocks there)
        std::sort(order.begin(), order.end(), row_major);
        for (int k : order) out.push_back(items[k]);
        items.swap(out);
        return;
    }
    // one wave of long items: blocks of per_block items with equal total cost
    // (largest item first to the lightest block with room), so that the SMs,
    // whichever blocks they get, carry equal work (coastal 1024^2: +2.6%; FP64
    // 512 x 384 290.6 -> 282.5 us a step in its blocks of two items); within a
    // block, row-major order. (When the item count is not a multiple of per_block
    // a packed block other than the last may hold fewer items, and the launch's
    // blocks then straddle packed blocks after it; keeping every short block last
    // measured no different.)
    std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return cost[a] > cost[b]; });
    typedef std::pair<long long, int> Load;
    std::priority_queue<Load, std::vector<Load>, std::greater<Load>> heap;
    for (int b = 0; b < nb; b++) heap.push(Load(0, b));
    std::vector<std::vector<int>> blk(nb);
    for (int k : order) {
        Load l = heap.top();
        heap.pop();
        blk[l.second].push_back(k);
        if ((int)blk[l.second].size() < per_block) heap.push(Load(l.first + cost[k], l.second));
    }
    for (int b = 0; b < nb; b++) {
        std::sort(blk[b].begin(), blk[b].end(), row_major);
        for (int k : blk[b]) out.push_back(items[k]);
    }
    items.swap(out);
}

int fast_pairs() { return kPairs; }

int fast_step_parts(bool faces) { return faces ? 3 : 2; }

const char *fast_part_name(int part, bool faces) {
    static const char *names[3] = {"speed", "stage1", "stage2"};
    if (faces) return part >= 0 && part < 3 ? names[part] : "";
    return part >= 0 && part < 2 ? names[part + 1] : "";
}

// Blocks (of kPairs warp items) a launch over n_items items needs.
int fast_tiles(int n_items) { return (n_items + kPairs - 1) / kPairs; }

// Per 28-column strip s and row j (out[s * ny + j], strip-major for the
// planner's walk down each strip): 0 where the strip holds no wet cell of row
// j (a cell is land when any of its corners is LAND), kWet, plus kRough where a
// lane of the march holds land or bed above the reference level (a drying
// shelf): those rows take the march's slow path.
//
// The march tells land by the sum of a cell's corners, at least LAND if one of
// them is. Depths no water has (infinite, or not a number in FP64) reach that
// sum without being land: the march would take such a cell for a coast, where
// the scheme gives no finite state. They are a numeric error of the domain.
template <typename T>
__global__ void wet_strips_kernel(const T *__restrict__ H, long long cpitch, int nx, int ny, int strips,
                                  unsigned char *__restrict__ out, StepCtl *ctl) {
    const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (t >= (long long)ny * strips) return;
    const int j = (int)(t / strips), s = (int)(t % strips);
    const int c0 = s * kStrip, c1 = min(c0 + kStrip, nx);
    const T *r0 = H + (long long)j * cpitch, *r1 = r0 + cpitch;
    bool wet = false, rough = false;
    for (int i = max(c0 - 2, 0); i < min(c1 + 2, nx); i++) {
        const T sum = (r0[i] + r0[i + 1]) + (r1[i] + r1[i + 1]);
        const bool land = r0[i] == kLand || r0[i + 1] == kLand || r1[i] == kLand || r1[i + 1] == kLand;
        wet |= !land && i >= c0 && i < c1;
        rough |= land || sum < T(0);
        if (!land && !(sum < T(kLand))) flag_error(ctl, j * nx + i);
    }
    out[(long long)s * ny + j] = wet ? (rough ? kWet | kRough : kWet) : 0;
}

template <typename T>
cudaError_t launch_wet_strips(const T *H, long long cpitch, int nx, int ny, unsigned char *out, StepCtl *ctl,
                              cudaStream_t st) {
    const int strips = fast_strips(nx);
    const long long n = (long long)ny * strips;
    wet_strips_kernel<T><<<(unsigned)((n + 255) / 256), 256, 0, st>>>(H, cpitch, nx, ny, strips, out, ctl);
    return cudaGetLastError();
}
template cudaError_t launch_wet_strips<float>(const float *, long long, int, int, unsigned char *, StepCtl *, cudaStream_t);
template cudaError_t launch_wet_strips<double>(const double *, long long, int, int, unsigned char *, StepCtl *, cudaStream_t);

// The external edge state of the current time level (stage-1 brackets).
__global__ void __launch_bounds__(256) edge_fill_kernel(const StageArgs<float> a) {
    edge_fill(a, a.ctl->parity, 0, blockIdx.x * blockDim.x + threadIdx.x, gridDim.x * blockDim.x);
}

long long edge_entries(int nx, int ny) { return 2LL * 4 * ((long long)nx + ny); }

cudaError_t launch_edge_fill(const StageArgs<float> &a, cudaStream_t st) {
    if (!a.edge || a.bnd.n <= 0) return cudaSuccess;
    const int total = 4 * (a.nx + a.ny);
    edge_fill_kernel<<<(total + 255) / 256, 256, 0, st>>>(a);
    return cudaGetLastError();
}

// Stage launches carry the programmatic-stream-serialisation attribute: a
// stage kernel that follows another one in the stream (or in a captured graph) is
// scheduled once every block of that one has triggered or ended, and waits in
// griddepcontrol.wait for its completion and its writes (back-to-back steps 2.2%
// faster on the coastal 1024^2 step). After any other stream work a launch is
// ordered as usual. What makes the early start safe:
//  * before their wait the speed pass and stage 1 read what no kernel writes:
//    arguments and items. They may be triggered by the kernel before them at its
//    start, as the speed pass and stage 2 do.
//  * stage 2 reads the clock and the state before its wait. So stage 1 triggers
//    only after its own wait (previous_kernel_done): when stage 2 starts, whatever
//    ran before stage 1 is complete, and stage 1 writes neither of the two. A
//    trigger of stage 1 at its start would let stage 2 read them while the stage 2
//    of the step before still writes them.
template <typename... Params, typename... Args>
static cudaError_t launch_stage(void (*kernel)(Params...), int blocks, cudaStream_t st, const Args &...args) {
    // one shared-memory split for all of them: an SM changes it only when idle
    cudaError_t e = cudaFuncSetAttribute((const void *)kernel, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof cfg);
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(kThreads);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    e = cudaLaunchKernelEx(&cfg, kernel, args...);
    return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t launch_batch_stage(const BatchTable &tab, int blocks, int stage, bool gridded, cudaStream_t st) {
    if (stage == 1)
        return launch_stage(gridded ? stage_batch_kernel<1, true> : stage_batch_kernel<1, false>, blocks, st, tab);
    return launch_stage(gridded ? stage_batch_kernel<2, true> : stage_batch_kernel<2, false>, blocks, st, tab);
}

cudaError_t launch_domain_stage(const OneDomain &domain, int stage, cudaStream_t st) {
    OneDomain one = domain;
    one.stage = stage;
    const bool gridded = one.args.wind.n > 0 && !one.args.clk.wind_uniform, kahan = one.args.comp[0] != nullptr;
    return launch_stage(gridded ? (kahan ? stage_kernel<true, true> : stage_kernel<true, false>)
                                : (kahan ? stage_kernel<false, true> : stage_kernel<false, false>),
                        one.tiles, st, one);
}

}  // namespace swe
