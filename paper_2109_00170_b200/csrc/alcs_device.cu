// Device-facing half of libalcs: upload of the packed weights and their launch schedules, launch
// planning, the convolution entry points, the tuner, the host-buffer variant and the layer stack.
#include <cuda_runtime.h>
#include <nvtx3/nvToolsExt.h>

#include <algorithm>
#include <cmath>
#include <memory>
#include <queue>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <new>
#include <vector>

#include "alcs_gather.h"
#include "alcs_internal.h"
#include "alcs_kernels.cuh"
#include "alcs_tc_prep.h"

namespace alcs {
void set_cuda_error_text(const char* s);
}

namespace {

using alcs::ConvArgs;
using alcs::KernelVariant;

#define ALCS_CUDA(call)                                        \
    do {                                                       \
        cudaError_t e_ = (call);                               \
        if (e_ != cudaSuccess) {                               \
            alcs::set_cuda_error_text(cudaGetErrorString(e_)); \
            (void)cudaGetLastError();                          \
            return ALCS_ERR_CUDA;                              \
        }                                                      \
    } while (0)

constexpr int kMaxSmem = 227 * 1024;

struct VariantInfo {
    KernelVariant v;
    int regs = 0;
    bool ready[64] = {};    // per device: the dynamic shared-memory attribute is a per-device setting
};

struct DeviceInfo {
    int sms = 0;
    int smem_optin = 0;
    double sm_hz = 0;       // maximum SM clock
    double hbm_bps = 0;     // nominal DRAM bandwidth (bus width x memory clock x 2), bytes per second
    bool ok = false;
};

std::mutex g_mu;
std::vector<VariantInfo> g_variants;
DeviceInfo g_dev[64];

void init_variants_locked()
{
    if (!g_variants.empty()) return;
    int n = 0;
    const KernelVariant* t = alcs::variants_f32_g4(&n);
    for (int i = 0; i < n; ++i) g_variants.push_back({t[i]});
    t = alcs::variants_f32_other(&n);
    for (int i = 0; i < n; ++i) g_variants.push_back({t[i]});
    t = alcs::variants_f16(&n);
    for (int i = 0; i < n; ++i) g_variants.push_back({t[i]});
    t = alcs::variants_f16_mma(&n);
    for (int i = 0; i < n; ++i) g_variants.push_back({t[i]});
    t = alcs::variants_bf16(&n);
    for (int i = 0; i < n; ++i) g_variants.push_back({t[i]});
}

// Which flavour of the launch schedule a variant takes (alcs_internal.h): the CUDA-core kernels take
// pair records balanced for their number of consumer warps and accumulator sets.
int flavour_of(const KernelVariant& v) { return v.mma ? 1 : alcs::balanced_flavour(v.nw, v.rw, v.split); }

// math_mode of alcs_launch_cfg for a variant
int mode_of(const KernelVariant& v) { return v.mma ? 2 : 1; }

int device_info(int dev, DeviceInfo* out)
{
    if (dev < 0 || dev >= 64) return ALCS_ERR_INVALID_ARG;
    std::lock_guard<std::mutex> lk(g_mu);
    if (!g_dev[dev].ok) {
        ALCS_CUDA(cudaDeviceGetAttribute(&g_dev[dev].sms, cudaDevAttrMultiProcessorCount, dev));
        ALCS_CUDA(cudaDeviceGetAttribute(&g_dev[dev].smem_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
        int khz = 0, mem_khz = 0, bus_bits = 0;
        ALCS_CUDA(cudaDeviceGetAttribute(&khz, cudaDevAttrClockRate, dev));
        ALCS_CUDA(cudaDeviceGetAttribute(&mem_khz, cudaDevAttrMemoryClockRate, dev));
        ALCS_CUDA(cudaDeviceGetAttribute(&bus_bits, cudaDevAttrGlobalMemoryBusWidth, dev));
        g_dev[dev].sm_hz = khz > 0 ? khz * 1e3 : 1.9e9;
        // the cost models only rank configurations, so the nominal figure (about 80 % of which a
        // streaming kernel reaches) is good enough
        const double nominal = 2.0 * mem_khz * 1e3 * (bus_bits / 8.0);
        g_dev[dev].hbm_bps = nominal > 0 ? 0.8 * nominal : 6.0e12;
        g_dev[dev].ok = true;
    }
    *out = g_dev[dev];
    return ALCS_OK;
}

// Make a variant launchable with large dynamic shared memory on the current device `dev` (once per
// device: the attribute belongs to the function as loaded on that device).
int prepare_variant(VariantInfo& vi, int dev)
{
    if (dev < 0 || dev >= 64) return ALCS_ERR_INVALID_ARG;
    std::lock_guard<std::mutex> lk(g_mu);
    if (vi.ready[dev]) return ALCS_OK;
    ALCS_CUDA(cudaFuncSetAttribute(vi.v.fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem));
    cudaFuncAttributes fa;
    ALCS_CUDA(cudaFuncGetAttributes(&fa, vi.v.fn));
    vi.regs = fa.numRegs;
    vi.ready[dev] = true;
    return ALCS_OK;
}

using alcs::Plan;
using alcs::Schedule;

struct StageLayout {
    int off_rec, off_rowoff, stage_bytes;
    int tail_bytes;     // shared memory after the ring (epilogue scratch of the tensor-core kernels)
};

StageLayout stage_layout(const KernelVariant& v, const Schedule& sc, int elt)
{
    StageLayout L;
    // X tile first; the tensor-core kernels pad every channel row by 16 bytes
    L.off_rec = sc.kc * (32 * v.p * elt + (v.mma ? 16 : 0));
    L.off_rowoff = L.off_rec + sc.wcap * 16;
    L.stage_bytes = L.off_rowoff + sc.ros * 4;
    L.tail_bytes = v.mma ? v.nw * 8 * (32 * v.p * 2 + 16) : 0;     // [8 channels][T pixels] fp16 per consumer warp
    // hand-over tiles of rows split into parts: a barrier, then two sets of max_x tiles of g*P*32 floats
    if (!v.mma && sc.max_x > 0) L.tail_bytes = 16 + 2 * sc.max_x * v.g * v.p * 32 * 4;
    return L;
}

size_t plan_smem(const StageLayout& L, int stages)
{
    return 16 * alcs::kMaxStages + (size_t)stages * L.stage_bytes + L.tail_bytes;
}

// The schedule for (kc, n_rg): sizes only (with_records = false) or complete.  Cached in w.
Schedule* get_schedule(const alcs_packed* w, int kc, int n_rg, bool with_records, int flavour)
{
    if (kc <= 0 || kc > w->cin) kc = w->cin;
    if (flavour >= 2) {     // the balanced builder raises n_rg to what the (warps x sets) capacity needs: key by the result
        const int cap = alcs::flavour_nwg(flavour) * alcs::flavour_rw(flavour);
        n_rg = std::max(std::max(1, (w->rows + cap - 1) / cap), std::min(n_rg, w->rows));
    }
    std::lock_guard<std::mutex> lk(w->mu);
    Schedule& sc = w->sched[alcs::sched_key(kc, n_rg, flavour)];
    try {
        if (sc.n_rg == 0 || (with_records && !sc.uploaded && sc.h_rec.empty() && sc.n_rec > 0)) {
            if (flavour == 1) alcs::build_schedule_mma(*w, kc, n_rg, with_records, sc);
            else if (flavour >= 2)
                alcs::build_schedule_balanced(*w, kc, n_rg, alcs::flavour_nwg(flavour), alcs::flavour_rw(flavour), with_records, sc,
                                              alcs::flavour_split(flavour) != 0);
            else alcs::build_schedule(*w, kc, n_rg, with_records, sc);
        }
    } catch (const std::bad_alloc&) {
        return nullptr;
    }
    return &sc;
}

int upload_schedule(const alcs_packed* w, Schedule* sc, cudaStream_t st)
{
    std::lock_guard<std::mutex> lk(w->mu);
    if (sc->uploaded) return ALCS_OK;
    auto fail = [&](cudaError_t e) {
        alcs::set_cuda_error_text(cudaGetErrorString(e));
        cudaFree(sc->rec); cudaFree(sc->slice); cudaFree(sc->rowoff); cudaFree(sc->rowmap);
        sc->rec = nullptr; sc->slice = sc->rowoff = sc->rowmap = nullptr;
        (void)cudaGetLastError();
        return e == cudaErrorMemoryAllocation ? ALCS_ERR_ALLOC : ALCS_ERR_CUDA;
    };
    cudaError_t e;
    if ((e = cudaMalloc(&sc->rec, sc->h_rec.size() + 64)) != cudaSuccess) return fail(e);
    if ((e = cudaMalloc(&sc->slice, sc->h_slice.size() * 4)) != cudaSuccess) return fail(e);
    if ((e = cudaMalloc(&sc->rowoff, sc->h_rowoff.size() * 4)) != cudaSuccess) return fail(e);
    if ((e = cudaMalloc(&sc->rowmap, sc->h_rowmap.size() * 4)) != cudaSuccess) return fail(e);
    // the sources are pageable host vectors: these copies return once the data has been staged
    if (!sc->h_rec.empty() &&
        (e = cudaMemcpyAsync(sc->rec, sc->h_rec.data(), sc->h_rec.size(), cudaMemcpyHostToDevice, st)) != cudaSuccess)
        return fail(e);
    if ((e = cudaMemcpyAsync(sc->slice, sc->h_slice.data(), sc->h_slice.size() * 4, cudaMemcpyHostToDevice, st)) != cudaSuccess) return fail(e);
    if ((e = cudaMemcpyAsync(sc->rowoff, sc->h_rowoff.data(), sc->h_rowoff.size() * 4, cudaMemcpyHostToDevice, st)) != cudaSuccess) return fail(e);
    if ((e = cudaMemcpyAsync(sc->rowmap, sc->h_rowmap.data(), sc->h_rowmap.size() * 4, cudaMemcpyHostToDevice, st)) != cudaSuccess) return fail(e);
    if ((e = cudaStreamSynchronize(st)) != cudaSuccess) return fail(e);
    sc->uploaded = true;
    std::vector<unsigned char>().swap(sc->h_rec);
    std::vector<int>().swap(sc->h_rowoff);
    return ALCS_OK;
}

void free_schedule_device(Schedule& sc)
{
    cudaFree(sc.rec); cudaFree(sc.slice); cudaFree(sc.rowoff); cudaFree(sc.rowmap);
    sc.rec = nullptr; sc.slice = sc.rowoff = sc.rowmap = nullptr;
    sc.uploaded = false;
}

// A rough per-layer time model (seconds) used to rank launch configurations.  Three resources
// are modelled per SM: FMA issue slots, shared-memory wavefronts and bytes arriving from L2;
// plus the HBM floor and the quantisation of work items over the persistent thread blocks.
double model_cost(const alcs_packed* w, const KernelVariant& v, const Schedule& sc, long long q,
                  const DeviceInfo& di, int occ)
{
    const int sms = di.sms;
    const int elt = (int)w->elt();
    const int T = 32 * v.p;
    const long long n_tiles = (q + T - 1) / T;
    const long long items = n_tiles * sc.n_rg;
    const long long slots = (long long)sms * occ;
    const long long rounds = (items + slots - 1) / slots;
    if (v.mma) {
        // shared-memory wavefronts dominate: per step and 16-pixel tile one 4-wavefront ldmatrix
        // (about 1.4 with the residual bank conflicts), plus the staging writes of the tile
        const double steps_item = (double)sc.n_rec * 16.0 / alcs::step_record_bytes(v.g) / sc.n_rg;
        const double lsu = steps_item * (2.0 * v.p * 4 * 1.4 + 3 + 2.0 * (v.g > 8 ? 2 : 1)) +
                           (double)sc.nch * sc.kc * T * elt / 128.0;
        const double issue = steps_item * (2.0 * v.p * (1 + (v.g > 8 ? 2 : 1)) * 2 + 12) / 4.0 +
                             (double)sc.rpg * sc.nch * 14.0 / 4.0;
        const double l2b = ((double)w->cin * T * elt + steps_item * alcs::step_record_bytes(v.g)) / (16.0 * v.npw);
        const double warps = (double)v.nw * occ;
        const double hide = std::min(1.0, 0.4 + warps / 20.0);
        const double item_cycles = (std::max(std::max(issue, lsu) / hide, l2b) + 2500.0) * (v.groups == 2 && rounds > 1 ? 0.7 : 1.0);
        const double t_sm = (double)rounds * occ * item_cycles / di.sm_hz;
        const double bytes = (double)q * (w->cin + w->cout) * elt;
        return std::max(t_sm, bytes / di.hbm_bps);
    }
    const int vg = (v.p * elt >= 16) ? 16 / elt : v.p;
    const int ng = v.p / vg;
    const int rec_b = alcs::record_bytes(v.g);
    const double pairs_item = (double)sc.n_rec * 16.0 / rec_b / sc.n_rg;
    const double seg_item = (double)std::min(sc.rpg, (w->rows + sc.n_rg - 1) / sc.n_rg) * sc.nch;
    const double fma_issue = pairs_item * (2.0 * v.g * v.p + 2 * ng + 6 + (elt == 2 ? v.p : 0)) / 4.0 + seg_item * 14.0 / 4.0;
    const double lsu = pairs_item * (2.0 * ng * (vg * elt * 32 / 128.0) + 1 + v.g / 2.0) +
                       (double)sc.nch * sc.kc * T * elt / 128.0;
    const double l2 = ((double)w->cin * T * elt + pairs_item * rec_b) / 48.0;
    const double warps = (double)v.nw * occ;
    const double hide = std::min(1.0, 0.5 + warps / 30.0);
    const double item_cycles = std::max(std::max(fma_issue, lsu), l2) / hide + 1500.0;
    const double t_sm = (double)rounds * occ * item_cycles / di.sm_hz;
    const double bytes = (double)q * (w->cin + w->cout) * elt;
    return std::max(t_sm, bytes / di.hbm_bps);
}

int occupancy_of(const VariantInfo& vi, size_t smem)
{
    int occ = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, vi.v.fn, (vi.v.nw + vi.v.npw) * 32, smem) != cudaSuccess) {
        (void)cudaGetLastError();
        return 0;
    }
    return occ;
}

// Where the kernel finds the unit words of a balanced schedule (they follow the row map on the device).
void set_unit_args(ConvArgs& a, const Schedule& sc, int mma)
{
    a.unit = nullptr; a.rgx = nullptr; a.off_xch = 0; a.xch_slots = 0;
    if (mma || !sc.balanced || sc.max_x <= 0) return;      // (only the split flavour of the kernel is given such schedules)
    a.unit = sc.rowmap + (size_t)sc.n_rg * sc.rpg;
    a.rgx = sc.rowmap + 2 * (size_t)sc.n_rg * sc.rpg;
    a.xch_slots = sc.max_x;
}

// Blocks of the longest block row.  (No lock: a caller may hold w->mu, and every thread computes the same value.)
int longest_row(const alcs_packed* w)
{
    int longest = w->max_row_blocks;
    if (longest < 0) {
        longest = 0;
        for (int r = 0; r < w->rows; ++r) longest = std::max(longest, w->row_ptr[r + 1] - w->row_ptr[r]);
        w->max_row_blocks = longest;
    }
    return longest;
}

// The small-problem kernel as a plan.  Its cost: a launch, then the longest of: the rounds of dependent loads (a warp
// issues the input vectors of four blocks and waits for them; a thread block's columns take `batches` such rounds) with
// each block's start and its sum over the warps, the bytes of X, which every block row fetches for itself from L2, and
// the arithmetic.  A fit to 1,600 launches of random shapes on one B200: median error 12 %.
bool gather_plan(const alcs_packed* w, int n, int hw, int p, int ks, const DeviceInfo& di, Plan* out)
{
    const int sms = di.sms;
    if (w->dt != ALCS_F32) return false;
    if (!alcs::gather_config_ok(w->g, p, ks, false)) return false;
    const long long tiles = (hw + 32 * p - 1) / (32 * p);
    const long long blocks = (long long)w->rows * n * tiles;
    if (blocks > (1ll << 22)) return false;
    Plan pl;
    pl.variant = -1; pl.gather = 1; pl.gp = p; pl.gks = ks;
    const bool vec = hw % 4 == 0 && p >= 4;
    const double per_row = w->rows ? (double)w->nb / w->rows : 0.0;
    const double batches = std::ceil(per_row / ks / 4.0), longest = std::ceil((double)longest_row(w) / ks / 4.0);
    const double resident = std::max(1, (w->g * p > 16 ? 512 : 1024) / (ks * 32));          // thread blocks per SM
    const double rounds = (double)blocks / (sms * resident), share = w->g * p / 32.0;       // of the most outputs a lane can hold
    const double batch_us = (p == 2 ? 0.74 : p == 4 ? 0.725 : 0.77) * (vec || p == 2 ? 1.0 : 1.08);
    const double loads = (std::max(1.0, rounds) * (batches * batch_us + 0.078 * ks * share) + rounds * 0.885 +
                          0.79 * std::max(0.0, longest - batches) * batch_us) * (1.0 + 0.32 * share);
    const double px = (double)n * tiles * 32.0 * p;
    const double l2 = (double)w->nb * px * 4 / (vec ? 9.9e6 : 4.4e6), fma = (double)w->nb * w->g * px * 28.1e-6 / sms;
    const double hbm = (double)n * hw * (w->cin + w->cout) * 4 / 7.0e6;
    // (a second fit, by whole waves of thread blocks, is the better one where there are several of them: 18 us, not 12, for
    // 96 -> 160 channels at 13x13, batch 48; the longer one counts)
    const double waves = std::ceil(rounds), wave_us = (p == 2 ? 0.55 : p == 4 ? 0.7 : 0.9) * (vec || p == 2 ? 1.0 : 1.3);
    const double by_waves = std::max(waves * batches * wave_us + (waves - 1) * 1.4, (double)w->nb * px * 4 / (vec ? 5.5e6 : 3.3e6));
    pl.cost = 1e-6 * std::max(2.0 + std::max({loads, l2, fma, hbm}), 2.6 + by_waves);
    *out = pl;
    return true;
}

// Most images for which the small-problem kernel is considered (beyond, the bytes of X decide against it anyway).
constexpr long long kGatherImages = 64;

// A layer as the planner sees it: output and input size, what the call adds to the convolution.
struct CallShape {
    int n, oh, ow, h, wd, stride = 1;
    bool residual = false;
    bool y32 = false;       // fp32 output of 16-bit operands
    int images() const { return std::max(1, n); }
    int hw() const { return oh * ow; }
    long long q() const { return (long long)images() * hw(); }
};

alcs::TcProblem tc_problem(const void* x, void* y, int n, int h, int wd, const float* bias, unsigned flags, const void* residual, int stride,
                           int h_in, int wd_in)
{
    const int k = stride > 1 ? 1 : 0;
    return {x, y, bias, residual, n, h, wd, h_in, wd_in, stride, 0, k, k, flags};
}

// A pointwise layer of n images of h x wd pixels.
CallShape pointwise(int n, int h, int wd, unsigned flags) { return {n, h, wd, h, wd, 1, false, (flags & ALCS_Y_F32) != 0}; }

// (for estimates: no buffers, any address for a residual)
alcs::TcProblem tc_problem(const CallShape& c)
{
    static const char some = 0;
    return tc_problem(nullptr, nullptr, c.images(), c.oh, c.ow, nullptr, c.y32 ? ALCS_Y_F32 : 0, c.residual ? &some : nullptr, c.stride, c.h, c.wd);
}

// Can the tcgen05 kernel take the layer (whatever the channels per tile)?  A strided one: rows of 4-byte copies only, as
// 16-bit 14x14 images have them, cost more than the gather pass of the other kernels (31 us against 15 for 231 -> 604
// channels, 14 x 14 at stride 2, batch 15, fp16).  The answer follows from the shape and the weights alone, so that calls
// with another X find what the first one prepared.
bool tc_ok(const alcs_packed* w, const CallShape& c)
{
    if (c.q() <= 0 || !alcs::tc_fits(w, 1, c.images(), (long long)c.h * c.wd, c.hw())) return false;
    return c.stride == 1 || ((size_t)c.wd * w->elt() % 8 == 0 && alcs::tc_patch_fits(w, tc_problem(c), alcs::kTcMaxN));
}

// alcs_tc16.cu takes 16-bit operands at stride 1.
bool tc16_ok(const alcs_packed* w, const CallShape& c) { return w->dt != ALCS_F32 && c.stride == 1; }
// producer_warps of a configuration that names the kernel of such a layer: alcs_tc.cu, alcs_tc16.cu.  Its `warps` are 32 pixels of the
// tile each then (with pixels_per_lane 1, as the staged kernels count).
constexpr int kTcProducers = 4, kTc16Producers = 8;

// The tcgen05 kernel that is named with n output channels per tile as a plan: alcs_tc.cu, or alcs_tc16.cu with the most pixels per tile
// that are no more than `pixels`, or with those that are expected to take the least.
constexpr int kAnyPixels = -1;
Plan tc_plan_on(const alcs_packed* w, int n, const CallShape& c, int sms, int pixels)
{
    Plan p;
    p.n_rg = (w->cout + n - 1) / n;
    p.tc_n = ((w->cout + p.n_rg - 1) / p.n_rg + 15) / 16 * 16;       // (the equal split into that many tiles)
    p.cost = 1e-6 * (pixels ? alcs::tc16_layer_us(w, tc_problem(c), p.tc_n, sms, std::max(0, pixels), &p.tc_px) : alcs::tc_layer_us(w, tc_problem(c), p.tc_n, sms));
    return p;
}

// Of these channels per tile, the plan that is expected to be the fastest; the two kernels are compared at the best of their own.
// Rows that alcs_tc16.cu picks apart have to promise 30 %: its estimate is 19 % off there (median), and no measure of the shape, output
// channels least of all, tells the layers that gain from those that don't.  200 layers of random shapes with such rows, against
// alcs_tc.cu alone: 31 chosen, 1.05 times as fast (geometric mean over all), none more than 4 % slower; at 20 %, 52 chosen, 1.06,
// six slower by up to 29 %.  Rows copied as they are, 5 %: 80 layers, 50 chosen, 1.28, one slower (7 %).
// against: what the staged kernels have to beat, the estimate of alcs_tc.cu where rows are picked apart (156 -> 43 @7, batch 11: 16 us
// where 9 are expected, 12 staged).
constexpr double kRawMargin = 1.3, kDirectMargin = 1.05;
Plan tc_best(const alcs_packed* w, const int* n, int count, const CallShape& c, int sms, double* against = nullptr)
{
    auto best_on = [&](int pixels) {
        Plan best = tc_plan_on(w, n[0], c, sms, pixels);
        for (int i = 1; i < count; ++i) {
            const Plan p = tc_plan_on(w, n[i], c, sms, pixels);
            if (p.cost < best.cost) best = p;
        }
        return best;
    };
    Plan best = best_on(0);
    if (against) *against = best.cost;
    if (!tc16_ok(w, c)) return best;
    const bool direct = (size_t)c.hw() * w->elt() % 8 == 0;
    const Plan other = best_on(kAnyPixels);
    if (other.cost * (direct ? kDirectMargin : kRawMargin) < best.cost) {
        best = other;
        if (against && direct) *against = best.cost;
    }
    return best;
}

// What a tuner compares with n output channels per tile: both kernels, and of alcs_tc16.cu a few heights beside the one that is expected to
// be the best (the estimate's median error is 9 %, the heights next to it differ by less).
void tc_plans(const alcs_packed* w, int n, const CallShape& c, int sms, std::vector<Plan>& out)
{
    out.push_back(tc_plan_on(w, n, c, sms, 0));
    if (!tc16_ok(w, c)) return;
    std::vector<int> px;
    for (int want : {kAnyPixels, alcs::kTc16Pixels, alcs::kTc16Pixels / 2, alcs::kTc16Pixels / 4}) {
        Plan p = tc_plan_on(w, n, c, sms, want);
        p.tc_named = true;
        if (std::find(px.begin(), px.end(), p.tc_px) != px.end()) continue;
        px.push_back(p.tc_px);
        out.push_back(p);
    }
}

// Channels per tile worth considering: the equal split of cout into as many tiles as each multiple of 16 asks for.
int tc_widths(const alcs_packed* w, int (&n)[8])
{
    int count = 0;
    for (int want = alcs::kTcMaxN; want >= 16; want -= 16) {
        const int tiles = (w->cout + want - 1) / want, v = ((w->cout + tiles - 1) / tiles + 15) / 16 * 16;
        if (!count || v != n[count - 1]) n[count++] = v;
    }
    return count;
}

// What the planner's own choice among the staged kernels takes, in microseconds, without listing their configurations
// (which takes up to some tenths of a second): the repacking pass, then the longer of the bytes and the arithmetic, the
// latency of a work item's chunks and of its longest row.  Fits to 990 launches of random shapes, types and densities on
// one B200: median errors of 15 to 19 %.
double staged_us(const alcs_packed* w, const CallShape& c, int sms)
{
    struct Fit { double launch, pass, pass_rate, rate, px, row, x, chunk, longest, block[5]; };
    static const Fit fits[3] = {      // fp32; 16 bits on the CUDA cores; fp16 on mma.sync
        {4.81, 1.42, 10.0e6, 2.48e6, 0.0120, 34.0e-6, 0.89e-6, 0.90, 0.045, {20.8e-6, 24.0e-6, 28.3e-6, 48.5e-6, 113e-6}},
        {7.06, 0.43, 4.73e6, 2.00e6, 0.0031, 256e-6, 17.2e-6, 0.85, 0.0355, {25.1e-6, 35.0e-6, 55.7e-6, 65.7e-6, 163e-6}},
        {7.25, 0.0, 4.89e6, 3.07e6, 0.0, 0.0, 185e-6, 0.40, 0.0045, {14.0e-6, 14.0e-6, 14.0e-6, 19.3e-6, 47.4e-6}}};
    const Fit& f = fits[w->dt == ALCS_F32 ? 0 : w->dt == ALCS_F16 && w->g >= 4 ? 2 : 1];
    const double q = (double)c.q(), elt = (double)w->elt(), x_bytes = q * w->cin * elt;
    const size_t row = (size_t)c.hw() * w->elt();
    double us = f.launch + f.chunk * w->cin / 64.0 + f.longest * longest_row(w);
    // (the pass over a strided input reads single elements)
    if (c.stride > 1 || (row % 16 != 0 && row % 16 != 8)) us += f.pass + x_bytes * (1 + c.stride) / (c.stride > 1 ? std::min(f.pass_rate, 4.0e6) : f.pass_rate);
    const int at = w->g == 1 ? 0 : w->g == 2 ? 1 : w->g == 4 ? 2 : w->g == 8 ? 3 : 4;
    const double work = q * f.px + w->nb * q * f.block[at] + w->rows * q * f.row + x_bytes * f.x * std::max(1.0, w->rows / 32.0);
    us += std::max(work / sms, (x_bytes + q * w->cout * elt) / f.rate);
    if (c.residual) us += q * w->cout * (w->dt == ALCS_F32 ? 3.2e-6 : 2.0e-6);
    return us;
}

// Can the producers stage the rows of X as they are, with 8-byte copies, where 16-byte copies would need
// the rows repacked?
bool direct_rows_ok(int hw, int elt) { return ((size_t)hw * elt) % 16 == 8; }

// How many of the best candidates the tuner times a second time and remembers for alcs_stack_tune.
constexpr size_t kFinalists = 12;

// Schedules a first call builds to choose among: about a millisecond's worth, and at least three.
size_t quick_schedules(const alcs_packed* w) { return (size_t)std::max(3, std::min(24, 500000 / std::max(1, w->nb))); }

// The sizes of a schedule without building it, for rows of equal length: a segment (block row, chunk) of `len` blocks takes
// about len / 2 + 1/4 pair records, or len / 16 + 1/2 step records.
Schedule guess_schedule(const alcs_packed* w, const KernelVariant& v, int kc, int n_rg)
{
    Schedule s;
    const int cap = v.nw / v.groups * v.rw;
    s.kc = kc;
    s.nch = (w->cin + kc - 1) / kc;
    s.n_rg = v.mma ? std::max(1, std::min(n_rg, w->rows)) : std::max(std::max(1, (w->rows + cap - 1) / cap), std::min(n_rg, w->rows));
    s.rpg = v.mma ? (w->rows + s.n_rg - 1) / s.n_rg : cap;
    s.ros = 4 * s.rpg;
    const double segments = (double)w->rows * s.nch, len = w->nb / segments, per = v.mma ? 16.0 : 2.0;
    const double records = segments * std::min(len, len / per + 0.5 * (1.0 - 1.0 / per));
    s.n_rec = (int)(records * (v.mma ? alcs::step_record_bytes(v.g) : alcs::record_bytes(v.g)) / 16.0);
    s.wcap = (int)(1.2 * s.n_rec / ((double)s.n_rg * s.nch)) + 16;
    return s;
}

// Internal bits of the flags in plan-cache keys, which else hold the output size alone: kExtra says that the call has a
// residual operand or a stride (which the small-problem kernel does not take), the others which, and how its input
// rows can be copied.
constexpr unsigned kExtra = 0x10000u, kResidual = 0x20000u, kStrideShift = 20, kRowShift = 24, kNoTc = 0x80000000u;

unsigned key_flags(const alcs_packed* w, unsigned flags, const CallShape& c)
{
    if (c.stride == 1 && !c.residual) return flags;
    const size_t row = (size_t)c.wd * w->elt();
    const unsigned align = c.stride == 1 ? 0 : row % 16 == 0 ? 2 : row % 8 == 0 ? 1 : 0;
    return flags | kExtra | (c.residual ? kResidual : 0u) | (unsigned)std::min(c.stride, 15) << kStrideShift | align << kRowShift | (tc_ok(w, c) ? 0u : kNoTc);
}

// Enumerate every valid launch configuration for this shape, cheapest (by the model) first.
// quick: the kernels that stage X through shared memory alone, ranked by guessed schedules; the first few are then built and
// the best of those is put in front.  For a first call, which cannot wait for all schedules to be built (a second or
// more for a 2048 x 2048 layer).
int enumerate_plans(const alcs_packed* w, const CallShape& c, std::vector<Plan>& out, bool quick = false)
{
    const long long q = std::max(1ll, c.q());
    const int hw = c.hw();
    DeviceInfo di;
    int rc = device_info(w->device, &di);
    if (rc) return rc;
    {
        std::lock_guard<std::mutex> lk(g_mu);
        init_variants_locked();
    }
    const int elt = (int)w->elt();
    const int smem_max = std::min(kMaxSmem, di.smem_optin);
    out.clear();
    for (size_t vi = 0; vi < g_variants.size(); ++vi) {
        const KernelVariant& v = g_variants[vi].v;
        if (v.is_f16 != (int)w->dt || v.g != w->g || (quick && v.split)) continue;
        rc = prepare_variant(g_variants[vi], w->device);
        if (rc) return rc;
        const int cap = v.nw / v.groups * v.rw;
        const int rg_min = (w->rows + cap - 1) / cap;
        int last_kc = -1;
        for (int ci = 0; ci < alcs::kNumChunkings; ++ci) {
            int kc = alcs::kChunkings[ci];
            if (kc == 0 || kc > w->cin) kc = w->cin;
            if (kc == last_kc) continue;
            last_kc = kc;
            if ((size_t)kc * 32 * v.p * elt * 2 > (size_t)smem_max) continue;
            if (!v.mma && kc >= alcs::kMaxBalancedKc) continue;
            int last_rpg = -1;
            // Row-group counts to consider: every count up to a few times the minimum, and, when
            // the pixel tiles alone are too few to occupy the GPU (small batches), a geometric
            // ladder of larger counts up to about two work items per SM.
            const long long tiles = (q + 32 * v.p - 1) / (32 * v.p);
            const int rg_dense = std::min(w->rows, rg_min * 4 + 2);
            const int rg_hi = std::max<long long>(rg_dense, std::min<long long>(w->rows, (2ll * di.sms + tiles - 1) / tiles));
            for (int n_rg = rg_min; n_rg <= rg_hi; n_rg = n_rg < rg_dense && !quick ? n_rg + 1 : std::max(n_rg + 1, n_rg * 5 / 4)) {
                const int rpg = (w->rows + n_rg - 1) / n_rg;
                if (rpg == last_rpg || rpg > cap) continue;
                last_rpg = rpg;
                const Schedule guess = quick ? guess_schedule(w, v, kc, n_rg) : Schedule();
                const Schedule* sc = quick ? &guess : get_schedule(w, kc, n_rg, false, flavour_of(v));
                if (!sc) return ALCS_ERR_ALLOC;
                if (v.split && sc->max_x == 0) continue;        // nothing to split: the plain variant covers it
                const StageLayout L = stage_layout(v, *sc, elt);
                for (int stages = 2; stages <= alcs::kMaxStages; ++stages) {
                    if (stages % v.groups) continue;        // every consumer group gets the same share of the ring
                    const size_t smem = plan_smem(L, stages);
                    if (smem > (size_t)smem_max) break;
                    const int occ = occupancy_of(g_variants[vi], smem);
                    if (occ < 1) continue;
                    Plan p;
                    p.variant = (int)vi; p.kc = sc->kc; p.n_rg = sc->n_rg; p.stages = stages;
                    p.occ = occ; p.smem = smem;
                    p.cost = model_cost(w, v, *sc, q, di, occ);
                    // deeper rings only help while there are chunks to prefetch; prefer the shallowest
                    p.cost *= 1.0 + 0.01 * stages;
                    // Bulk copies pay a fixed cost per copy, so they win when a tile row is one long
                    // run (images at least as large as the tile) and lose when it is cut into pieces.
                    const bool rows_aligned = true;     // unaligned rows are repacked to aligned ones
                    p.bulk = hw >= 32 * v.p ? 1 : 0;
                    out.push_back(p);
                    if (rows_aligned) {
                        Plan p2 = p;
                        p2.bulk = 1 - p.bulk;
                        p2.cost *= 1.25;
                        out.push_back(p2);
                    }
                    // Rows that are a multiple of 8 but not of 16 bytes long (16-bit 14x14 images) can also be
                    // staged as they are, with 8-byte copies: twice the copy instructions, no repacking pass.
                    if (direct_rows_ok(hw, elt)) {
                        Plan p3 = p;
                        p3.bulk = 2;
                        p3.cost *= 1.1;
                        out.push_back(p3);
                    }
                    // A tile-major copy of X first (one more pass over X where its rows need no repacking
                    // anyway), then a chunk is staged by a few large bulk copies: no copy instructions to
                    // speak of, so one producer warp is enough.
                    if (v.npw <= 2 && q > 8ll * hw) {
                        Plan p4 = p;
                        p4.bulk = 3;
                        const double pass = 2.0 * (double)q * w->cin * elt / di.hbm_bps + 3e-6;
                        p4.cost = p.cost * 0.9 + ((((size_t)hw * elt) % 16 == 0) ? pass : 0.0);
                        out.push_back(p4);
                    }
                }
            }
        }
    }
    if (!quick && tc_ok(w, c)) {
        int n[8];
        const int count = tc_widths(w, n);
        for (int i = 0; i < count; ++i) tc_plans(w, n[i], c, di.sms, out);
    }
    if (!quick && c.stride == 1 && !c.residual && hw > 0 && c.images() <= kGatherImages) {        // small batches only: one thread block per (block row, image, pixel tile)
        for (int p = 8; p >= 2; p /= 2)
            for (int ks = 4; ks <= 16; ks *= 2) {
                Plan g;
                if (gather_plan(w, c.images(), hw, p, ks, di, &g)) out.push_back(g);
            }
    }
    std::stable_sort(out.begin(), out.end(), [](const Plan& a, const Plan& b) { return a.cost < b.cost; });
    if (quick && !out.empty()) {
        Plan best;
        best.cost = 1e30;
        std::vector<std::array<int, 3>> built;
        for (const Plan& guess : out) {
            const std::array<int, 3> key = {guess.variant, guess.kc, guess.n_rg};
            if (std::find(built.begin(), built.end(), key) != built.end()) continue;
            if (built.size() >= quick_schedules(w) && best.cost < 1e30) break;
            built.push_back(key);
            const KernelVariant& v = g_variants[guess.variant].v;
            const Schedule* sc = get_schedule(w, guess.kc, guess.n_rg, false, flavour_of(v));
            if (!sc) return ALCS_ERR_ALLOC;
            Plan p = guess;
            p.n_rg = sc->n_rg;
            p.smem = plan_smem(stage_layout(v, *sc, elt), p.stages);
            if (p.smem > (size_t)smem_max || (p.occ = occupancy_of(g_variants[p.variant], p.smem)) < 1) continue;
            p.cost = guess.cost * model_cost(w, v, *sc, q, di, p.occ) / model_cost(w, v, guess_schedule(w, v, guess.kc, guess.n_rg), q, di, guess.occ);
            if (p.cost < best.cost) best = p;
        }
        if (best.cost >= 1e30) return ALCS_ERR_UNSUPPORTED;
        out.assign(1, best);
    }
    return out.empty() ? ALCS_ERR_UNSUPPORTED : ALCS_OK;
}

// The staged kernels' plan for a call without a configuration: of the quick list, or, should no guessed schedule have fitted
// shared memory, of the full one.
int staged_best(const alcs_packed* w, const CallShape& c, Plan* out)
{
    std::vector<Plan> list;
    int rc = enumerate_plans(w, c, list, true);
    if (rc == ALCS_ERR_UNSUPPORTED) rc = enumerate_plans(w, c, list);
    if (rc) return rc;
    for (const Plan& p : list)
        if (!p.tc_n && !p.gather) { *out = p; return ALCS_OK; }
    return ALCS_ERR_UNSUPPORTED;
}

void plan_to_cfg(const alcs_packed* w, const CallShape& shape, const Plan& p, alcs_launch_cfg* c)
{
    if (p.gather) {
        std::memset(c, 0, sizeof *c);
        c->pixels_per_lane = p.gp;
        c->warps = p.gks;
        c->math_mode = 3;
        return;
    }
    if (p.tc_n) {
        std::memset(c, 0, sizeof *c);
        c->pixels_per_lane = 1;
        c->warps = p.tc_px / 32;
        c->math_mode = 4;
        c->row_groups = p.n_rg;
        c->producer_warps = p.tc_px ? kTc16Producers : tc16_ok(w, shape) ? kTcProducers : 0;
        return;
    }
    const KernelVariant& v = g_variants[p.variant].v;
    c->pixels_per_lane = v.p;
    c->rows_per_warp = v.rw;
    c->warps = v.nw;
    c->chunk_channels = p.kc;
    c->stages = p.stages;
    c->row_groups = p.n_rg;
    c->min_blocks = v.minb;
    c->copy_mode = p.bulk + 1;
    c->producer_warps = v.npw;
    c->math_mode = mode_of(v);
    c->consumer_groups = v.groups;
    c->split_rows = v.split ? 1 : 2;
}

// Resolve a (possibly partial) configuration into a concrete plan.
int cfg_to_plan(const alcs_packed* w, const CallShape& shape, const alcs_launch_cfg* c, Plan* out)
{
    DeviceInfo di;
    int rc = device_info(w->device, &di);
    if (rc) return rc;
    const bool allow_small = shape.stride == 1 && !shape.residual;
    const int hw = shape.hw();
    const bool tc = (!c || c->math_mode == 4) && tc_ok(w, shape);
    if (c && c->math_mode == 4) {       // the tcgen05 kernel as asked for: row_groups channel tiles
        if (!tc) return ALCS_ERR_UNSUPPORTED;
        int n[8], count = tc_widths(w, n);
        if (c->row_groups) {
            const int tiles = std::max(1, c->row_groups);
            n[0] = ((w->cout + tiles - 1) / tiles + 15) / 16 * 16;
            count = 1;
            if (n[0] > alcs::kTcMaxN) return ALCS_ERR_UNSUPPORTED;
        }
        const int named = tc16_ok(w, shape) ? c->producer_warps : 0;       // (the others have one kernel)
        if (named != kTcProducers && named != kTc16Producers) {
            *out = tc_best(w, n, count, shape, di.sms);
            return ALCS_OK;
        }
        const int pixels = named == kTcProducers ? 0 : c->warps > 0 ? 32 * std::min(c->warps, alcs::kTc16Pixels / 32) : kAnyPixels;
        for (int i = 0; i < count; ++i) {
            const Plan p = tc_plan_on(w, n[i], shape, di.sms, pixels);
            if (!i || p.cost < out->cost) *out = p;
        }
        out->tc_named = true;
        return ALCS_OK;
    }
    if (!c) {
        // Nobody asked for anything: the tcgen05 kernel; the small-problem kernel where a few images leave most SMs without a
        // tile and the latency of one item's chunk chain is all there is; or the staged kernels, whose time falls with the
        // density where the dense tiles' does not, if they are expected to be clearly faster.  Their estimate is the
        // rougher one, most of all for long calls (512 -> 512 at 14 x 14, batch 256, 10 % kept: 252 us where 100 were
        // expected, 120 dense), so those have to promise more.  2048 -> 2048 at 7 x 7, batch 32, 5 % kept: 92 us dense, 49.
        Plan best;
        double against = best.cost = 1e30;
        if (tc) {
            const alcs::TcForms forms = alcs::tc_forms(w);
            int n[8], count = 0;
            for (int i = 0, all = tc_widths(w, n); i < all; ++i)
                if (alcs::tc_form_free(w, forms, {n[i], 0, 0})) n[count++] = n[i];
            if (count) best = tc_best(w, n, count, shape, di.sms, &against);
        }
        if (allow_small && hw > 0 && shape.images() <= kGatherImages)
            for (int p = 8; p >= 2; p /= 2)
                for (int ks = 4; ks <= 16; ks *= 2) {
                    Plan g;
                    if (gather_plan(w, shape.images(), hw, p, ks, di, &g) && g.cost < best.cost) {
                        best = g;
                        against = g.cost;
                    }
                }
        const double staged = 1e-6 * staged_us(w, shape, di.sms);
        if (staged * (against < 100e-6 ? 1.15 : 1.5) < against) {
            Plan p;
            rc = staged_best(w, shape, &p);
            if (rc && (rc != ALCS_ERR_UNSUPPORTED || best.cost >= 1e30)) return rc;
            if (!rc) {
                best = p;
                best.cost = staged;
            }
        }
        *out = best;
        return ALCS_OK;
    }
    std::vector<Plan> all;
    rc = enumerate_plans(w, shape, all);
    if (rc) return rc;
    if (c->math_mode == 3 && !allow_small) return ALCS_ERR_UNSUPPORTED;
    if (c->math_mode == 3) {        // the small-problem kernel, with the given (or the best-ranked) shape
        for (const Plan& p : all)
            if (p.gather && (!c->pixels_per_lane || c->pixels_per_lane == p.gp) && (!c->warps || c->warps == p.gks)) {
                *out = p;
                return ALCS_OK;
            }
        if (hw > 0 && c->pixels_per_lane && c->warps &&
            gather_plan(w, shape.images(), hw, c->pixels_per_lane, c->warps, di, out)) return ALCS_OK;
        return ALCS_ERR_UNSUPPORTED;
    }
    auto variant_ok = [&](const Plan& p) {
        if (p.gather || p.tc_n) return false;
        const KernelVariant& v = g_variants[p.variant].v;
        if (c->pixels_per_lane && c->pixels_per_lane != v.p) return false;
        if (c->rows_per_warp && c->rows_per_warp != v.rw) return false;
        if (c->warps && c->warps != v.nw) return false;
        if (c->min_blocks && c->min_blocks != v.minb) return false;
        if (c->producer_warps && c->producer_warps != v.npw) return false;
        if (c->math_mode && c->math_mode != mode_of(v)) return false;
        if (c->consumer_groups && c->consumer_groups != v.groups) return false;
        if (c->split_rows && (c->split_rows == 1) != (v.split == 1)) return false;
        if (c->chunk_channels && std::min(c->chunk_channels, w->cin) != p.kc) return false;
        if (c->stages && c->stages != p.stages) return false;
        if (c->copy_mode) {     // (3 where the rows cannot be staged as they are: like 1)
            const int want = (c->copy_mode == 3 && !direct_rows_ok(hw, (int)w->elt())) ? 1 : c->copy_mode;
            if (want != p.bulk + 1) return false;
        }
        return true;
    };
    for (const Plan& p : all)
        if (variant_ok(p) && (!c->row_groups || c->row_groups == p.n_rg)) { *out = p; return ALCS_OK; }
    // a row-group count outside the enumerated range: accept it for a matching variant if it fits
    if (c->row_groups > 0 && c->row_groups <= w->rows) {
        for (const Plan& p0 : all) {
            if (!variant_ok(p0)) continue;
            const KernelVariant& v = g_variants[p0.variant].v;
            const int rpg = (w->rows + c->row_groups - 1) / c->row_groups;
            if (rpg > v.nw / v.groups * v.rw) continue;
            const Schedule* sc = get_schedule(w, p0.kc, c->row_groups, false, flavour_of(v));
            if (!sc) return ALCS_ERR_ALLOC;
            if (v.split && sc->max_x == 0) continue;        // nothing to split with this many row groups
            Plan p = p0;
            p.n_rg = sc->n_rg;
            p.smem = plan_smem(stage_layout(v, *sc, (int)w->elt()), p.stages);
            if (p.smem > (size_t)std::min(kMaxSmem, di.smem_optin)) continue;
            p.occ = occupancy_of(g_variants[p.variant], p.smem);
            if (p.occ < 1) continue;
            *out = p;
            return ALCS_OK;
        }
    }
    return ALCS_ERR_UNSUPPORTED;
}

// X whose (image, channel) rows are not a multiple of 16 bytes long (H*W = 49, ...) cannot be staged
// with 16-byte copies, and a strided pointwise convolution reads only every stride-th pixel of every
// stride-th row.  Such inputs are first gathered into scratch memory: the pixels the convolution
// reads, row after row, every (image, channel) row padded with zeros to the next multiple of 16
// bytes; the main kernel then runs on the padded pixel axis and simply does not store the padding
// pixels.  Each thread writes one 16-byte piece of a padded row (EPV elements), reading its elements
// one by one: the source rows start at arbitrary element offsets.
// rows = n*cin; hw_in = elements per source row; output pixel p of a row is source pixel
// (p / ow) * stride * wd_in + (p % ow) * stride; hw_out real and hwp padded pixels per output row.
template <typename T>
__global__ void repack_rows_kernel(const T* __restrict__ in, T* __restrict__ out, long long rows, int hw_in, int wd_in,
                                   int ow, int stride, int hw_out, int hwp)
{
    constexpr int EPV = 16 / (int)sizeof(T);
    // The convolution kernel behind this one on the stream may set up (barriers, schedule bounds) while
    // the copy runs; it waits for this grid to finish before it touches the scratch.
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int vpr = hwp / EPV;                       // 16-byte pieces per padded row
    const long long total = rows * vpr;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total;
         i += (long long)gridDim.x * blockDim.x) {
        const long long r = i / vpr;
        const int p0 = (int)(i - r * vpr) * EPV;
        const T* src = in + r * hw_in;
        alignas(16) T v[EPV];
        if (stride == 1) {
#pragma unroll
            for (int t = 0; t < EPV; ++t) v[t] = p0 + t < hw_out ? __ldg(src + p0 + t) : T(0);
        } else {
#pragma unroll
            for (int t = 0; t < EPV; ++t) {
                const int p = p0 + t;
                const int oy = p / ow, ox = p - oy * ow;
                v[t] = p < hw_out ? __ldg(src + (size_t)oy * stride * wd_in + (size_t)ox * stride) : T(0);
            }
        }
        *reinterpret_cast<uint4*>(out + r * hwp + p0) = *reinterpret_cast<const uint4*>(v);
    }
}

// The same copy into a TILE-MAJOR layout: out[tile][channel][tile_px pixels (+ padding up to rowb elements)],
// where pixel q = image * hwp + p of the padded pixel axis lies in tile q / tile_px.  A work item of the
// convolution kernel then finds the channel rows of its tile one after the other and stages a whole chunk
// of them with a few large bulk copies.  Pixels beyond the last image are written as zeros.
template <typename T>
__global__ void repack_tiles_kernel(const T* __restrict__ in, T* __restrict__ out, int n, int cin, int hw_in, int wd_in,
                                    int ow, int stride, int hw_out, int hwp, int tile_px, int rowb, long long n_tiles)
{
    constexpr int EPV = 16 / (int)sizeof(T);
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int vpr = tile_px / EPV;                   // 16-byte pieces per (tile, channel) row
    const long long total = n_tiles * cin * vpr;
    const long long q_total = (long long)n * hwp;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total;
         i += (long long)gridDim.x * blockDim.x) {
        const long long row = i / vpr;
        const int piece = (int)(i - row * vpr);
        const long long tile = row / cin;
        const int c = (int)(row - tile * cin);
        const long long q = tile * tile_px + (long long)piece * EPV;
        alignas(16) T v[EPV];
        if (q < q_total) {
            const long long img = q / hwp;
            const int p0 = (int)(q - img * hwp);      // (hwp is a multiple of EPV: the piece lies in one image)
            const T* src = in + ((size_t)img * cin + c) * hw_in;
#pragma unroll
            for (int t = 0; t < EPV; ++t) {
                const int p = p0 + t;
                if (p >= hw_out) { v[t] = T(0); continue; }
                if (stride == 1) {
                    v[t] = __ldg(src + p);
                } else {
                    const int oy = p / ow, ox = p - oy * ow;
                    v[t] = __ldg(src + (size_t)oy * stride * wd_in + (size_t)ox * stride);
                }
            }
        } else {
#pragma unroll
            for (int t = 0; t < EPV; ++t) v[t] = T(0);
        }
        *reinterpret_cast<uint4*>(out + (size_t)row * rowb + (size_t)piece * EPV) = *reinterpret_cast<const uint4*>(v);
    }
}

// pixels per image after padding the rows of X to a multiple of 16 bytes
int padded_hw(int hw, int elt) { const int m = 16 / elt; return (hw + m - 1) / m * m; }

// Bytes per channel row of a pixel tile in shared memory and in the tile-major copy of X.
int tile_row_bytes(const KernelVariant& v, int elt) { return 32 * v.p * elt + (v.mma ? 16 : 0); }

// Bytes of the tile-major copy of X for kernel variant v: n images of hw pixels (rows padded to 16 bytes).
size_t tiled_bytes(const KernelVariant& v, int elt, int n, int cin, int hw)
{
    const long long q = (long long)n * padded_hw(hw, elt);
    const long long tiles = (q + 32 * v.p - 1) / (32 * v.p);
    return (size_t)tiles * cin * tile_row_bytes(v, elt);
}

int launch_repack_tiles(const KernelVariant& v, int elt, const void* x, void* out, int n, int cin, int h_in, int wd_in,
                        int ow, int stride, int hw, int sms, cudaStream_t st)
{
    const int hwp = padded_hw(hw, elt);
    const int T = 32 * v.p;
    const long long tiles = ((long long)n * hwp + T - 1) / T;
    const long long pieces = tiles * cin * (T * elt / 16);
    const unsigned blocks = (unsigned)std::min<long long>((pieces + 255) / 256, (long long)sms * 8);
    const int rowb = tile_row_bytes(v, elt) / elt;
    if (elt == 4)
        repack_tiles_kernel<float><<<blocks, 256, 0, st>>>(static_cast<const float*>(x), static_cast<float*>(out), n, cin,
                                                          h_in * wd_in, wd_in, ow, stride, hw, hwp, T, rowb, tiles);
    else
        repack_tiles_kernel<unsigned short><<<blocks, 256, 0, st>>>(static_cast<const unsigned short*>(x),
                                                                   static_cast<unsigned short*>(out), n, cin, h_in * wd_in,
                                                                   wd_in, ow, stride, hw, hwp, T, rowb, tiles);
    ALCS_CUDA(cudaGetLastError());
    return ALCS_OK;
}

// Make sure the scratch of w can hold `bytes`.  Growing it frees the old block, which waits for
// all earlier work on the device.
int ensure_xpad(const alcs_packed* w, size_t bytes)
{
    std::lock_guard<std::mutex> lk(w->mu);
    if (w->xpad_bytes >= bytes) return ALCS_OK;
    if (w->d_xpad) cudaFree(w->d_xpad);
    w->d_xpad = nullptr;
    w->xpad_bytes = 0;
    cudaError_t e = cudaMalloc(&w->d_xpad, bytes);
    if (e != cudaSuccess) {
        alcs::set_cuda_error_text(cudaGetErrorString(e));
        (void)cudaGetLastError();
        return ALCS_ERR_ALLOC;
    }
    w->xpad_bytes = bytes;
    return ALCS_OK;
}

int check_conv_args(const alcs_packed* w, const void* x, const void* y, int n, int h, int wd,
                    unsigned flags, long long* q_out)
{
    if (!w) return ALCS_ERR_INVALID_ARG;
    if (n < 0 || h < 0 || wd < 0) return ALCS_ERR_INVALID_ARG;
    if (flags & ~(ALCS_RELU | ALCS_Y_F32)) return ALCS_ERR_INVALID_ARG;
    if ((flags & ALCS_Y_F32) && w->dt == ALCS_F32) return ALCS_ERR_INVALID_ARG;
    if (w->g != 1 && w->g != 2 && w->g != 4 && w->g != 8 && w->g != 16) return ALCS_ERR_UNSUPPORTED;
    const long long hw = (long long)h * wd;
    const long long q = hw * n;
    if (hw > (1ll << 30) || q > (1ll << 30)) return ALCS_ERR_SHAPE;
    *q_out = q;
    if (q == 0) return ALCS_OK;
    if (!x || !y) return ALCS_ERR_INVALID_ARG;
    const size_t xe = w->elt(), ye = (w->dt != ALCS_F32 && !(flags & ALCS_Y_F32)) ? 2 : 4;
    if ((uintptr_t)x % xe || (uintptr_t)y % ye) return ALCS_ERR_INVALID_ARG;
    const uintptr_t xb = (uintptr_t)x, xend = xb + (size_t)q * w->cin * xe;
    const uintptr_t yb = (uintptr_t)y, yend = yb + (size_t)q * w->cout * ye;
    if (xb < yend && yb < xend) return ALCS_ERR_INVALID_ARG;   // x and y overlap
    return ALCS_OK;
}

// Device copy of the canonical storage format (row_ptr, col_idx, vals) for the small-problem kernel:
// made the first time that kernel is used with w (allocates, and waits for the copy), kept until w is freed.
int ensure_canonical_on_device(const alcs_packed* w, cudaStream_t st)
{
    std::lock_guard<std::mutex> lk(w->mu);
    if (w->d_row_ptr) return ALCS_OK;
    // one block for the three arrays: an allocation costs more than the copies
    auto up = [](size_t b) { return (b + 255) / 256 * 256; };
    const size_t o_col = up(w->row_ptr.size() * 4), o_val = o_col + up(w->col_idx.size() * 4);
    unsigned char* base = nullptr;
    cudaError_t e = cudaMalloc(&base, o_val + std::max<size_t>(w->vals.size(), 16));
    if (e == cudaSuccess) e = cudaMemcpyAsync(base, w->row_ptr.data(), w->row_ptr.size() * 4, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess && !w->col_idx.empty())
        e = cudaMemcpyAsync(base + o_col, w->col_idx.data(), w->col_idx.size() * 4, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess && !w->vals.empty()) e = cudaMemcpyAsync(base + o_val, w->vals.data(), w->vals.size(), cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) {
        alcs::set_cuda_error_text(cudaGetErrorString(e));
        cudaFree(base);
        (void)cudaGetLastError();
        return e == cudaErrorMemoryAllocation ? ALCS_ERR_ALLOC : ALCS_ERR_CUDA;
    }
    int32_t* const rp = reinterpret_cast<int32_t*>(base);
    int32_t* const ci = reinterpret_cast<int32_t*>(base + o_col);
    void* const va = base + o_val;
    w->d_col_idx = ci; w->d_vals = va;
    w->d_row_ptr = rp;
    return ALCS_OK;
}

// Launch the small-problem kernel; the canonical arrays must be on the device.
int launch_gather_plan(const alcs_packed* w, const Plan& p, const void* x, void* y, int n, int h, int wd,
                       const float* bias, unsigned flags, cudaStream_t st)
{
    alcs::GatherArgs a;
    a.x = static_cast<const float*>(x); a.y = static_cast<float*>(y); a.bias = bias;
    a.row_ptr = w->d_row_ptr; a.col_idx = w->d_col_idx; a.vals = static_cast<const float*>(w->d_vals);
    a.rows = w->rows; a.cin = w->cin; a.cout = w->cout; a.hw = h * wd; a.n = n;
    a.tiles = (a.hw + 32 * p.gp - 1) / (32 * p.gp);
    a.relu = (flags & ALCS_RELU) ? 1 : 0;
    a.vec = (p.gp >= 4 && a.hw % 4 == 0 && (uintptr_t)x % 16 == 0) ? 1 : 0;
    const int longest = longest_row(w);
    a.stage_blocks = alcs::gather_stage_blocks(w->g, longest);
    ALCS_CUDA(alcs::launch_gather(w->g, p.gp, p.gks, a, st));
    return ALCS_OK;
}

// Which form of the expanded weights a problem takes: strided layers, and small images that are staged as runs of
// all columns, cannot use a tile's column list.
alcs::TcKey tc_key(const alcs_packed* w, const Plan& p, const alcs::TcProblem& pr)
{
    const int k = pr.kh || alcs::tc_whole_images(w, pr) ? 1 : 0;
    return {p.tc_n, k, k};
}

// Pixels per tile on alcs_tc16.cu (0: alcs_tc.cu) for a call with the X of `pr`.  A plan is made for rows that can be copied as they
// are, where their length allows it; where X starts elsewhere they have to be picked apart, which the other kernel, whose
// expanded weights are the same, is mostly the better one at: 80 layers with X on an odd multiple of 2 or 4 bytes, up to 6.2 times as
// fast; by the rule for odd rows (tc_best) 14 of 55 stay here and none is slower than there.
int tc_pixels(const alcs_packed* w, const Plan& p, const alcs::TcProblem& pr)
{
    if (!p.tc_px || p.tc_named || (size_t)pr.oh * pr.ow * w->elt() % 8 != 0 || alcs::tc16_direct(w, pr)) return p.tc_px;
    DeviceInfo di;
    int px;
    if (device_info(w->device, &di)) return 0;
    return alcs::tc16_layer_us(w, pr, p.tc_n, di.sms, 0, &px) * kRawMargin < alcs::tc_layer_us(w, pr, p.tc_n, di.sms) ? px : 0;
}

// Launch the tcgen05 kernel for one layer; strided layers run by patch staging.
int launch_tc_plan(const alcs_packed* w, const Plan& p, alcs::TcProblem pr, cudaStream_t st)
{
    pr.pixels = tc_pixels(w, p, pr);
    alcs::TcForm t;
    const int rc = alcs::tc_prepare(w, tc_key(w, p, pr), st, &t);
    return rc ? rc : alcs::tc_run(w, *t, pr, st);
}

// scratch / scratch_bytes: where X is repacked when its rows are not 16-byte multiples.  nullptr means
// the scratch that w owns (allocated or grown here); a layer stack passes its own, fixed for the
// stack's lifetime, so that a captured graph never refers to memory a later call may free.
// residual (may be null): same shape and element type as y, added before the activation.  stride > 1:
// h and wd are the OUTPUT size, h_in x wd_in the input size, and the pixels the convolution reads
// are gathered into the scratch first.
int launch_plan(const alcs_packed* w, const Plan& p, const void* x, void* y, int n, int h, int wd,
                const float* bias, unsigned flags, cudaStream_t st, void* scratch = nullptr, size_t scratch_bytes = 0,
                const void* residual = nullptr, int stride = 1, int h_in = 0, int wd_in = 0)
{
    if (stride <= 1) { stride = 1; h_in = h; wd_in = wd; }
    if (p.gather) {
        if (residual || stride != 1) return ALCS_ERR_STATE;        // (plans for such calls never list that kernel)
        const int rc = ensure_canonical_on_device(w, st);
        return rc ? rc : launch_gather_plan(w, p, x, y, n, h, wd, bias, flags, st);
    }
    if (p.tc_n) return launch_tc_plan(w, p, tc_problem(x, y, n, h, wd, bias, flags, residual, stride, h_in, wd_in), st);
    const KernelVariant& v = g_variants[p.variant].v;
    Schedule* sc = get_schedule(w, p.kc, p.n_rg, true, flavour_of(v));
    if (!sc) return ALCS_ERR_ALLOC;
    if (v.split && sc->max_x == 0) return ALCS_ERR_UNSUPPORTED;    // (the split flavour needs its hand-over area)
    if (!sc->uploaded) {
        const int rc = upload_schedule(w, sc, st);
        if (rc) return rc;
    }
    DeviceInfo di;
    int rc = device_info(w->device, &di);
    if (rc) return rc;
    const int elt = (int)w->elt();
    const int hw = h * wd;
    // Rows of X that are not a multiple of 16 bytes long: repack X into scratch with padded rows.
    int hwx = hw;
    const void* xk = x;
    const bool direct = p.bulk == 2 && stride == 1 && direct_rows_ok(hw, elt) && (uintptr_t)x % 8 == 0;
    bool tiled = false;
    if (p.bulk == 3 && (long long)n * padded_hw(hw, elt) <= (1ll << 30)) {
        // tile-major copy of X (also gathers the pixels a strided convolution reads)
        const size_t need = tiled_bytes(v, elt, n, w->cin, hw);
        if (scratch ? scratch_bytes >= need : ensure_xpad(w, need) == ALCS_OK) {
            void* const xt = scratch ? scratch : w->d_xpad;
            rc = launch_repack_tiles(v, elt, x, xt, n, w->cin, h_in, wd_in, wd, stride, hw, di.sms, st);
            if (rc) return rc;
            xk = xt;
            hwx = padded_hw(hw, elt);
            tiled = true;
        }       // else: staged like copy mode 1
    }
    if (!tiled && ((((size_t)hw * elt) % 16 != 0 && !direct) || stride != 1)) {
        const int hwp = padded_hw(hw, elt);
        const size_t need = (size_t)n * w->cin * hwp * elt;
        if (scratch && scratch_bytes < need) return ALCS_ERR_STATE;
        const bool have = (long long)n * hwp <= (1ll << 30) && (scratch || ensure_xpad(w, need) == ALCS_OK);
        if (!have && stride != 1) return ALCS_ERR_ALLOC;         // a strided input cannot be staged in place
        if (have) {
            void* const xpad = scratch ? scratch : w->d_xpad;
            const long long rows = (long long)n * w->cin;
            const unsigned blocks = (unsigned)std::min<long long>((rows * (hwp * elt / 16) + 255) / 256, (long long)di.sms * 8);     // one wave of 256-thread blocks
            if (elt == 4)
                repack_rows_kernel<float><<<blocks, 256, 0, st>>>(static_cast<const float*>(x), static_cast<float*>(xpad), rows,
                                                                  h_in * wd_in, wd_in, wd, stride, hw, hwp);
            else
                repack_rows_kernel<unsigned short><<<blocks, 256, 0, st>>>(static_cast<const unsigned short*>(x),
                                                                          static_cast<unsigned short*>(xpad), rows,
                                                                          h_in * wd_in, wd_in, wd, stride, hw, hwp);
            ALCS_CUDA(cudaGetLastError());
            xk = xpad;
            hwx = hwp;
        }   // else: fall back to element-wise staging of the unpadded rows
    }
    ConvArgs a;
    a.x = xk; a.y = y; a.bias = bias; a.res = residual;
    a.rec = sc->rec; a.slice = sc->slice; a.rowoff = sc->rowoff; a.rowmap = sc->rowmap;
    set_unit_args(a, *sc, v.mma);
    a.err = w->d_err;
    a.rows = w->rows; a.cin = w->cin; a.cout = w->cout; a.hw = hwx; a.hwy = hw;
    a.q_total = n * hwx;
    const int T = 32 * v.p;
    a.n_tiles = (a.q_total + T - 1) / T;
    a.n_rg = sc->n_rg; a.rpg = sc->rpg;
    a.kc = sc->kc; a.nch = sc->nch; a.stages = p.stages;
    a.relu = (flags & ALCS_RELU) ? 1 : 0;
    a.y_f32 = (flags & ALCS_Y_F32) ? 1 : 0;
    const StageLayout L = stage_layout(v, *sc, elt);
    a.off_rec = L.off_rec; a.off_rowoff = L.off_rowoff; a.stage_bytes = L.stage_bytes;
    if (a.unit) a.off_xch = 16 * alcs::kMaxStages + a.stages * L.stage_bytes;
    // widest staging copy that every (image, channel) row start and length allows
    int ld = 16;
    while (ld > elt && (((size_t)hwx * elt) % ld || (uintptr_t)xk % ld)) ld >>= 1;
    a.ld_bytes = ld;
    a.bulk = tiled ? 2 : (ld == 16 && p.bulk == 1) ? 1 : 0;
    a.ros = sc->ros;
    const int vg = (v.p * elt >= 16) ? 16 / elt : v.p;
    a.st_vec = (hwx == hw && hw % vg == 0 && (uintptr_t)y % 16 == 0 && (uintptr_t)residual % 16 == 0) ? 1 : 0;
    a.st_grp = hwx % vg == 0 ? 1 : 0;
    // 16-bit rows of Y that do not all start on an 8-byte boundary (7x7 images): nothing wider than one
    // element can be stored, and the tensor-core kernel then lets consecutive lanes take consecutive pixels
    if (v.mma && !a.y_f32 && !a.st_vec && ((size_t)hw * elt) % 8 != 0) a.st_grp = 2;
    const long long items = (long long)a.n_tiles * a.n_rg;
    if (items > 0x7fffffffll) return ALCS_ERR_SHAPE;
    // persistent thread blocks: as many as can be resident, each walks items with that stride
    const long long grid = std::min<long long>(items, (long long)di.sms * std::max(1, p.occ));
    void* args[] = {&a};
    // programmatic dependent launch: this kernel's set-up may overlap the tail of the kernel before
    // it on the stream; it waits for that kernel before it reads X or writes Y
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3((unsigned)grid);
    lc.blockDim = dim3((v.nw + v.npw) * 32);
    lc.dynamicSmemBytes = p.smem;
    lc.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    lc.attrs = attr;
    lc.numAttrs = 1;
    ALCS_CUDA(cudaLaunchKernelExC(&lc, v.fn, args));
    return ALCS_OK;
}

int check_device(const alcs_packed* w)
{
    if (w->device < 0) return ALCS_ERR_STATE;
    int cur = -1;
    ALCS_CUDA(cudaGetDevice(&cur));
    return cur == w->device ? ALCS_OK : ALCS_ERR_STATE;
}

int resolve_plan(const alcs_packed* w, const CallShape& c, unsigned flags, const alcs_launch_cfg* cfg, Plan* plan)
{
    alcs::ShapeKey key{c.n, c.oh, c.ow, key_flags(w, flags, c)};
    if (cfg) {
        const int v[12] = {cfg->pixels_per_lane, cfg->rows_per_warp, cfg->warps, cfg->chunk_channels,
                           cfg->stages, cfg->row_groups, cfg->min_blocks, cfg->copy_mode, cfg->producer_warps,
                           cfg->math_mode, cfg->consumer_groups, cfg->split_rows};
        for (int i = 0; i < 12; ++i) key.c[i] = v[i];
    }
    alcs_launch_cfg stored;
    const alcs_launch_cfg* use = cfg;
    {
        std::lock_guard<std::mutex> lk(w->mu);
        auto it = w->plan_cache.find(key);
        if (it != w->plan_cache.end()) { *plan = it->second; return ALCS_OK; }
        if (!use) {     // a configuration tuned or set for the shape (stored under the public flags)
            auto t = w->tuned.find(alcs::ShapeKey{c.n, c.oh, c.ow, flags});
            if (t != w->tuned.end() && !((key.flags & kExtra) && t->second.math_mode == 3) && !((key.flags & kNoTc) && t->second.math_mode == 4)) {
                stored = t->second;
                use = &stored;
            }
        }
    }
    const int rc = cfg_to_plan(w, c, use, plan);
    if (rc) return rc;
    std::lock_guard<std::mutex> lk(w->mu);
    w->plan_cache[key] = *plan;
    return ALCS_OK;
}

// The plan of a call by default whose expanded weights found no memory: the staged kernels, for later calls of the shape, too.
bool no_room(const Plan& plan, const alcs_launch_cfg* cfg, int rc)
{
    return plan.tc_n && !cfg && (rc == ALCS_ERR_ALLOC || rc == ALCS_ERR_SHAPE);
}

int staged_instead(const alcs_packed* w, const CallShape& c, unsigned flags, Plan* plan)
{
    const int rc = staged_best(w, c, plan);
    if (rc) return rc;
    std::lock_guard<std::mutex> lk(w->mu);
    w->plan_cache[alcs::ShapeKey{c.n, c.oh, c.ow, key_flags(w, flags, c)}] = *plan;
    return ALCS_OK;
}

}  // namespace

// The same helpers for the other translation units of the library (alcs_internal.h).
namespace alcs {

int device_limits(int device, int* sms, int* smem_optin)
{
    DeviceInfo di;
    const int rc = device_info(device, &di);
    if (rc) return rc;
    *sms = di.sms;
    *smem_optin = di.smem_optin;
    return ALCS_OK;
}

int schedule_upload(const alcs_packed* w, Schedule* sc, void* cuda_stream)
{
    return upload_schedule(w, sc, static_cast<cudaStream_t>(cuda_stream));
}

int canonical_on_device(const alcs_packed* w, void* cuda_stream)
{
    return ensure_canonical_on_device(w, static_cast<cudaStream_t>(cuda_stream));
}

int require_current_device(const alcs_packed* w) { return check_device(w); }

}  // namespace alcs

namespace {
int noalloc_scratch_address(int dev, void** out);      // defined with alcs_spconv1x1_noalloc below
}

struct alcs_stack {
    struct Item {
        alcs_layer layer;
        Plan plan;
        long long q;
        int oh, ow;         // output size (= h, wd unless the layer has a stride)
    };
    std::vector<Item> items;
    // What one pass launches, in order: a layer by its plan, or (args) consecutive layers on the tcgen05 kernel, none
    // of which reads or writes what another one writes, in one launch.  Made from the items by build_runs().
    struct Run {
        int first, count;
        std::unique_ptr<alcs::TcArgs<alcs::kTcMaxLayers>> args;
        int* sched = nullptr;       // device
        std::vector<alcs::TcForm> forms;        // what args refer to
    };
    std::vector<Run> runs;
    bool runs_valid = false;
    unsigned flags = 0;
    cudaGraphExec_t exec = nullptr;
    // repack scratch of the stack's own (the layers run one after the other, so they share it):
    // allocated by alcs_stack_create, freed by alcs_stack_destroy, never moved in between
    void* xpad = nullptr;
    size_t xpad_bytes = 0;
};

namespace {

// Streams and events with which one alcs_spconv1x1_host call overlaps its uploads, convolutions and downloads.  A device
// has at most kMaxPipes of them.  A call takes one that nobody is enqueueing on and whose copies are either done or
// those of an earlier call on the same stream, which this one follows anyway: a call never waits for another
// stream's.  Re-recording an event does not disturb waits that were enqueued on its earlier state.
constexpr int kPipePieces = 4;
constexpr int kMaxPipes = 8;
struct CopyPipe {
    cudaStream_t in = nullptr, out = nullptr, user = nullptr;
    cudaEvent_t start = nullptr, in_done = nullptr, out_done = nullptr, uploaded[kPipePieces] = {}, computed[kPipePieces] = {};
    bool leased = false;
    bool make()
    {
        bool ok = cudaStreamCreateWithFlags(&in, cudaStreamNonBlocking) == cudaSuccess && cudaStreamCreateWithFlags(&out, cudaStreamNonBlocking) == cudaSuccess;
        auto event = [&](cudaEvent_t& e) { ok = ok && cudaEventCreateWithFlags(&e, cudaEventDisableTiming) == cudaSuccess; };
        event(start); event(in_done); event(out_done);
        for (int i = 0; i < kPipePieces; ++i) { event(uploaded[i]); event(computed[i]); }
        return ok;
    }
    bool idle() const { return cudaEventQuery(in_done) == cudaSuccess && cudaEventQuery(out_done) == cudaSuccess; }
    ~CopyPipe()
    {
        for (cudaEvent_t e : {start, in_done, out_done}) if (e) cudaEventDestroy(e);
        for (int i = 0; i < kPipePieces; ++i) {
            if (uploaded[i]) cudaEventDestroy(uploaded[i]);
            if (computed[i]) cudaEventDestroy(computed[i]);
        }
        if (in) cudaStreamDestroy(in);
        if (out) cudaStreamDestroy(out);
    }
};
std::mutex g_pipe_mu;
std::vector<std::unique_ptr<CopyPipe>>* const g_pipes = new std::vector<std::unique_ptr<CopyPipe>>[64];     // (never destroyed: the CUDA runtime may be gone by then)

struct PipeLease {
    CopyPipe* pipe = nullptr;       // null: all busy, or st is being captured (whose graph must not hold streams of other calls)
    PipeLease(int dev, cudaStream_t st)
    {
        // (queries and new streams must not end a capture that another thread has under way)
        cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
        cudaThreadExchangeStreamCaptureMode(&mode);
        cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
        if (cudaStreamIsCapturing(st, &capture) == cudaSuccess && capture == cudaStreamCaptureStatusNone) {
            std::lock_guard<std::mutex> lk(g_pipe_mu);
            auto& list = g_pipes[dev];
            for (const bool same : {true, false})
                for (auto& p : list)
                    if (!pipe && !p->leased && (same ? p->user == st : p->idle())) pipe = p.get();
            if (!pipe && list.size() < (size_t)kMaxPipes) {
                std::unique_ptr<CopyPipe> made(new (std::nothrow) CopyPipe());
                if (made && made->make()) {
                    pipe = made.get();
                    list.push_back(std::move(made));
                }
            }
            if (pipe) {
                pipe->leased = true;
                pipe->user = st;
            }
        }
        (void)cudaGetLastError();
        cudaThreadExchangeStreamCaptureMode(&mode);
    }
    ~PipeLease()
    {
        if (!pipe) return;
        std::lock_guard<std::mutex> lk(g_pipe_mu);
        pipe->leased = false;
    }
    PipeLease(const PipeLease&) = delete;
    PipeLease& operator=(const PipeLease&) = delete;
};

bool page_locked(const void* p)
{
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, p) == cudaSuccess) return a.type == cudaMemoryTypeHost;
    (void)cudaGetLastError();
    return false;
}

// Images per piece of a host-buffer call: four pieces of at least a megabyte whose X starts on 16-byte
// boundaries; n if the call is too small to gain from overlapping its copies (a piece costs about 10 us of calls).
int images_per_piece(int n, size_t x_image, size_t y_image)
{
    const size_t total = (x_image + y_image) * n;
    const int pieces = (int)std::min<size_t>({(size_t)kPipePieces, total >> 20, (size_t)n});
    if (pieces < 2) return n;
    for (int p = (n + pieces - 1) / pieces; p < n; ++p)
        if (x_image * p % 16 == 0 && y_image * p % 16 == 0) return p;
    return n;
}

}  // namespace

extern "C" {

ALCS_API int alcs_packed_upload(alcs_packed* p, int device, void* cuda_stream)
{
    if (!p) return ALCS_ERR_INVALID_ARG;
    if (p->device >= 0) return ALCS_ERR_STATE;
    int ndev = 0;
    ALCS_CUDA(cudaGetDeviceCount(&ndev));
    if (device < 0 || device >= ndev) return ALCS_ERR_INVALID_ARG;
    int prev = -1;
    ALCS_CUDA(cudaGetDevice(&prev));
    ALCS_CUDA(cudaSetDevice(device));
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    cudaError_t e = cudaMalloc(&p->d_err, 256);
    if (e == cudaSuccess) e = cudaMemsetAsync(p->d_err, 0, 256, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) {
        alcs::set_cuda_error_text(cudaGetErrorString(e));
        cudaFree(p->d_err);
        p->d_err = nullptr;
        (void)cudaGetLastError();
        cudaSetDevice(prev);
        return e == cudaErrorMemoryAllocation ? ALCS_ERR_ALLOC : ALCS_ERR_CUDA;
    }
    p->device = device;
    // Resolve the fixed scratch array of alcs_spconv1x1_noalloc now, at set-up time and with this
    // device current: the module that holds it is then loaded and the array backed on this device
    // before any phase in which the caller may no longer allocate.  (A failure here only matters to
    // that entry point, which looks the address up again and reports it.)
    void* scratch = nullptr;
    (void)noalloc_scratch_address(device, &scratch);
    cudaSetDevice(prev);
    return ALCS_OK;
}

ALCS_API int alcs_packed_status(const alcs_packed* p, int* code)
{
    if (!p || !code) return ALCS_ERR_INVALID_ARG;
    *code = 0;
    if (p->device < 0) return ALCS_ERR_STATE;
    ALCS_CUDA(cudaMemcpy(code, p->d_err, sizeof(int), cudaMemcpyDeviceToHost));
    return ALCS_OK;
}

ALCS_API void alcs_packed_free(alcs_packed* p)
{
    if (!p) return;
    if (p->device >= 0) {
        int prev = -1;
        if (cudaGetDevice(&prev) == cudaSuccess && cudaSetDevice(p->device) == cudaSuccess) {
            for (auto& kv : p->sched) free_schedule_device(kv.second);
            for (auto& kv : p->sched2d) free_schedule_device(kv.second);
            p->tc.clear();
            cudaFree(p->d_err);
            cudaFree(p->d_xpad);
            cudaFree(p->d_row_ptr);      // (the other two arrays lie in the same block)
            cudaSetDevice(prev);
        }
        (void)cudaGetLastError();
    }
    delete p;
}

ALCS_API int alcs_variant_count(void)
{
    std::lock_guard<std::mutex> lk(g_mu);
    init_variants_locked();
    return (int)g_variants.size();
}

ALCS_API int alcs_variant_get(int index, alcs_dtype* dt, int* g, alcs_launch_cfg* cfg)
{
    std::lock_guard<std::mutex> lk(g_mu);
    init_variants_locked();
    if (index < 0 || index >= (int)g_variants.size()) return ALCS_ERR_INVALID_ARG;
    const KernelVariant& v = g_variants[index].v;
    if (dt) *dt = (alcs_dtype)v.is_f16;
    if (g) *g = v.g;
    if (cfg) {
        std::memset(cfg, 0, sizeof *cfg);
        cfg->pixels_per_lane = v.p;
        cfg->rows_per_warp = v.rw;
        cfg->warps = v.nw;
        cfg->min_blocks = v.minb;
        cfg->copy_mode = 0;
        cfg->producer_warps = v.npw;
        cfg->math_mode = mode_of(v);
        cfg->consumer_groups = v.groups;
        cfg->split_rows = v.split ? 1 : 2;
    }
    return ALCS_OK;
}

ALCS_API int alcs_spconv1x1_cfg(const alcs_packed* w, const void* x, void* y, int n, int h, int wd,
                       const float* bias, unsigned flags, const alcs_launch_cfg* cfg,
                       void* cuda_stream)
{
    long long q = 0;
    int rc = check_conv_args(w, x, y, n, h, wd, flags, &q);
    if (rc) return rc;
    rc = check_device(w);
    if (rc) return rc;
    if (q == 0) return ALCS_OK;
    Plan plan;
    const CallShape shape = pointwise(n, h, wd, flags);
    rc = resolve_plan(w, shape, flags, cfg, &plan);
    if (rc) return rc;
    rc = launch_plan(w, plan, x, y, n, h, wd, bias, flags, static_cast<cudaStream_t>(cuda_stream));
    if (no_room(plan, cfg, rc) && (rc = staged_instead(w, shape, flags, &plan)) == ALCS_OK)
        rc = launch_plan(w, plan, x, y, n, h, wd, bias, flags, static_cast<cudaStream_t>(cuda_stream));
    return rc;
}

ALCS_API int alcs_spconv1x1(const alcs_packed* w, const void* x, void* y, int n, int h, int wd,
                   const float* bias, unsigned flags, void* cuda_stream)
{
    return alcs_spconv1x1_cfg(w, x, y, n, h, wd, bias, flags, nullptr, cuda_stream);
}

ALCS_API int alcs_spconv1x1_ex(const alcs_packed* w, const void* x, void* y, int n, int h, int wd, int stride,
                               const float* bias, const void* residual, unsigned flags,
                               const alcs_launch_cfg* cfg, void* cuda_stream)
{
    if (stride < 1 || h < 0 || wd < 0) return ALCS_ERR_INVALID_ARG;
    if (stride == 1 && !residual) return alcs_spconv1x1_cfg(w, x, y, n, h, wd, bias, flags, cfg, cuda_stream);
    const int oh = (h + stride - 1) / stride, ow = (wd + stride - 1) / stride;
    long long q = 0;
    // argument checks on the output-sized problem ...
    int rc = check_conv_args(w, x, y, n, oh, ow, flags, &q);
    if (rc) return rc;
    rc = check_device(w);
    if (rc) return rc;
    if (q == 0) return ALCS_OK;
    // ... plus what is specific to this entry point: the true extent of x, and the residual
    const size_t xe = w->elt(), ye = (w->dt != ALCS_F32 && !(flags & ALCS_Y_F32)) ? 2 : 4;
    if ((long long)h * wd > (1ll << 30) || (long long)h * wd * n > (1ll << 31)) return ALCS_ERR_SHAPE;
    const uintptr_t xb = (uintptr_t)x, xend = xb + (size_t)n * w->cin * h * wd * xe;
    const uintptr_t yb = (uintptr_t)y, yend = yb + (size_t)q * w->cout * ye;
    if (xb < yend && yb < xend) return ALCS_ERR_INVALID_ARG;
    if (residual) {
        const uintptr_t rb = (uintptr_t)residual, rend = rb + (size_t)q * w->cout * ye;
        if (rb % ye) return ALCS_ERR_INVALID_ARG;
        if (rb < yend && yb < rend) return ALCS_ERR_INVALID_ARG;     // the residual may not overlap y
    }
    Plan plan;
    const CallShape shape{n, oh, ow, h, wd, stride, residual != nullptr, (flags & ALCS_Y_F32) != 0};
    rc = resolve_plan(w, shape, flags, cfg, &plan);
    if (rc) return rc;
    auto launch = [&] { return launch_plan(w, plan, x, y, n, oh, ow, bias, flags, static_cast<cudaStream_t>(cuda_stream), nullptr, 0, residual, stride, h, wd); };
    rc = launch();
    if (no_room(plan, cfg, rc) && (rc = staged_instead(w, shape, flags, &plan)) == ALCS_OK) rc = launch();
    return rc;
}

ALCS_API int alcs_spconv1x1_plan(const alcs_packed* w, int n, int h, int wd, unsigned flags,
                        alcs_launch_cfg* out)
{
    if (!w || !out || n < 0 || h < 0 || wd < 0) return ALCS_ERR_INVALID_ARG;
    if (flags & ~(ALCS_RELU | ALCS_Y_F32)) return ALCS_ERR_INVALID_ARG;
    if ((flags & ALCS_Y_F32) && w->dt == ALCS_F32) return ALCS_ERR_INVALID_ARG;
    if (w->g != 1 && w->g != 2 && w->g != 4 && w->g != 8 && w->g != 16) return ALCS_ERR_UNSUPPORTED;
    if (w->device < 0) return ALCS_ERR_STATE;
    const long long q = (long long)n * h * wd;
    if ((long long)h * wd > (1ll << 30) || q > (1ll << 30)) return ALCS_ERR_SHAPE;
    Plan plan;
    const int rc = resolve_plan(w, pointwise(n, h, wd, flags), flags, nullptr, &plan);
    if (rc) return rc;
    plan_to_cfg(w, pointwise(n, h, wd, flags), plan, out);
    return ALCS_OK;
}

ALCS_API int alcs_spconv1x1_tune(alcs_packed* w, const void* x, void* y, int n, int h, int wd,
                        const float* bias, unsigned flags, void* cuda_stream,
                        alcs_launch_cfg* best)
{
    long long q = 0;
    int rc = check_conv_args(w, x, y, n, h, wd, flags, &q);
    if (rc) return rc;
    rc = check_device(w);
    if (rc) return rc;
    if (q == 0) return ALCS_OK;
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    const alcs::TcForms forms = alcs::tc_forms(w);
    std::vector<Plan> all;
    rc = enumerate_plans(w, pointwise(n, h, wd, flags), all);
    if (rc) return rc;
    const size_t max_try = 1200;
    if (all.size() > max_try) all.resize(max_try);
    // a buffer larger than L2, rewritten before every timed launch so that each candidate is
    // timed with cold caches, as it will run inside a network
    const size_t flush_bytes = 256u << 20;
    void* flush = nullptr;
    if (cudaMalloc(&flush, flush_bytes) != cudaSuccess) { (void)cudaGetLastError(); flush = nullptr; }
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    auto cleanup = [&]() {
        if (e0) cudaEventDestroy(e0);
        if (e1) cudaEventDestroy(e1);
        if (flush) cudaFree(flush);
    };
    if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess) {
        cleanup();
        alcs::set_cuda_error_text("cudaEventCreate failed");
        return ALCS_ERR_CUDA;
    }
    // one cold-cache launch of candidate i, in milliseconds (negative: the launch failed)
    auto time_once = [&](size_t i, int fill) -> float {
        if (flush) cudaMemsetAsync(flush, fill, flush_bytes, st);
        cudaEventRecord(e0, st);
        const bool ok = launch_plan(w, all[i], x, y, n, h, wd, bias, flags, st) == ALCS_OK;
        cudaEventRecord(e1, st);
        if (cudaEventSynchronize(e1) != cudaSuccess || !ok) return -1.0f;
        float ms = 0;
        cudaEventElapsedTime(&ms, e0, e1);
        return ms;
    };
    // First pass: every candidate, the best of `reps` launches after one untimed launch.
    const int reps = 3;
    std::vector<std::pair<float, int>> ranked;
    for (size_t i = 0; i < all.size(); ++i) {
        float tmin = 1e30f;
        bool ok = true;
        for (int r = 0; r < reps + 1 && ok; ++r) {
            const float ms = time_once(i, r);
            ok = ms >= 0;
            if (r > 0 && ok) tmin = std::min(tmin, ms);
        }
        if (ok) ranked.emplace_back(tmin, (int)i);
    }
    // Second pass: the few best candidates differ by less than the noise of three launches, so they
    // are timed again, in turn, and the one with the lowest median wins.
    std::sort(ranked.begin(), ranked.end());
    if (ranked.size() > kFinalists) ranked.resize(kFinalists);
    int best_i = -1;
    float best_ms = 1e30f;
    const int rounds = 15;
    std::vector<std::vector<float>> samples(ranked.size());
    for (int r = 0; r < rounds; ++r)
        for (size_t f = 0; f < ranked.size(); ++f) {
            const float ms = time_once((size_t)ranked[f].second, r);
            if (ms >= 0) samples[f].push_back(ms);
        }
    std::vector<std::pair<float, int>> by_median;
    for (size_t f = 0; f < ranked.size(); ++f) {
        if (samples[f].size() < (size_t)rounds) continue;
        std::nth_element(samples[f].begin(), samples[f].begin() + rounds / 2, samples[f].end());
        const float med = samples[f][rounds / 2];
        by_median.emplace_back(med, ranked[f].second);
        if (med < best_ms) { best_ms = med; best_i = ranked[f].second; }
    }
    std::sort(by_median.begin(), by_median.end());
    cudaError_t e = cudaStreamSynchronize(st);
    cleanup();
    if (e != cudaSuccess) { alcs::set_cuda_error_text(cudaGetErrorString(e)); return ALCS_ERR_CUDA; }
    if (best_i < 0) return ALCS_ERR_CUDA;
    alcs_launch_cfg c;
    plan_to_cfg(w, pointwise(n, h, wd, flags), all[best_i], &c);
    all[best_i].cost = 1e-3 * best_ms;
    {
        std::lock_guard<std::mutex> lk(w->mu);
        w->tuned[alcs::ShapeKey{n, h, wd, flags}] = c;
        w->tuned_alone.insert(alcs::ShapeKey{n, h, wd, flags});
        w->plan_cache[alcs::ShapeKey{n, h, wd, flags}] = all[best_i];
        std::vector<Plan>& fin = w->finalists[alcs::ShapeKey{n, h, wd, flags}];
        fin.clear();
        for (const auto& m : by_median) fin.push_back(all[m.second]);
    }
    {   // release the device copies of the schedules that did not win
        std::lock_guard<std::mutex> lk(w->mu);
        auto key_of = [&](const Plan& pl) {      // (kernels that use no schedule: a key that matches none)
            return pl.gather || pl.tc_n ? std::make_pair(0, 0) : alcs::sched_key(pl.kc, pl.n_rg, flavour_of(g_variants[pl.variant].v));
        };
        for (auto& kv : w->sched)
            if (kv.second.uploaded && kv.first != key_of(all[best_i])) {
                bool used = false;
                for (auto& pc : w->plan_cache) used |= (key_of(pc.second) == kv.first);
                if (!used) { free_schedule_device(kv.second); kv.second.n_rg = 0; }
            }
    }
    alcs::tc_release(w, forms);         // the expanded weights of the widths that did not win
    // leave y holding the result of the chosen configuration
    rc = launch_plan(w, all[best_i], x, y, n, h, wd, bias, flags, st);
    if (best) *best = c;
    return rc;
}

ALCS_API int alcs_spconv1x1_set_cfg(alcs_packed* w, int n, int h, int wd, unsigned flags,
                                    const alcs_launch_cfg* cfg)
{
    if (!w || !cfg || n < 0 || h < 0 || wd < 0) return ALCS_ERR_INVALID_ARG;
    if (flags & ~(ALCS_RELU | ALCS_Y_F32)) return ALCS_ERR_INVALID_ARG;
    if (w->device < 0) return ALCS_ERR_STATE;
    const long long q = (long long)n * h * wd;
    if ((long long)h * wd > (1ll << 30) || q > (1ll << 30)) return ALCS_ERR_SHAPE;
    Plan plan;
    const int rc = cfg_to_plan(w, pointwise(n, h, wd, flags), cfg, &plan);
    if (rc) return rc;
    alcs_launch_cfg full;
    plan_to_cfg(w, pointwise(n, h, wd, flags), plan, &full);
    std::lock_guard<std::mutex> lk(w->mu);
    const alcs::ShapeKey key{n, h, wd, flags};
    w->tuned[key] = full;
    w->tuned_alone.erase(key);
    w->plan_cache[key] = plan;
    return ALCS_OK;
}

ALCS_API size_t alcs_spconv1x1_host_workspace(const alcs_packed* w, int n, int h, int wd, unsigned flags)
{
    if (!w || n < 0 || h < 0 || wd < 0) return 0;
    const size_t q = (size_t)n * h * wd;
    const size_t ye = (w->dt != ALCS_F32 && !(flags & ALCS_Y_F32)) ? 2 : 4;
    auto up = [](size_t b) { return (b + 255) / 256 * 256; };
    return up(q * w->cin * w->elt()) + up(q * w->cout * ye) + up((size_t)w->cout * 4);
}

ALCS_API int alcs_spconv1x1_host(const alcs_packed* w, const void* x_host, void* y_host, int n, int h,
                        int wd, const float* bias_host, unsigned flags, void* workspace,
                        size_t workspace_bytes, void* cuda_stream)
{
    if (!w || !workspace || (uintptr_t)workspace % 256) return ALCS_ERR_INVALID_ARG;
    if (n < 0 || h < 0 || wd < 0) return ALCS_ERR_INVALID_ARG;
    const size_t need = alcs_spconv1x1_host_workspace(w, n, h, wd, flags);
    if (workspace_bytes < need) return ALCS_ERR_SHAPE;
    const size_t q = (size_t)n * h * wd;
    if (q == 0) return ALCS_OK;
    if (!x_host || !y_host) return ALCS_ERR_INVALID_ARG;
    const size_t ye = (w->dt != ALCS_F32 && !(flags & ALCS_Y_F32)) ? 2 : 4;
    auto up = [](size_t b) { return (b + 255) / 256 * 256; };
    const size_t xb = q * w->cin * w->elt(), yb = q * w->cout * ye;
    unsigned char* dx = static_cast<unsigned char*>(workspace);
    unsigned char* dy = dx + up(xb);
    float* db = reinterpret_cast<float*>(dy + up(yb));
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    int rc = check_device(w);
    if (rc) return rc;
    if (bias_host) ALCS_CUDA(cudaMemcpyAsync(db, bias_host, (size_t)w->cout * 4, cudaMemcpyHostToDevice, st));
    const size_t x_image = xb / n, y_image = yb / n;
    int per = images_per_piece(n, x_image, y_image);
    // Copies of pageable memory wait on the host, so pieces would overlap nothing and cost their calls (measured: a
    // call of 1.2 MB up and 2.4 MB down takes 340 us whole, 490 us in pieces).
    if (per < n && !(page_locked(x_host) && page_locked(y_host))) per = n;
    const unsigned char* const xh = static_cast<const unsigned char*>(x_host);
    unsigned char* const yh = static_cast<unsigned char*>(y_host);
    // A configuration stored for the call's shape holds for its pieces, too, where it can run them.
    alcs_launch_cfg stored;
    bool use_stored = false;
    if (per < n) {
        std::lock_guard<std::mutex> lk(w->mu);
        const auto it = w->tuned.find(alcs::ShapeKey{n, h, wd, flags});
        if (it != w->tuned.end()) { stored = it->second; use_stored = true; }
    }
    if (per < n) {
        // The bus carries both directions at once: piece i is downloaded while piece i + 1 is multiplied and piece
        // i + 2 uploaded.  Everything is ordered after what is on cuda_stream now and before what comes next.
        // Without a pipe the pieces follow one another on cuda_stream.
        PipeLease lease(w->device, st);
        CopyPipe* const pipe = lease.pipe;
        const cudaStream_t in = pipe ? pipe->in : st, out = pipe ? pipe->out : st;
        rc = ALCS_OK;
        cudaError_t e = cudaSuccess;
        auto ok = [&](cudaError_t c) { if (e == cudaSuccess) e = c; };
        if (pipe) {
            ok(cudaEventRecord(pipe->start, st));
            ok(cudaStreamWaitEvent(in, pipe->start, 0));
        }
        for (int i = 0, at = 0; at < n && rc == ALCS_OK && e == cudaSuccess; ++i, at += per) {
            const int m = std::min(per, n - at);
            unsigned char* const px = dx + x_image * at;
            unsigned char* const py = dy + y_image * at;
            ok(cudaMemcpyAsync(px, xh + x_image * at, x_image * m, cudaMemcpyHostToDevice, in));
            if (pipe) {
                ok(cudaEventRecord(pipe->uploaded[i], in));
                ok(cudaStreamWaitEvent(st, pipe->uploaded[i], 0));
            }
            const float* const b = bias_host ? db : nullptr;
            if (e == cudaSuccess) {
                rc = alcs_spconv1x1_cfg(w, px, py, m, h, wd, b, flags, use_stored ? &stored : nullptr, cuda_stream);
                if (rc == ALCS_ERR_UNSUPPORTED && use_stored) rc = alcs_spconv1x1(w, px, py, m, h, wd, b, flags, cuda_stream);
            }
            if (rc) break;
            if (pipe) {
                ok(cudaEventRecord(pipe->computed[i], st));
                ok(cudaStreamWaitEvent(out, pipe->computed[i], 0));
            }
            ok(cudaMemcpyAsync(yh + y_image * at, py, y_image * m, cudaMemcpyDeviceToHost, out));
        }
        if (pipe) {     // (also on an error: the caller's stream must not run ahead of the copies that were enqueued)
            const cudaError_t a1 = cudaEventRecord(pipe->in_done, in), a2 = cudaStreamWaitEvent(st, pipe->in_done, 0);
            const cudaError_t a3 = cudaEventRecord(pipe->out_done, out), a4 = cudaStreamWaitEvent(st, pipe->out_done, 0);
            for (const cudaError_t c : {a1, a2, a3, a4}) ok(c);
        }
        if (rc) return rc;
        ALCS_CUDA(e);
        return ALCS_OK;
    }
    ALCS_CUDA(cudaMemcpyAsync(dx, x_host, xb, cudaMemcpyHostToDevice, st));
    rc = alcs_spconv1x1(w, dx, dy, n, h, wd, bias_host ? db : nullptr, flags, cuda_stream);
    if (rc) return rc;
    ALCS_CUDA(cudaMemcpyAsync(y_host, dy, yb, cudaMemcpyDeviceToHost, st));
    return ALCS_OK;
}

}  // extern "C"

namespace {

// Bytes [first, last) of a layer's buffers.
struct Extent {
    uintptr_t b, e;
    bool meets(const Extent& o) const { return b < o.e && o.b < e; }
};

struct LayerExtents {
    Extent x, y, res, bias;
};

LayerExtents extents(const alcs_stack::Item& it)
{
    const alcs_layer& L = it.layer;
    const size_t xe = L.w->elt(), ye = (L.w->dt != ALCS_F32 && !(L.flags & ALCS_Y_F32)) ? 2 : 4;
    const size_t yb = (size_t)it.q * L.w->cout * ye;
    LayerExtents r;
    r.x = {(uintptr_t)L.x, (uintptr_t)L.x + (size_t)L.n * L.w->cin * L.h * L.wd * xe};
    r.y = {(uintptr_t)L.y, (uintptr_t)L.y + yb};
    r.res = {(uintptr_t)L.residual, L.residual ? (uintptr_t)L.residual + yb : 0};
    r.bias = {(uintptr_t)L.bias, L.bias ? (uintptr_t)(L.bias + L.w->cout) : 0};
    return r;
}

// May the two layers run at the same time?
bool independent(const LayerExtents& a, const LayerExtents& b)
{
    auto writes_input = [](const Extent& y, const LayerExtents& o) { return y.meets(o.x) || y.meets(o.res) || y.meets(o.bias); };
    return !(a.y.meets(b.y) || writes_input(a.y, b) || writes_input(b.y, a));
}

CallShape call_shape(const alcs_stack::Item& it)
{
    const alcs_layer& L = it.layer;
    return {L.n, it.oh, it.ow, L.h, L.wd, L.stride > 1 ? L.stride : 1, L.residual != nullptr, (L.flags & ALCS_Y_F32) != 0};
}

alcs::TcProblem tc_problem(const alcs_stack::Item& it)
{
    const alcs_layer& L = it.layer;
    return tc_problem(L.x, L.y, L.n, it.oh, it.ow, L.bias, L.flags, L.residual, L.stride > 1 ? L.stride : 1, L.h, L.wd);
}

// Layers [first, end) that one launch of the tcgen05 kernel could take, starting at `first`; eligible(i) says
// whether layer i may be part of it.
template <typename F>
size_t merge_end(const alcs_stack* s, size_t first, F eligible)
{
    std::vector<LayerExtents> ext;
    size_t end = first;
    for (; end < s->items.size() && end - first < (size_t)alcs::kTcMaxLayers; ++end) {
        const alcs_stack::Item& it = s->items[end];
        if (it.q == 0 || !eligible(it) || it.layer.w->dt != s->items[first].layer.w->dt || it.layer.w->device != s->items[first].layer.w->device) break;
        const LayerExtents e = extents(it);
        bool free = true;
        for (const LayerExtents& o : ext) free = free && independent(e, o);
        if (!free) break;
        ext.push_back(e);
    }
    return end;
}

// Fixed cost of a merged launch, first copies and last stores included, in microseconds.
constexpr double kMergedRampUs = 5.0;

// Consecutive independent layers whose configuration nobody fixed for the stack: one launch of a tcgen05 kernel for
// all of them, where its estimate is below the sum of the layers' own (measured ones, after alcs_spconv1x1_tune).  With few items in all, narrower tiles shorten
// the longest SM's share; with many, wide ones do the least work.
// by: what decides; alcs_stack_tune measures both ways, of whatever was fixed, too.
enum class MergeBy { estimates, one_launch, kernels };
void stack_merge(alcs_stack* s, MergeBy by = MergeBy::estimates)
{
    auto open = [&](const alcs_stack::Item& it) {
        const alcs_layer& L = it.layer;
        if (L.stride > 1 || !tc_ok(L.w, call_shape(it)) || (long long)L.w->rows * L.w->g * L.w->cin > alcs::kTcMaxWeights) return false;
        if (by != MergeBy::estimates) return true;
        const alcs::ShapeKey key{L.n, it.oh, it.ow, L.flags};
        std::lock_guard<std::mutex> lk(L.w->mu);
        return L.w->tuned.find(key) == L.w->tuned.end() || L.w->tuned_alone.count(key) != 0;
    };
    for (size_t i = 0; i < s->items.size();) {
        const size_t end = s->items[i].q ? merge_end(s, i, open) : i;
        DeviceInfo di;
        if (end - i < 2 || device_info(s->items[i].layer.w->device, &di)) { i = std::max(end, i + 1); continue; }
        std::vector<int> widths(end - i), pixels(end - i), choice, choice_px;
        // Layers [from, to) in one launch of one of the two kernels: the widths (and pixels) that take the least, and the time.
        auto together = [&](size_t from, size_t to, bool sixteen) {
            double best = 0;
            std::vector<int> n_of(to - from), px_of(to - from);
            for (int cap = alcs::kTcMaxN; cap >= (sixteen ? 32 : 16); cap /= 2)
                for (int cap_px = sixteen ? alcs::kTc16Pixels : alcs::kTcM; cap_px >= (sixteen ? 32 : alcs::kTcM); cap_px /= 2) {
                    double total = 0, longest = 0;
                    for (size_t k = from; k < to; ++k) {
                        const alcs_stack::Item& it = s->items[k];
                        const alcs_packed* w = it.layer.w;
                        const alcs::TcProblem pr = tc_problem(it);
                        int n[8], at = 0;
                        const int count = tc_widths(w, n);
                        while (at + 1 < count && n[at] > cap) ++at;
                        std::vector<double> us;
                        int px = alcs::kTcM;
                        if (sixteen) {
                            const std::vector<int> steps = alcs::tc_tile_steps(w, pr, n[at]);
                            px = alcs::tc16_capped(w, pr, steps.empty() ? 0 : *std::max_element(steps.begin(), steps.end()), cap_px);
                            for (int k16 : steps) us.push_back(alcs::tc16_item_us(w, pr, n[at], k16, px));
                        } else {
                            us = alcs::tc_tiles_us(w, pr, n[at]);
                        }
                        for (const double t : us) {
                            total += t * (double)((it.q + px - 1) / px);
                            longest = std::max(longest, t);
                        }
                        n_of[k - from] = n[at];
                        px_of[k - from] = sixteen ? px : 0;
                    }
                    const double t = kMergedRampUs + std::max(total / di.sms, longest) + 0.25 * longest;
                    if (best > 0 && t >= best) continue;
                    best = t;
                    std::copy(n_of.begin(), n_of.end(), widths.begin() + (from - i));
                    std::copy(px_of.begin(), px_of.end(), pixels.begin() + (from - i));
                }
            return best;
        };
        double best = 0;
        for (size_t k = i; k < end; ++k) best += s->items[k].plan.cost * 1e6;
        const double one = by == MergeBy::kernels ? 0 : together(i, end, false);
        if (by == MergeBy::one_launch || (by == MergeBy::estimates && one < best)) { best = one; choice = widths; choice_px = pixels; }
        // 16-bit operands: layers whose rows can be copied as they are on alcs_tc16.cu, a launch per sequence of layers of one kind.
        // Several launches have to promise a tenth, as the estimates favour them: of 80 stacks of pointwise layers (two networks, inputs of
        // 160 to 288, batches of 1 to 48) 8 run so, 2 to 19 % faster than in one launch; were all of them to run so, others would
        // gain up to 24 % and lose up to 43 %.
        auto direct = [&](size_t k) { return alcs::tc16_direct(s->items[k].layer.w, tc_problem(s->items[k])); };
        if (by != MergeBy::one_launch && s->items[i].layer.w->dt != ALCS_F32) {
            double t = 0;
            int launches = 0;
            bool any = false;
            for (size_t from = i, to; from < end; from = to, ++launches) {
                for (to = from + 1; to < end && direct(to) == direct(from);) ++to;
                t += together(from, to, direct(from));
                any = any || direct(from);
            }
            if (any && (by == MergeBy::kernels || t * (launches > 1 ? 1.1 : 1.0) < best)) { best = t; choice = widths; choice_px = pixels; }
        }
        for (size_t k = i; k < end && !choice.empty(); ++k) {
            alcs_stack::Item& it = s->items[k];
            it.plan = tc_plan_on(it.layer.w, choice[k - i], call_shape(it), di.sms, choice_px[k - i]);
        }
        i = end;
    }
}

// What the layers' plans need on the device must be there before any launch is captured.
int stack_make_resident(alcs_stack* s)
{
    for (auto& it : s->items) {
        if (it.q == 0) continue;
        const alcs_packed* w = it.layer.w;
        int rc = ALCS_OK;
        if (it.plan.gather) {
            rc = ensure_canonical_on_device(w, nullptr);
        } else if (it.plan.tc_n) {
            alcs::TcForm t;
            rc = alcs::tc_prepare(w, tc_key(w, it.plan, tc_problem(it)), nullptr, &t);
            if (no_room(it.plan, nullptr, rc)) rc = staged_instead(w, call_shape(it), it.layer.flags, &it.plan);
        }
        if (!rc && !it.plan.gather && !it.plan.tc_n) {
            Schedule* sc = get_schedule(w, it.plan.kc, it.plan.n_rg, true, flavour_of(g_variants[it.plan.variant].v));
            rc = sc ? upload_schedule(w, sc, nullptr) : ALCS_ERR_ALLOC;
        }
        if (rc) return rc;
    }
    return ALCS_OK;
}

// Scratch for the repacked inputs of the staged kernels: of the layers that run on one, or (any_plan) of every
// layer, with room for copy mode 4 at any tile width, so that alcs_stack_tune may switch a layer to it.
int stack_scratch(alcs_stack* s, bool any_plan)
{
    size_t need = 0;
    for (const auto& it : s->items) {
        if (it.q == 0 || (!any_plan && (it.plan.gather || it.plan.tc_n))) continue;
        const alcs_layer& L = it.layer;
        const int elt = (int)L.w->elt();
        const long long hw = (long long)it.oh * it.ow;
        const size_t px = (size_t)L.n * padded_hw((int)hw, elt);
        if (px > (1ull << 30)) continue;
        if ((hw * elt) % 16 != 0 || L.stride > 1) need = std::max(need, px * L.w->cin * elt);
        if (it.q > 8 * hw) need = std::max(need, (px + 512) * L.w->cin * (elt + 1));
    }
    if (need <= s->xpad_bytes) return ALCS_OK;
    void* room = nullptr;
    if (cudaMalloc(&room, need) != cudaSuccess) {       // (the old scratch, which a captured graph may name, stays)
        (void)cudaGetLastError();
        return ALCS_ERR_ALLOC;
    }
    if (s->exec) { cudaGraphExecDestroy(s->exec); s->exec = nullptr; }
    if (s->xpad) cudaFree(s->xpad);
    s->xpad = room;
    s->xpad_bytes = need;
    return ALCS_OK;
}

void drop_runs(alcs_stack* s)
{
    for (auto& r : s->runs)
        if (r.sched) cudaFree(r.sched);
    s->runs.clear();
    s->runs_valid = false;
}

// One launch for items [first, end): arguments, and which SM takes which items.  Items of different layers take
// different times, so they are dealt out by a greedy list: in order, the next item to the SM that is free first;
// where each SM gets only a few, the longest ones go first.
int build_merged(alcs_stack* s, size_t first, size_t end)
{
    const alcs_packed* w0 = s->items[first].layer.w;
    DeviceInfo di;
    int rc = device_info(w0->device, &di);
    if (rc) return rc;
    alcs_stack::Run run;
    run.first = (int)first;
    run.count = (int)(end - first);
    run.args.reset(new alcs::TcArgs<alcs::kTcMaxLayers>());
    alcs::TcArgs<alcs::kTcMaxLayers>& a = *run.args;
    a.n_layers = run.count;
    for (int i = 0; i < run.count; ++i) {
        const auto& it = s->items[first + i];
        alcs::TcForm t;
        rc = alcs::tc_prepare(it.layer.w, tc_key(it.layer.w, it.plan, tc_problem(it)), nullptr, &t);
        if (rc) return rc;
        run.forms.push_back(t);
    }
    std::vector<std::vector<double>> us(run.count);       // per layer and channel tile
    for (int i = 0; i < run.count; ++i) {
        const auto& it = s->items[first + i];
        const alcs::TcForm& t = run.forms[i];
        alcs::TcProblem pr = tc_problem(it);
        pr.pixels = it.plan.tc_px ? alcs::tc16_capped(it.layer.w, pr, t->k16_max, it.plan.tc_px) : 0;
        rc = alcs::tc_fill(it.layer.w, *t, pr, &a.layer[i]);
        if (rc) return rc;
        for (int k16 : t->k16)
            us[i].push_back(pr.pixels ? alcs::tc16_item_us(it.layer.w, pr, t->n, k16, a.layer[i].ppt) : alcs::tc_merged_item_us(w0->dt, t->n, k16));
    }
    rc = alcs::tc_finish(w0, a, false);
    if (rc) return rc;
    if (run.count > 1) {
        const int blocks = std::min(a.n_items, di.sms);
        std::vector<std::pair<double, int>> items;
        items.reserve(a.n_items);
        for (int i = 0; i < run.count; ++i) {
            const alcs::TcLayer& y = a.layer[i];
            for (int k = 0; k < y.n_tiles.d * y.px_tiles.d; ++k)
                items.emplace_back(us[i][y.tile_major ? k / y.px_tiles.d : k % y.n_tiles.d], y.first_item + k);
        }
        if (a.n_items <= 16 * blocks || a.layer[0].n_px)
            std::stable_sort(items.begin(), items.end(), [](const auto& x, const auto& y) { return x.first > y.first; });
        std::priority_queue<std::pair<double, int>, std::vector<std::pair<double, int>>, std::greater<std::pair<double, int>>> idle;
        for (int b = 0; b < blocks; ++b) idle.emplace(0.0, b);
        std::vector<std::vector<int>> list(blocks);
        size_t longest = 0;
        for (const auto& it : items) {
            auto b = idle.top();
            idle.pop();
            list[b.second].push_back(it.second);
            longest = std::max(longest, list[b.second].size());
            idle.emplace(b.first + it.first, b.second);
        }
        std::vector<int> table((longest + 1) * blocks, -1);
        for (int b = 0; b < blocks; ++b)
            for (size_t k = 0; k < list[b].size(); ++k) table[k * blocks + b] = list[b][k];
        if (cudaMalloc(&run.sched, table.size() * 4) != cudaSuccess) {
            (void)cudaGetLastError();
            return ALCS_ERR_ALLOC;
        }
        a.sched = run.sched;
        const cudaError_t e = cudaMemcpy(run.sched, table.data(), table.size() * 4, cudaMemcpyHostToDevice);
        if (e != cudaSuccess) {
            cudaFree(run.sched);
            alcs::set_cuda_error_text(cudaGetErrorString(e));
            (void)cudaGetLastError();
            return ALCS_ERR_CUDA;
        }
    }
    s->runs.push_back(std::move(run));
    return ALCS_OK;
}

int build_runs(alcs_stack* s)
{
    drop_runs(s);
    auto on_tc = [](const alcs_stack::Item& it) { return it.plan.tc_n != 0 && it.layer.stride <= 1; };
    for (size_t i = 0; i < s->items.size();) {
        if (s->items[i].q == 0) { ++i; continue; }
        // (layers of one kernel)
        const size_t end = merge_end(s, i, [&](const alcs_stack::Item& it) { return on_tc(it) && !it.plan.tc_px == !s->items[i].plan.tc_px; });
        if (end > i) {
            const int rc = build_merged(s, i, end);
            if (rc) { drop_runs(s); return rc; }
            i = end;
        } else {
            alcs_stack::Run run;
            run.first = (int)i;
            run.count = 1;
            s->runs.push_back(std::move(run));
            ++i;
        }
    }
    s->runs_valid = true;
    return ALCS_OK;
}

}  // namespace

extern "C" {

ALCS_API int alcs_stack_destroy(alcs_stack* s);

ALCS_API int alcs_stack_create(const alcs_layer* layers, int n_layers, unsigned stack_flags, alcs_stack** out)
{
    if (!out) return ALCS_ERR_INVALID_ARG;
    *out = nullptr;
    if (!layers || n_layers < 0 || (stack_flags & ~ALCS_STACK_GRAPH)) return ALCS_ERR_INVALID_ARG;
    alcs_stack* s = new (std::nothrow) alcs_stack();
    if (!s) return ALCS_ERR_ALLOC;
    s->flags = stack_flags;
    for (int i = 0; i < n_layers; ++i) {
        const alcs_layer& L = layers[i];
        alcs_stack::Item it;
        it.layer = L;
        if (L.stride < 0) { delete s; return ALCS_ERR_INVALID_ARG; }
        const int stride = L.stride > 1 ? L.stride : 1;
        it.oh = (L.h + stride - 1) / stride;
        it.ow = (L.wd + stride - 1) / stride;
        int rc = check_conv_args(L.w, L.x, L.y, L.n, it.oh, it.ow, L.flags, &it.q);
        if (!rc) rc = check_device(L.w);
        if (!rc && it.q > 0) rc = resolve_plan(L.w, call_shape(it), L.flags, nullptr, &it.plan);
        if (!rc && it.q > 0) it.plan.tc_px = tc_pixels(L.w, it.plan, tc_problem(it));
        if (rc) { delete s; return rc; }
        s->items.push_back(it);
    }
    stack_merge(s);
    int rc = stack_make_resident(s);
    if (!rc) rc = stack_scratch(s, false);
    if (!rc) rc = build_runs(s);
    if (rc) { alcs_stack_destroy(s); return rc; }
    *out = s;
    return ALCS_OK;
}

static int stack_enqueue(alcs_stack* s, cudaStream_t st)
{
    for (auto& run : s->runs) {
        const auto& it = s->items[run.first];
        const alcs_layer& L = it.layer;
        // one named range per launch: a timeline then shows the per-layer run times T^(l) whose sum the
        // paper's latency model is about (a no-op unless a profiler has attached itself to the process)
        char name[96];
        if (run.count > 1) std::snprintf(name, sizeof name, "alcs layers %d to %d", run.first + 1, run.first + run.count);
        else std::snprintf(name, sizeof name, "alcs layer %d: %d->%d @%dx%d n=%d", run.first + 1, L.w->cin, L.w->cout, L.h, L.wd, L.n);
        nvtxRangePushA(name);
        struct Pop { ~Pop() { nvtxRangePop(); } } pop;
        const int rc = run.args ? alcs::tc_launch(L.w, *run.args, false, st)
                                : launch_plan(L.w, it.plan, L.x, L.y, L.n, it.oh, it.ow, L.bias, L.flags, st, s->xpad, s->xpad_bytes,
                                              L.residual, L.stride > 1 ? L.stride : 1, L.h, L.wd);
        if (rc) return rc;
    }
    return ALCS_OK;
}

ALCS_API int alcs_stack_run(alcs_stack* s, void* cuda_stream)
{
    if (!s) return ALCS_ERR_INVALID_ARG;
    if (!s->runs_valid) {
        const int rc = build_runs(s);
        if (rc) return rc;
    }
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    if (!(s->flags & ALCS_STACK_GRAPH)) return stack_enqueue(s, st);
    if (!s->exec) {
        cudaStream_t cap = nullptr;
        // capture on a private stream so that the caller's stream may be the legacy default one
        ALCS_CUDA(cudaStreamCreateWithFlags(&cap, cudaStreamNonBlocking));
        cudaGraph_t graph = nullptr;
        cudaError_t e = cudaStreamBeginCapture(cap, cudaStreamCaptureModeThreadLocal);
        int rc = ALCS_OK;
        if (e == cudaSuccess) {
            rc = stack_enqueue(s, cap);
            e = cudaStreamEndCapture(cap, &graph);
        }
        if (e == cudaSuccess && rc == ALCS_OK) e = cudaGraphInstantiate(&s->exec, graph, 0);
        if (graph) cudaGraphDestroy(graph);
        cudaStreamDestroy(cap);
        if (rc) return rc;
        if (e != cudaSuccess) {
            alcs::set_cuda_error_text(cudaGetErrorString(e));
            (void)cudaGetLastError();
            s->exec = nullptr;
            return ALCS_ERR_CUDA;
        }
    }
    ALCS_CUDA(cudaGraphLaunch(s->exec, st));
    return ALCS_OK;
}

namespace {

bool same_plan(const Plan& a, const Plan& b)
{
    return a.variant == b.variant && a.kc == b.kc && a.n_rg == b.n_rg && a.stages == b.stages && a.bulk == b.bulk &&
           a.gather == b.gather && a.gp == b.gp && a.gks == b.gks && a.tc_n == b.tc_n && a.tc_px == b.tc_px;
}

// Run time of one pass over the whole stack in microseconds, as alcs_stack_run runs it (a graph stack
// is captured again with the plans it holds now): the best of three batches of `reps` runs after two
// untimed ones.  Negative if a launch failed.
double time_stack(alcs_stack* s, cudaStream_t st, cudaEvent_t e0, cudaEvent_t e1, int reps)
{
    if (s->exec) { cudaGraphExecDestroy(s->exec); s->exec = nullptr; }
    s->runs_valid = false;
    for (int i = 0; i < 2; ++i)
        if (alcs_stack_run(s, st) != ALCS_OK) return -1.0;
    double best = 1e30;
    for (int b = 0; b < 3; ++b) {
        cudaEventRecord(e0, st);
        for (int i = 0; i < reps; ++i)
            if (alcs_stack_run(s, st) != ALCS_OK) return -1.0;
        cudaEventRecord(e1, st);
        if (cudaEventSynchronize(e1) != cudaSuccess) return -1.0;
        float ms = 0;
        cudaEventElapsedTime(&ms, e0, e1);
        best = std::min(best, (double)ms * 1e3 / reps);
    }
    return best;
}

// The plans worth trying for one layer of a stack: what the last alcs_spconv1x1_tune of its shape ranked
// best, else the model's best few and every shape of the small-problem kernel that applies.
int stack_candidates(const alcs_stack::Item& it, std::vector<Plan>& out)
{
    const alcs_layer& L = it.layer;
    const bool extra = (L.stride > 1) || L.residual;
    out.clear();
    {
        std::lock_guard<std::mutex> lk(L.w->mu);
        auto f = L.w->finalists.find(alcs::ShapeKey{L.n, it.oh, it.ow, L.flags});
        if (f != L.w->finalists.end())
            for (const Plan& p : f->second)
                if (!(extra && p.gather) && !(L.stride > 1 && p.tc_n)) out.push_back(p);
    }
    const bool had = !out.empty();
    const bool small = !extra && it.oh * it.ow > 0 && it.q / ((long long)it.oh * it.ow) <= kGatherImages;
    if (had && !small) return ALCS_OK;
    std::vector<Plan> all;
    const int rc = enumerate_plans(L.w, call_shape(it), all);
    if (rc) return rc;
    int ranked = 0;
    std::vector<int> widths;
    for (size_t i = 0; i < all.size(); ++i) {
        // (the tcgen05 kernels with as many channels per tile count once)
        const bool again = all[i].tc_n && std::find(widths.begin(), widths.end(), all[i].tc_n) != widths.end();
        if (all[i].tc_n && !again) widths.push_back(all[i].tc_n);
        ranked += !again;
        if (!((!had && ranked <= 8) || all[i].gather) || (L.stride > 1 && all[i].tc_n)) continue;
        bool dup = false;
        for (const Plan& p : out) dup |= same_plan(p, all[i]);
        if (!dup) out.push_back(all[i]);
    }
    return ALCS_OK;
}

}  // namespace

ALCS_API int alcs_stack_tune(alcs_stack* s, int passes, void* cuda_stream, double* us_before, double* us_after)
{
    if (!s || passes < 0) return ALCS_ERR_INVALID_ARG;
    if (passes == 0) passes = 2;
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess) {
        if (e0) cudaEventDestroy(e0);
        (void)cudaGetLastError();
        alcs::set_cuda_error_text("cudaEventCreate failed");
        return ALCS_ERR_CUDA;
    }
    struct Done { cudaEvent_t a, b; ~Done() { cudaEventDestroy(a); cudaEventDestroy(b); } } done{e0, e1};
    const int scratch_rc = stack_scratch(s, true);
    if (scratch_rc) return scratch_rc;
    std::map<const alcs_packed*, alcs::TcForms> forms;
    for (const auto& it : s->items)
        if (!forms.count(it.layer.w)) forms[it.layer.w] = alcs::tc_forms(it.layer.w);
    double cur = time_stack(s, st, e0, e1, 3);
    if (cur < 0) return ALCS_ERR_CUDA;
    const int reps = (int)std::min(100.0, std::max(3.0, 3000.0 / std::max(cur, 1.0)));     // batches of about 3 ms
    cur = time_stack(s, st, e0, e1, reps);
    if (cur < 0) return ALCS_ERR_CUDA;
    if (us_before) *us_before = cur;
    for (MergeBy by : {MergeBy::one_launch, MergeBy::kernels}) {
        // one launch for all independent layers, or for each sequence of one kernel: no sequence of single-layer changes leads there
        std::vector<Plan> keep;
        bool changed = false;
        for (const auto& it : s->items) keep.push_back(it.plan);
        stack_merge(s, by);
        for (size_t i = 0; i < keep.size(); ++i) changed |= !same_plan(keep[i], s->items[i].plan);
        if (!changed) continue;
        const double t = time_stack(s, st, e0, e1, reps);
        if (t > 0 && t < cur * 0.996) cur = t;
        else
            for (size_t i = 0; i < keep.size(); ++i) s->items[i].plan = keep[i];
    }
    for (int pass = 0; pass < passes; ++pass) {
        bool changed = false;
        for (auto& it : s->items) {
            if (it.q == 0) continue;
            const alcs_layer& L = it.layer;
            int rc = check_device(L.w);
            if (rc) return rc;
            std::vector<Plan> cands;
            rc = stack_candidates(it, cands);
            if (rc) return rc;
            Plan best = it.plan;
            double best_t = cur;
            for (const Plan& c : cands) {
                if (same_plan(c, best) || same_plan(c, it.plan)) continue;
                if (c.gather) {
                    if (ensure_canonical_on_device(L.w, nullptr) != ALCS_OK) continue;
                } else if (!c.tc_n) {
                    const KernelVariant& v = g_variants[c.variant].v;
                    Schedule* sc = get_schedule(L.w, c.kc, c.n_rg, true, flavour_of(v));
                    if (!sc || (v.split && sc->max_x == 0) || upload_schedule(L.w, sc, nullptr) != ALCS_OK) continue;
                }
                const Plan keep = it.plan;
                it.plan = c;
                const double t = time_stack(s, st, e0, e1, reps);
                it.plan = keep;
                // a candidate must beat the incumbent by more than the timing noise
                if (t > 0 && t < best_t * 0.996) { best_t = t; best = c; }
            }
            if (!same_plan(best, it.plan)) {
                it.plan = best;
                cur = best_t;
                changed = true;
            }
        }
        if (!changed) break;
    }
    for (auto& it : s->items) {
        if (it.q == 0) continue;
        const alcs_layer& L = it.layer;
        alcs_launch_cfg c;
        it.plan.tc_named = tc16_ok(L.w, call_shape(it));
        plan_to_cfg(L.w, call_shape(it), it.plan, &c);
        const alcs::ShapeKey key{L.n, it.oh, it.ow, key_flags(L.w, L.flags, call_shape(it))};
        std::lock_guard<std::mutex> lk(L.w->mu);
        L.w->tuned[alcs::ShapeKey{L.n, it.oh, it.ow, L.flags}] = c;
        L.w->tuned_alone.erase(alcs::ShapeKey{L.n, it.oh, it.ow, L.flags});
        L.w->plan_cache[key] = it.plan;
    }
    cur = time_stack(s, st, e0, e1, reps);      // (also leaves a graph stack captured with the chosen plans)
    if (cur < 0) return ALCS_ERR_CUDA;
    for (const auto& f : forms) alcs::tc_release(f.first, f.second);
    if (us_after) *us_after = cur;
    return ALCS_OK;
}

ALCS_API int alcs_stack_layer_cfg(const alcs_stack* s, int layer, alcs_launch_cfg* out)
{
    if (!s || !out || layer < 0 || layer >= (int)s->items.size()) return ALCS_ERR_INVALID_ARG;
    std::memset(out, 0, sizeof *out);
    if (s->items[layer].q == 0) return ALCS_OK;
    plan_to_cfg(s->items[layer].layer.w, call_shape(s->items[layer]), s->items[layer].plan, out);
    return ALCS_OK;
}

ALCS_API int alcs_stack_destroy(alcs_stack* s)
{
    if (!s) return ALCS_OK;
    if (s->exec) cudaGraphExecDestroy(s->exec);
    drop_runs(s);
    if (s->xpad) cudaFree(s->xpad);     // waits for the device, so no replay can still be using it
    delete s;
    return ALCS_OK;
}

}  // extern "C"

// ---------------------------------------------------------------------------------------------
// alcs_spconv1x1_noalloc: the convolution for callers that cannot allocate device memory.
//
// Everything this entry point needs beyond the caller's buffers is either already resident (the
// launch schedule, put there by an earlier ordinary call for the same shape) or lives in the fixed
// array below, which is part of the library image.  The array's name is only a handle in host
// code: its device address is looked up once per device with cudaGetSymbolAddress and that pointer
// is what the kernels receive.
// ---------------------------------------------------------------------------------------------
static __device__ __align__(256) unsigned char g_noalloc_scratch[ALCS_NOALLOC_SCRATCH_BYTES];

namespace {

void* g_noalloc_ptr[64] = {nullptr};     // device address of g_noalloc_scratch, per device
std::mutex g_noalloc_mu;

// Device address of the fixed scratch array on the current device `dev` (looked up on first use).
int noalloc_scratch_address(int dev, void** out)
{
    if (dev < 0 || dev >= 64) return ALCS_ERR_INVALID_ARG;
    std::lock_guard<std::mutex> lk(g_noalloc_mu);
    if (!g_noalloc_ptr[dev]) {
        void* p = nullptr;
        ALCS_CUDA(cudaGetSymbolAddress(&p, g_noalloc_scratch));
        g_noalloc_ptr[dev] = p;
    }
    *out = g_noalloc_ptr[dev];
    return ALCS_OK;
}

}  // namespace

extern "C" ALCS_API int alcs_spconv1x1_noalloc(const alcs_packed* w, const void* x, void* y, int n, int h, int wd,
                                               const float* bias, unsigned flags, void* cuda_stream)
{
    long long q = 0;
    int rc = check_conv_args(w, x, y, n, h, wd, flags, &q);
    if (rc) return rc;
    rc = check_device(w);
    if (rc) return rc;
    if (q == 0) return ALCS_OK;
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);

    // The plan and its schedule must already be resident: looking them up allocates nothing.
    Plan plan;
    Schedule* sc = nullptr;
    {
        std::lock_guard<std::mutex> lk(w->mu);
        auto it = w->plan_cache.find(alcs::ShapeKey{n, h, wd, flags});
        if (it == w->plan_cache.end()) return ALCS_ERR_STATE;
        plan = it->second;
        if (plan.gather && w->d_row_ptr)      // the small-problem kernel: needs only its resident copy of the storage format
            return launch_gather_plan(w, plan, x, y, n, h, wd, bias, flags, st);
        if (!plan.gather && !plan.tc_n) {
            auto si = w->sched.find(alcs::sched_key(plan.kc, plan.n_rg, flavour_of(g_variants[plan.variant].v)));
            if (si != w->sched.end() && si->second.uploaded) sc = &si->second;
        }
        if (!sc) {
            // The tcgen05 kernel, in the form that the plan names or in any other that is resident: alcs_stack_create
            // prepares the form of the launch it merged the layer into, the plan is that of a call by itself.  It
            // needs no scratch, but what does not fit that is refused whatever kernel the plan names.
            const size_t row = (size_t)h * wd * w->elt();
            if (row % 16 != 0 && (size_t)n * w->cin * ((row + 15) / 16 * 16) > ALCS_NOALLOC_SCRATCH_BYTES) return ALCS_ERR_TOO_LARGE;
            alcs::TcProblem pr = tc_problem(x, y, n, h, wd, bias, flags, nullptr, 1, h, wd);
            pr.pixels = tc_pixels(w, plan, pr);
            const alcs::TcPrep* t = plan.tc_n ? alcs::tc_find(w, tc_key(w, plan, pr)).get() : nullptr;
            if (!t) t = alcs::tc_any_pointwise(w);
            if (!t) return ALCS_ERR_STATE;
            rc = alcs::tc_run(w, *t, pr, st);
            return rc == ALCS_ERR_UNSUPPORTED ? ALCS_ERR_STATE : rc;
        }
    }
    DeviceInfo di;
    rc = device_info(w->device, &di);
    if (rc) return rc;

    const KernelVariant& v = g_variants[plan.variant].v;
    const int elt = (int)w->elt();
    const int hw = h * wd;
    int hwx = hw;
    const void* xk = x;
    const bool direct = plan.bulk == 2 && direct_rows_ok(hw, elt) && (uintptr_t)x % 8 == 0;
    bool tiled = false;
    if (plan.bulk == 3 && (long long)n * padded_hw(hw, elt) <= (1ll << 30) &&
        tiled_bytes(v, elt, n, w->cin, hw) <= ALCS_NOALLOC_SCRATCH_BYTES) {
        void* scratch = nullptr;
        rc = noalloc_scratch_address(w->device, &scratch);
        if (rc) return rc;
        rc = launch_repack_tiles(v, elt, x, scratch, n, w->cin, h, wd, wd, 1, hw, di.sms, st);
        if (rc) return rc;
        xk = scratch;
        hwx = padded_hw(hw, elt);
        tiled = true;
    }
    if (!tiled && ((size_t)hw * elt) % 16 != 0 && !direct) {
        // rows that cannot be staged with 16-byte copies: repack into the fixed array
        const int hwp = padded_hw(hw, elt);
        const unsigned long long need = (unsigned long long)n * w->cin * hwp * elt;
        if (need > ALCS_NOALLOC_SCRATCH_BYTES || (long long)n * hwp > (1ll << 30)) return ALCS_ERR_TOO_LARGE;
        void* scratch = nullptr;
        rc = noalloc_scratch_address(w->device, &scratch);
        if (rc) return rc;
        const long long rows = (long long)n * w->cin;
        const unsigned blocks = (unsigned)std::min<long long>((rows * (hwp * elt / 16) + 255) / 256, (long long)di.sms * 16);
        // the kernel writes every element of the region it uses, zero padding included, so nothing
        // left behind by an earlier call can leak into this one
        if (elt == 4)
            repack_rows_kernel<float><<<blocks, 256, 0, st>>>(static_cast<const float*>(x), static_cast<float*>(scratch), rows,
                                                              hw, wd, wd, 1, hw, hwp);
        else
            repack_rows_kernel<unsigned short><<<blocks, 256, 0, st>>>(static_cast<const unsigned short*>(x),
                                                                      static_cast<unsigned short*>(scratch), rows,
                                                                      hw, wd, wd, 1, hw, hwp);
        ALCS_CUDA(cudaGetLastError());
        xk = scratch;
        hwx = hwp;
    }

    ConvArgs a;
    a.x = xk; a.y = y; a.bias = bias; a.res = nullptr;
    a.rec = sc->rec; a.slice = sc->slice; a.rowoff = sc->rowoff; a.rowmap = sc->rowmap;
    set_unit_args(a, *sc, v.mma);
    a.err = w->d_err;
    a.rows = w->rows; a.cin = w->cin; a.cout = w->cout; a.hw = hwx; a.hwy = hw;
    a.q_total = n * hwx;
    const int T = 32 * v.p;
    a.n_tiles = (a.q_total + T - 1) / T;
    a.n_rg = sc->n_rg; a.rpg = sc->rpg;
    a.kc = sc->kc; a.nch = sc->nch; a.stages = plan.stages;
    a.relu = (flags & ALCS_RELU) ? 1 : 0;
    a.y_f32 = (flags & ALCS_Y_F32) ? 1 : 0;
    const StageLayout L = stage_layout(v, *sc, elt);
    a.off_rec = L.off_rec; a.off_rowoff = L.off_rowoff; a.stage_bytes = L.stage_bytes;
    if (a.unit) a.off_xch = 16 * alcs::kMaxStages + a.stages * L.stage_bytes;
    int ld = 16;
    while (ld > elt && (((size_t)hwx * elt) % ld || (uintptr_t)xk % ld)) ld >>= 1;
    a.ld_bytes = ld;
    a.bulk = tiled ? 2 : (ld == 16 && plan.bulk == 1) ? 1 : 0;
    a.ros = sc->ros;
    const int vg = (v.p * elt >= 16) ? 16 / elt : v.p;
    a.st_vec = (hwx == hw && hw % vg == 0 && (uintptr_t)y % 16 == 0) ? 1 : 0;
    a.st_grp = hwx % vg == 0 ? 1 : 0;
    if (v.mma && !a.y_f32 && !a.st_vec && ((size_t)hw * elt) % 8 != 0) a.st_grp = 2;
    const long long items = (long long)a.n_tiles * a.n_rg;
    if (items > 0x7fffffffll) return ALCS_ERR_SHAPE;
    const long long grid = std::min<long long>(items, (long long)di.sms * std::max(1, plan.occ));
    void* args[] = {&a};
    ALCS_CUDA(cudaLaunchKernel(v.fn, dim3((unsigned)grid), dim3((v.nw + v.npw) * 32), args, plan.smem, st));
    return ALCS_OK;
}
