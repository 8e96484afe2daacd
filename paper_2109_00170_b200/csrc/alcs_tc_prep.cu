// Host side of the tensor-core path: which output channels form a tile, which columns a tile needs,
// the expanded weight tiles (built on the device from the storage format) and the launch arguments.
#include "alcs_tc_prep.h"

#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <functional>
#include <new>
#include <numeric>

namespace alcs {
void set_cuda_error_text(const char* s);

namespace {

int cuda_fail(cudaError_t e)
{
    set_cuda_error_text(cudaGetErrorString(e));
    (void)cudaGetLastError();
    return e == cudaErrorMemoryAllocation ? ALCS_ERR_ALLOC : ALCS_ERR_CUDA;
}

// Expand the kept blocks into the weight tiles (zeroed before): tile of n channels, chunks of KC
// columns, per chunk the planes one after the other, in a plane [8-column group][channel][8 columns]
// 16-bit values, which is what the MMA's shared-memory descriptor describes.  One warp per block row;
// `place` is where the row's first channel stands (tile * n + channel inside the tile).
template <typename T, int P>
__global__ void expand_kernel(const int* __restrict__ row_ptr, const int* __restrict__ col_idx, const T* __restrict__ vals,
                              const int* __restrict__ place, const TcTile* __restrict__ tiles, const int* __restrict__ inv,
                              int rows, int g, int n, int cols, int taps, int splits, int split_blocks, unsigned char* __restrict__ b)
{
    const int r = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (r >= rows) return;
    const int at = place[r], tile = at / n, n0 = at - tile * n;
    const int beg = row_ptr[r], cnt = row_ptr[r + 1] - beg;
    for (int i = threadIdx.x & 31; i < cnt * g; i += 32) {
        const int blk = i / g, j = i - blk * g;
        int k = col_idx[beg + blk];
        if (inv) k = inv[(size_t)tile * cols + k];
        else if (taps > 1) k = (k / taps / 16 * taps + k % taps) * 16 + k / taps % 16;      // [16 channels][tap]
        // (a split tile: the part that has this block of channels, columns counted from its first)
        const int part = splits > 1 ? k / (16 * taps) / split_blocks : 0;
        k -= part * split_blocks * 16 * taps;
        const TcTile t = tiles[tile * splits + part];
        unsigned char* const bt = b + (size_t)t.b16 * 16;
        constexpr int KC = P == 3 ? kTcKC32 : kTcKC16;
        const int chunk = k / KC, ns = min(KC / 16, t.k16 - KC / 16 * chunk);
        unsigned char* d = bt + (size_t)chunk * (P * KC * 2) * n + ((size_t)((k % KC) >> 3) * n + n0 + j) * 16 + (k & 7) * 2;
        const size_t plane = (size_t)ns * 32 * n;
        const T v = vals[(size_t)beg * g + i];
        if constexpr (P == 3) {
            // three bfloat16 parts, rounded to nearest: v = part 0 + part 1 + part 2 exactly
            __nv_bfloat16 h = __float2bfloat16(v);
            if (__hisinf(h) && !isinf(v)) h = __float2bfloat16_rz(v);
            const float rest = v - __bfloat162float(h);
            const __nv_bfloat16 m = __float2bfloat16(rest);
            *reinterpret_cast<__nv_bfloat16*>(d) = h;
            *reinterpret_cast<__nv_bfloat16*>(d + plane) = m;
            *reinterpret_cast<__nv_bfloat16*>(d + 2 * plane) = __float2bfloat16(rest - __bfloat162float(m));
        } else {
            *reinterpret_cast<T*>(d) = v;
        }
    }
}

// Union of the columns that rows order[i0 .. i1) keep, ascending.
void union_of(const alcs_packed& w, const std::vector<int>& order, int i0, int i1, std::vector<unsigned char>& mark, std::vector<int>& out)
{
    out.clear();
    std::fill(mark.begin(), mark.end(), 0);
    for (int i = i0; i < i1; ++i)
        for (int k = w.row_ptr[order[i]]; k < w.row_ptr[order[i] + 1]; ++k) mark[w.col_idx[k]] = 1;
    for (int c = 0; c < w.cin; ++c)
        if (mark[c]) out.push_back(c);
}

struct Layout {
    std::vector<int> order;
    std::vector<std::vector<int>> cols;      // per tile
    long long k16 = 0;
};

// all: take every column, where a tile keeps any (its column list is then not wanted, only whether it is empty)
void layout_of(const alcs_packed& w, int rows_per_tile, bool sorted, bool all, Layout& L)
{
    L.order.resize(w.rows);
    std::iota(L.order.begin(), L.order.end(), 0);
    if (sorted)
        std::stable_sort(L.order.begin(), L.order.end(), [&](int a, int b) {
            return w.row_ptr[a + 1] - w.row_ptr[a] > w.row_ptr[b + 1] - w.row_ptr[b];
        });
    const int tiles = (w.rows + rows_per_tile - 1) / rows_per_tile;
    L.cols.resize(tiles);
    std::vector<unsigned char> mark(w.cin);
    L.k16 = 0;
    for (int t = 0; t < tiles; ++t) {
        const int r0 = t * rows_per_tile, r1 = std::min(w.rows, r0 + rows_per_tile);
        if (all) {
            if (w.row_ptr[r1] > w.row_ptr[r0]) L.cols[t].push_back(0);
            continue;
        }
        union_of(w, L.order, r0, r1, mark, L.cols[t]);
        L.k16 += (L.cols[t].size() + 15) / 16;
    }
}

// Are the rows so unequal that sorting them by length may empty columns of whole tiles?
bool skewed(const alcs_packed& w)
{
    double s = 0, s2 = 0;
    for (int r = 0; r < w.rows; ++r) {
        const double c = w.row_ptr[r + 1] - w.row_ptr[r];
        s += c;
        s2 += c * c;
    }
    const double mean = s / w.rows;
    return s2 / w.rows - mean * mean > 0.25 * mean * mean + mean;
}

}  // namespace

TcForm tc_find(const alcs_packed* w, const TcKey& key)
{
    auto it = w->tc.find(key.id());
    return it == w->tc.end() ? nullptr : it->second;
}

// Any form whose columns are input channels in order or by a list takes every pointwise layer of stride 1.
const TcPrep* tc_any_pointwise(const alcs_packed* w)
{
    const TcPrep* best = nullptr;
    for (const auto& kv : w->tc)
        if (kv.first[1] <= 1 && kv.first[2] <= 1 && kv.second->splits == 1 && (!best || kv.second->n > best->n)) best = kv.second.get();
    return best;
}

TcForms tc_forms(const alcs_packed* w)
{
    std::lock_guard<std::mutex> lk(w->mu);
    TcForms keys;
    for (const auto& kv : w->tc) keys.push_back(kv.first);
    return keys;
}

bool tc_form_free(const alcs_packed* w, const TcForms& forms, const TcKey& key)
{
    if ((long long)w->rows * w->g * w->cin > kTcMaxWeights) return false;
    int same = 0;
    for (const auto& f : forms) {
        // (a pointwise layer's two forms, of all columns and of lists, go together)
        const bool size = key.kh <= 1 && key.kw <= 1 ? f[1] <= 1 && f[2] <= 1 : f[1] == key.kh && f[2] == key.kw;
        if (size && f[0] == key.n && f[3] == key.splits) return true;
        same += size;
    }
    return same < kTcMaxForms;
}

void tc_release(const alcs_packed* w, const TcForms& before)
{
    std::lock_guard<std::mutex> lk(w->mu);
    for (auto it = w->tc.begin(); it != w->tc.end();) {
        bool keep = it->first[1] > 1 || it->first[2] > 1 || it->first[3] > 1 || it->second.use_count() > 1 ||
                    std::find(before.begin(), before.end(), it->first) != before.end();
        for (const auto& pc : w->plan_cache) keep = keep || pc.second.tc_n == it->first[0];
        it = keep ? std::next(it) : w->tc.erase(it);        // (cudaFree waits for whatever still runs)
    }
}

int tc_prepare(const alcs_packed* w, const TcKey& key, cudaStream_t st, TcForm* out)
{
    {
        std::lock_guard<std::mutex> lk(w->mu);
        if ((*out = tc_find(w, key)) != nullptr) return ALCS_OK;
    }
    int rc = canonical_on_device(w, st);
    if (rc) return rc;
    {
        // the shared-memory attribute belongs to the kernel as loaded on a device
        static std::mutex mu;
        static bool ready[64][3] = {};
        std::lock_guard<std::mutex> lk(mu);
        bool& r = ready[w->device & 63][(int)w->dt];
        if (!r) {
            cudaError_t e = prepare_tc(w->dt);
            if (e == cudaSuccess && w->dt != ALCS_F32) e = prepare_tc16(w->dt);
            if (e != cudaSuccess) return cuda_fail(e);
            r = true;
        }
    }
    std::lock_guard<std::mutex> lk(w->mu);
    if ((*out = tc_find(w, key)) != nullptr) return ALCS_OK;
    try {
        const int P = tc_planes(w->dt), n = key.n, rpt = n / w->g;
        const int taps = std::max(1, key.kh * key.kw);
        const int dense16 = (w->cin / taps + 15) / 16 * taps;
        Layout L;
        layout_of(*w, rpt, false, key.kh > 0, L);
        bool sorted = false;
        if (!key.kh && skewed(*w)) {
            Layout S;
            layout_of(*w, rpt, true, false, S);
            if (S.k16 * 20 <= L.k16 * 19) { L = std::move(S); sorted = true; }
        }
        const int n_tiles = (int)L.cols.size(), splits = key.splits, n_blocks = dense16 / taps, split_blocks = (n_blocks + splits - 1) / splits;
        // A column list costs the converters its loads: without at least a tenth of the steps to save,
        // take all columns in order.
        const bool list = !key.kh && L.k16 * 10 <= (long long)dense16 * n_tiles * 9;
        std::vector<TcTile> tiles;
        std::vector<int> cols, inv, chan, place(w->rows);
        size_t bytes = 0;
        TcPrep p;
        p.n = n;
        p.n_tiles = n_tiles * splits;
        p.splits = splits;
        p.k16_min = 1 << 30;
        for (int t = 0; t < n_tiles; ++t) {
            const int used = (int)L.cols[t].size();
            const int k16 = !list ? (used ? dense16 : 0) : (used + 15) / 16;
            const int list_start = (int)cols.size();
            if (list && used)
                for (int i = 0; i < k16 * 16; ++i) cols.push_back(L.cols[t][std::min(i, used - 1)]);
            if (list) {
                inv.resize((size_t)(t + 1) * w->cin, 0);
                for (int i = 0; i < used; ++i) inv[(size_t)t * w->cin + L.cols[t][i]] = i;
            }
            for (int part = 0; part < splits; ++part) {
                const int first = part * split_blocks;
                const int steps = splits == 1 || k16 == 0 ? k16 : std::max(0, std::min(split_blocks, n_blocks - first)) * taps;
                tiles.push_back({(unsigned)(bytes / 16), steps, list ? list_start : splits > 1 ? first : 0});
                bytes += (size_t)P * steps * 16 * n * 2;
                p.k16.push_back(steps);
                p.k16_max = std::max(p.k16_max, steps);
                p.k16_min = std::min(p.k16_min, steps);
            }
        }
        if (bytes / 16 > 0xffffffffull) return ALCS_ERR_SHAPE;
        for (int i = 0; i < w->rows; ++i) place[L.order[i]] = i / rpt * n + i % rpt * w->g;
        if (sorted || rpt * w->g != n) {
            chan.assign((size_t)n_tiles * n, -1);
            for (int r = 0; r < w->rows; ++r)
                for (int j = 0; j < w->g; ++j)
                    if (r * w->g + j < w->cout) chan[place[r] + j] = r * w->g + j;
        }
        // one device block: weights, then the small arrays (each on a 256-byte boundary); the inverse
        // column map and the places are needed by the expansion only
        auto up = [](size_t v) { return (v + 255) / 256 * 256; };
        const TcSparse sparse = {w->d_row_ptr, w->d_col_idx, w->d_vals, w->g, w->cout, splits};
        const size_t o_tiles = up(bytes), o_sparse = o_tiles + up(tiles.size() * sizeof(TcTile)), o_cols = o_sparse + up(sizeof sparse), o_chan = o_cols + up(cols.size() * 4);
        const size_t o_place = o_chan + up(chan.size() * 4), o_inv = o_place + up(place.size() * 4), end = o_inv + up(inv.size() * 4);
        std::vector<unsigned char> small(end - o_tiles);
        std::memcpy(small.data(), tiles.data(), tiles.size() * sizeof(TcTile));
        std::memcpy(small.data() + (o_sparse - o_tiles), &sparse, sizeof sparse);
        std::memcpy(small.data() + (o_cols - o_tiles), cols.data(), cols.size() * 4);
        std::memcpy(small.data() + (o_chan - o_tiles), chan.data(), chan.size() * 4);
        std::memcpy(small.data() + (o_place - o_tiles), place.data(), place.size() * 4);
        std::memcpy(small.data() + (o_inv - o_tiles), inv.data(), inv.size() * 4);
        unsigned char* d = nullptr;
        cudaError_t e = cudaMalloc(&d, std::max<size_t>(end, 256));
        if (e != cudaSuccess) return cuda_fail(e);
        e = cudaMemcpyAsync(d + o_tiles, small.data(), small.size(), cudaMemcpyHostToDevice, st);
        if (e == cudaSuccess && bytes) e = cudaMemsetAsync(d, 0, bytes, st);
        if (e == cudaSuccess && w->nb > 0) {
            const int* dp = reinterpret_cast<const int*>(d + o_place);
            const int* di = list ? reinterpret_cast<const int*>(d + o_inv) : nullptr;
            const TcTile* dt = reinterpret_cast<const TcTile*>(d + o_tiles);
            const unsigned blocks = (unsigned)((w->rows + 3) / 4);
            if (w->dt == ALCS_F32)
                expand_kernel<float, 3><<<blocks, 128, 0, st>>>(w->d_row_ptr, w->d_col_idx, static_cast<const float*>(w->d_vals), dp, dt, di,
                                                               w->rows, w->g, n, w->cin, taps, splits, split_blocks, d);
            else
                expand_kernel<unsigned short, 1><<<blocks, 128, 0, st>>>(w->d_row_ptr, w->d_col_idx,
                                                                        static_cast<const unsigned short*>(w->d_vals), dp, dt, di,
                                                                        w->rows, w->g, n, w->cin, taps, splits, split_blocks, d);
            e = cudaGetLastError();
        }
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);      // (the host arrays go away; other streams may use the tiles)
        if (e != cudaSuccess) {
            cudaFree(d);
            return cuda_fail(e);
        }
        p.b = d;
        p.tiles = reinterpret_cast<TcTile*>(d + o_tiles);
        p.sparse = reinterpret_cast<TcSparse*>(d + o_sparse);
        p.cols = list ? reinterpret_cast<int*>(d + o_cols) : nullptr;
        p.chan = chan.empty() ? nullptr : reinterpret_cast<int*>(d + o_chan);
        p.uploaded = true;
        *out = TcForm(new TcPrep(p), [](TcPrep* f) {
            cudaFree(f->b);
            delete f;
        });
        w->tc[key.id()] = *out;
    } catch (const std::bad_alloc&) {
        return ALCS_ERR_ALLOC;
    }
    return ALCS_OK;
}

namespace {

// Patch staging of one problem: copy width, elements per channel of the largest patch, input rows taken.
struct PatchPlan {
    int vec_bytes, pitch, row_step;
};

PatchPlan patch_plan(const alcs_packed* w, const TcProblem& p)
{
    const int elt = (int)w->elt();
    PatchPlan r;
    r.vec_bytes = 16;
    while (r.vec_bytes > 2 && ((size_t)p.w_in * elt % r.vec_bytes || (uintptr_t)p.x % r.vec_bytes)) r.vec_bytes >>= 1;
    r.row_step = p.kh == 1 && p.pad == 0 ? p.stride : 1;
    // A tile of 128 consecutive output pixels touches at most (126 / ow) + 2 output rows and (126 / hw) + 2 images.
    const long long hw = (long long)p.oh * p.ow, images = std::min<long long>(p.n, (kTcM - 2) / hw + 2);
    const long long out_rows = std::min<long long>((kTcM - 2) / p.ow + 2, images * p.oh);
    long long rows = r.row_step > 1 ? out_rows : (out_rows - images) * p.stride + images * std::max(p.kh, p.stride);
    rows = std::min(rows, images * p.h_in);
    r.pitch = (int)((rows * p.w_in + 7) / 8 * 8);
    return r;
}

// Blocks of 16 channels per slot: as many as a chunk has steps, if at least three slots then fit.
int patch_blocks(const alcs_packed* w, const TcProblem& p, const PatchPlan& pl, int room)
{
    const int want = std::max(1, tc_kc(w->dt) / 16 / (p.kh * p.kw));
    const long long block = 16ll * pl.pitch * w->elt();
    return (int)std::max(1ll, std::min<long long>(want, room / 3 / block));
}

int patch_room(int dt, int n) { return 227 * 1024 - kTcHeaderBytes - 2 * tc_stage_bytes(dt, n); }

}  // namespace

bool tc_patch_fits(const alcs_packed* w, const TcProblem& p, int n)
{
    if (p.kh * p.kw > 32 || w->cin % (p.kh * p.kw)) return false;
    const PatchPlan pl = patch_plan(w, p);
    return 2 * 16ll * pl.pitch * (long long)w->elt() <= patch_room(w->dt, n);
}

// Small images whose rows do not start on copy boundaries (7x7): a tile takes whole images, of which the columns of
// a chunk are one run of memory, if those runs keep to 16 bytes.  A property of the shape alone, since the form of the
// expanded weights follows from it: an X that does not start on 16 bytes is copied element by element instead.
bool tc_whole_images(const alcs_packed* w, const TcProblem& p)
{
    const size_t elt = w->elt(), row = (size_t)p.oh * p.ow * elt;
    return !p.kh && row % 16 != 0 && (elt == 4 || row % 4 != 0) && row <= kTcM * elt && w->cin % 16 == 0;
}

namespace {

// Bytes of the widest piece (16 ... elt) of rows of `row` bytes that start at `at` that keeps to one row and to its alignment.
int widest(size_t row, const void* at, int elt)
{
    int v = 16;
    while (v > elt && (row % v || (uintptr_t)at % v)) v >>= 1;
    return v;
}

// How alcs_tc16.cu copies X: 16 or 8 bytes at a time; less: rows fetched as they are.
int x_piece(const alcs_packed* w, const TcProblem& p) { return widest((size_t)p.oh * p.ow * w->elt(), p.x, (int)w->elt()); }

}  // namespace

bool tc16_direct(const alcs_packed* w, const TcProblem& p) { return x_piece(w, p) >= 8; }

// Rows fetched as they are: a tile's runs of consecutive pixels, of an image each, in whole 16-byte words.
void tc16_raw(const TcProblem& p, int pixels, int* pitch, int* row)
{
    const long long hw = (long long)p.oh * p.ow, runs = std::min<long long>(std::max(1, p.n), (pixels - 2) / hw + 2);
    *pitch = (int)((std::min<long long>(hw, pixels) * 2 + 14 + 15) / 16 * 16);
    *row = (int)(runs * *pitch);
}

int tc16_raw_bytes(const TcProblem& p, int pixels)
{
    int pitch, row;
    tc16_raw(p, pixels, &pitch, &row);
    return kTc16Chunk * row;
}

namespace {

// The most pixels per tile that a layer can take.
int tc16_most(const alcs_packed* w, const TcProblem& p, int k16_max)
{
    int most = k16_max > kTc16Group ? kTc16Pixels / 2 : kTc16Pixels;
    if (!tc16_direct(w, p)) {
        most = std::min(most, kTc16Raw);
        while (most > 32 && tc16_raw_bytes(p, most) > kTc16RawMost) most -= 32;
    }
    return most;
}

}  // namespace

// The most pixels per tile that are no more than `cap`.
int tc16_capped(const alcs_packed* w, const TcProblem& p, int k16_max, int cap)
{
    return std::max(32, std::min(tc16_most(w, p, k16_max), cap / 32 * 32));
}

// UNSUPPORTED: beyond the kernel's 32-bit offsets, or rows that patch staging cannot copy (see tc_fits, tc_patch_fits).
int tc_fill(const alcs_packed* w, const TcPrep& t, const TcProblem& p, TcLayer* out)
{
    const int taps = std::max(1, p.kh * p.kw);
    if (!tc_fits(w, taps, p.n, (long long)p.h_in * p.w_in, (long long)p.oh * p.ow) || (p.kh && !tc_patch_fits(w, p, t.n)))
        return ALCS_ERR_UNSUPPORTED;
    TcLayer& y = *out;
    y.x = p.x; y.y = p.y; y.bias = p.bias; y.res = p.res;
    y.b = t.b; y.tiles = t.cols || t.k16_min != t.k16_max || t.splits > 1 ? t.tiles : nullptr; y.k16 = t.k16_max; y.cols = t.cols; y.chan = t.chan; y.sparse = t.sparse;
    y.err = w->d_err;
    y.hw = tc_div(p.oh * p.ow);
    y.q = p.n * y.hw.d;
    y.n_tiles = tc_div(t.n_tiles);
    // tiles of unequal work: all pixel tiles of the heaviest channel tile first, so that the light ones
    // fill the end; otherwise the channel tiles of a pixel tile run together and share its reads of X
    y.tile_major = t.k16_max > t.k16_min + t.k16_min / 4 ? 1 : 0;
    y.n = t.n;
    y.cin = p.kh ? w->cin / (p.kh * p.kw) : w->cin;
    y.cout = w->cout;
    y.hw_in = p.h_in * p.w_in; y.w_in = p.w_in; y.h_in = p.h_in;
    y.ow = tc_div(p.ow); y.oh = p.oh; y.stride = p.stride; y.pad = p.pad;
    y.kh = p.kh; y.kw = p.kw;
    y.n_img = p.n;
    y.images = 0;
    const int elt = (int)w->elt();
    y.n_px = 0;
    if (p.pixels) {
        const int e = (p.flags & ALCS_Y_F32) ? 4 : 2;
        const size_t row = (size_t)y.hw.d * e;
        const int v = x_piece(w, p);
        y.vec_bytes = v >= 8 ? v : kTcRaw;
        y.y_vec = widest(row, p.y, e);
        y.res_vec = p.res ? widest(row, p.res, e) : 16;
        y.ppt = tc16_capped(w, p, t.k16_max, p.pixels);      // (the weights, or an X that starts anywhere, may allow less than was planned)
        if (y.vec_bytes == kTcRaw) {
            tc16_raw(p, y.ppt, &y.raw_pitch, &y.raw_row);
            y.raw_bytes = kTc16Chunk * y.raw_row;
        }
        y.n_px = y.ppt;
        y.px_tiles = tc_div((y.q + y.ppt - 1) / y.ppt);
        y.relu = (p.flags & ALCS_RELU) ? 1 : 0;
        y.y32 = e == 4;
        return ALCS_OK;
    }
    if (p.kh) {
        const PatchPlan pl = patch_plan(w, p);
        y.taps = tc_div(p.kh * p.kw); y.kwd = tc_div(p.kw);
        y.vec_bytes = pl.vec_bytes;
        y.w_vec = tc_div(p.w_in * elt / pl.vec_bytes);
        y.row_step = pl.row_step;
        y.pitch = pl.pitch;
        y.blocks = patch_blocks(w, p, pl, patch_room(w->dt, t.n));
    } else {
        // the widest copy that keeps to one image and to its alignment
        int vb = 16;
        while (vb > elt && (((size_t)y.hw.d * elt) % vb || (uintptr_t)p.x % vb)) vb >>= 1;
        y.vec_bytes = vb == 16 || (elt == 2 && vb > elt) ? vb : 0;      // (8 bytes of fp32: as single elements)
        if (!t.cols && tc_whole_images(w, p) && (uintptr_t)p.x % 16 == 0) y.images = kTcM / y.hw.d;
    }
    y.ppt = y.images ? y.images * y.hw.d : kTcM;
    y.px_tiles = tc_div((y.q + y.ppt - 1) / y.ppt);
    y.relu = (p.flags & ALCS_RELU) ? 1 : 0;
    y.y32 = (p.flags & ALCS_Y_F32) ? 1 : 0;
    return ALCS_OK;
}

namespace {

// What one item costs, in microseconds: least-squares fits (of the logarithm) to 2,500 launches of random shapes, types and
// densities on one B200; the median error is 7 %, one in ten is off by more than 25 %.
struct TileFit {
    double ramp;                 // a launch, with its first and last item's latencies that nothing overlaps
    double mma, mma_n;           // a 16-column step on the tensor cores: mma + mma_n * channels
    double list;                 // a step that follows a column list, beyond its copies
    double store, store_n;       // bias, activation and stores: store + store_n * channels, ...
    double sorted, res;          // ... store_n times this where every row's channel is looked up, and with a residual
    double tail;                 // share of a tile's stores behind the last item
    double copy[5], first[5];    // a step's copies, and the first chunk's latency per step: 16, 8, 4 bytes, elements, whole images
};
constexpr TileFit kTileFit[2] = {
    {2.0, 0.217, 0.0011, 0.062, 0.75, 0.0100, 4.2, 8.0, 0.53, {0.258, 0.510, 0.510, 0.510, 0.317}, {0.75, 1.51, 1.51, 1.51, 0.38}},
    {2.15, 0.097, 0.00096, 0.089, 0.745, 0.0086, 6.0, 9.0, 0.91, {0.187, 0.190, 0.282, 0.467, 0.108}, {0.36, 0.49, 0.59, 1.74, 0.0}}};
// Patch staging: a step on the tensor cores; reading and splitting a step's values; one copy instruction of a warp.
constexpr double kPatchRamp = 3.75, kPatchMma[2] = {0.195, 0.097}, kPatchMmaN = 0.00098, kPatchConvert[2] = {0.233, 0.15}, kPatchCopy = 0.0231,
                 kPatchFirst = 0.24;
constexpr double kBytesPerUs = 7.0e6;

int copy_kind(const alcs_packed* w, const TcProblem& p)
{
    if (tc_whole_images(w, p)) return 4;
    const int v = x_piece(w, p);
    return v == 16 ? 0 : w->dt == ALCS_F32 || v < 4 ? 3 : v == 8 ? 1 : 2;
}

double store_us(const alcs_packed* w, const TcProblem& p, int n, bool sorted)
{
    const TileFit& f = kTileFit[w->dt != ALCS_F32];
    return f.store + f.store_n * n * std::max(sorted ? f.sorted : 1.0, p.res ? f.res : 1.0);
}

// X, Y and the residual, once.
double layer_bytes(const alcs_packed* w, const TcProblem& p)
{
    const double q = (double)std::max(1, p.n) * p.oh * p.ow, y_elt = (p.flags & ALCS_Y_F32) ? 4.0 : (double)w->elt();
    return q * (w->cin * (double)w->elt() + w->cout * y_elt * (p.res ? 2.0 : 1.0));
}

// Copy instructions of a warp for one block of 16 channels of the widest patch, of an aligned X.
double patch_copies(const alcs_packed* w, TcProblem p)
{
    p.x = nullptr;
    const PatchPlan pl = patch_plan(w, p);
    return 16.0 * pl.pitch * (double)w->elt() / pl.vec_bytes / 32.0;
}

// Channel tiles as tc_prepare would lay them out, from the lengths of the block rows: a tile of rows that keep a share
// d_r of the columns at random keeps 1 - prod(1 - d_r) of them.
struct TileGuess {
    std::vector<int> k16;
    bool list = false, sorted = false;
};

TileGuess guess_tiles(const alcs_packed* w, const TcProblem& p, int n)
{
    const int rpt = n / w->g, tiles = (w->rows + rpt - 1) / rpt, dense16 = (w->cin + 15) / 16;
    std::vector<int> len(w->rows);
    for (int r = 0; r < w->rows; ++r) len[r] = w->row_ptr[r + 1] - w->row_ptr[r];
    auto steps = [&](std::vector<int>& out) {
        long long sum = 0;
        out.resize(tiles);
        for (int t = 0; t < tiles; ++t) {
            double none = 1.0;
            int any = 0;
            for (int r = t * rpt; r < std::min(w->rows, (t + 1) * rpt); ++r) {
                none *= 1.0 - (double)len[r] / w->cin;
                any |= len[r];
            }
            out[t] = any ? std::max(1, (int)std::ceil(w->cin * (1.0 - none) / 16.0)) : 0;
            sum += out[t];
        }
        return sum;
    };
    TileGuess g;
    long long sum = steps(g.k16);
    const bool lists = !p.kh && !tc_whole_images(w, p);
    if (lists && skewed(*w)) {
        std::vector<int> k16;
        std::sort(len.begin(), len.end(), std::greater<int>());
        const long long s = steps(k16);
        if (s * 20 <= sum * 19) { g.k16.swap(k16); g.sorted = true; sum = s; }
    }
    g.list = lists && sum * 10 <= (long long)dense16 * tiles * 9;
    if (!g.list)
        for (int& k : g.k16) k = k ? dense16 : 0;
    return g;
}

}  // namespace

double tc_tile_us(const alcs_packed* w, const TcProblem& p, int n, int k16, bool list, bool sorted)
{
    const int half = w->dt != ALCS_F32;
    const TileFit& f = kTileFit[half];
    const double store = store_us(w, p, n, sorted);
    if (k16 == 0) return 1.5 * store;
    if (p.kh)
        return k16 * std::max({kPatchConvert[half], kPatchMma[half] + kPatchMmaN * n, kPatchCopy * patch_copies(w, p) / (p.kh * p.kw)}) + store;
    const double work = k16 * std::max(f.copy[copy_kind(w, p)] + (list ? f.list : 0.0), f.mma + f.mma_n * n);
    // (the epilogue adds up the chunk sums of a long item and then stores: a residual's loads are not hidden there)
    return p.res && k16 * 16 > 2 * tc_kc(w->dt) ? work + 0.65 * store : std::max(work, store);
}

// An item among those of other layers in one launch, where staging, tensor cores and stores of different items overlap: what
// the list of a merged launch is made from (ResNet-50's layers in fp16: 99 us; dealt by tc_tile_us, 108).
double tc_merged_item_us(int dt, int n, int k16)
{
    const int nch = (k16 * 16 + tc_kc(dt) - 1) / tc_kc(dt);
    const double chunk = dt == ALCS_F32 ? std::max(0.95, 0.1 + 0.0096 * n) : std::max(0.9, 0.3 + 0.006 * n);
    return nch * chunk + 0.3 + 0.005 * n;
}

std::vector<double> tc_tiles_us(const alcs_packed* w, const TcProblem& p, int n)
{
    const TileGuess g = guess_tiles(w, p, n);
    std::vector<double> us;
    for (int k16 : g.k16) us.push_back(tc_tile_us(w, p, n, k16, g.list, g.sorted));
    return us;
}

double tc_layer_us(const alcs_packed* w, const TcProblem& p, int n, int sms)
{
    const TileFit& f = kTileFit[w->dt != ALCS_F32];
    const TileGuess g = guess_tiles(w, p, n);
    const long long hw = (long long)p.oh * p.ow, q = hw * std::max(1, p.n);
    const int ppt = !p.kh && tc_whole_images(w, p) ? (int)(kTcM / hw * hw) : kTcM, kind = copy_kind(w, p);
    const double px = (double)((q + ppt - 1) / ppt);
    double sum = 0, longest = 0;
    int k_max = 0;
    for (int k16 : g.k16) {
        const double t = tc_tile_us(w, p, n, k16, g.list, g.sorted);
        sum += t;
        longest = std::max(longest, t);
        k_max = std::max(k_max, k16);
    }
    const double rounds = std::ceil(px * g.k16.size() / sms);
    const double main = std::max(rounds * sum / g.k16.size(), longest);
    const double bytes = layer_bytes(w, p);
    if (p.kh) return std::max(kPatchRamp + main + kPatchFirst * std::min(k_max, 4), kPatchRamp + bytes / kBytesPerUs);
    const double first = f.first[kind] * std::min(k_max, tc_kc(w->dt) / 16);
    return std::max(f.ramp + main + first + f.tail * store_us(w, p, n, g.sorted), f.ramp + bytes / kBytesPerUs);
}

// alcs_tc16.cu: least-squares fits (of the logarithm) to 1,087 launches of random shapes, densities and tile sizes on one B200; median
// error 9 %, and the tile sizes they choose take 2 % more than the best of those measured.  A chunk: by how X is copied (16 bytes,
// 8, rows fetched as they are), or by its bytes; the stores of 128 pixels by their width.
double tc16_item_us(const alcs_packed* w, const TcProblem& p, int n, int k16, int pixels)
{
    const size_t hw = (size_t)p.oh * p.ow, e = (p.flags & ALCS_Y_F32) ? 4 : 2;
    const int v = x_piece(w, p);
    const double px = pixels, store_px[4] = {0.68 * e / 2.0, 0.96, 1.5, 2.14};
    const int width = hw * e % 16 == 0 ? 0 : hw * e % 8 == 0 ? 1 : hw * e % 4 == 0 ? 2 : 3;
    const double store = 1.25 + px / 128.0 * store_px[width] * (p.res ? 3.0 : 1.0);
    double chunk = v == 16 ? 0.41 + 0.00027 * px : v == 8 ? 0.41 + 0.0024 * px : 2.6;
    if (k16 * 16 < w->cin) chunk += 0.1;        // (a column list)
    chunk = std::max(chunk, 0.0024 * px + 0.0019 * n);
    return std::max((k16 + 3) / 4 * chunk, store);
}

double tc16_layer_us(const alcs_packed* w, const TcProblem& p, int n, int sms, int cap, int* pixels)
{
    const std::vector<int> k16 = tc_tile_steps(w, p, n);
    const long long q = (long long)std::max(1, p.n) * p.oh * p.ow;
    const int k_max = k16.empty() ? 0 : *std::max_element(k16.begin(), k16.end());
    const bool raw = !tc16_direct(w, p);
    double best = 0;
    *pixels = 0;
    const int most = cap ? tc16_capped(w, p, k_max, cap) : tc16_most(w, p, k_max);
    for (int px = most; px >= (cap ? most : 32); px -= 32) {
        const double tiles = (double)((q + px - 1) / px);
        double sum = 0, longest = 0;
        for (int k : k16) {
            const double us = tc16_item_us(w, p, n, k, px);
            sum += us;
            longest = std::max(longest, us);
        }
        const double rounds = std::ceil(tiles * k16.size() / sms);
        const double us = 2.3 + (raw ? 3.0 : 0.0) + std::max(rounds * sum / k16.size(), longest) + 1.2 * std::min(longest, 1.25 + px / 128.0 * 0.7);
        if (!*pixels || us < best * 0.98) { best = us; *pixels = px; }
    }
    const double bytes = layer_bytes(w, p);
    return std::max(best, 2.0 + bytes / kBytesPerUs);
}

std::vector<int> tc_tile_steps(const alcs_packed* w, const TcProblem& p, int n) { return guess_tiles(w, p, n).k16; }

// Number items and choose the ring depth for the a.n_layers layers filled in.
int tc_finish(const alcs_packed* w, TcArgs<kTcMaxLayers>& a, bool patch)
{
    int sms = 0, smem = 0;
    const int rc = device_limits(w->device, &sms, &smem);
    if (rc) return rc;
    int n = 16;
    long long items = 0;
    for (int i = 0; i < a.n_layers; ++i) {
        a.layer[i].first_item = (int)items;
        items += (long long)a.layer[i].n_tiles.d * a.layer[i].px_tiles.d;
        n = std::max(n, a.layer[i].n);
    }
    if (items > 0x7fffffffll) return ALCS_ERR_SHAPE;
    a.n_items = (int)items;
    a.sched = nullptr;
    a.raw_slots = a.raw_bytes = 0;
    if (a.layer[0].n_px) {
        int px = 32;
        for (int i = 0; i < a.n_layers; ++i) px = std::max(px, a.layer[i].n_px);
        a.slots = 0;
        a.slot_bytes = tc16_weight_bytes(n);
        a.stage_bytes = tc16_stage_bytes(n, px);
        int room = std::min(smem, 227 * 1024) - kTc16Fixed;
        for (int i = 0; i < a.n_layers; ++i)
            if (a.layer[i].vec_bytes == kTcRaw) a.raw_bytes = std::max(a.raw_bytes, (a.layer[i].raw_bytes + 127) / 128 * 128);
        if (a.raw_bytes) {      // two stages, then slots, as many as there is room for: what is in flight is there
            a.raw_slots = std::min(4, (room - 2 * a.stage_bytes) / a.raw_bytes);
            if (a.raw_slots < 1) return ALCS_ERR_UNSUPPORTED;
            room -= a.raw_slots * a.raw_bytes;
        }
        a.stages = std::min(8, room / a.stage_bytes);
        return a.stages >= 2 ? ALCS_OK : ALCS_ERR_UNSUPPORTED;
    }
    a.stage_bytes = tc_stage_bytes(w->dt, n);
    int room = std::min(smem, 227 * 1024) - kTcHeaderBytes;
    a.slots = a.slot_bytes = 0;
    if (patch) {
        for (int i = 0; i < a.n_layers; ++i) a.slot_bytes = std::max(a.slot_bytes, a.layer[i].blocks * 16 * a.layer[i].pitch * (int)w->elt());
        a.slots = std::min(4, (room - 2 * a.stage_bytes) / a.slot_bytes);
        if (a.slots < 2) return ALCS_ERR_UNSUPPORTED;
        room -= a.slots * a.slot_bytes;
    } else {
        room -= kTcRingBytes;
    }
    // (an even number: of two MMA issuers each then always meets the same stages)
    a.stages = ~1 & std::min(8, room / a.stage_bytes);
    return a.stages >= 2 ? ALCS_OK : ALCS_ERR_UNSUPPORTED;
}

int tc_launch(const alcs_packed* w, const TcArgs<kTcMaxLayers>& a, bool patch, cudaStream_t st)
{
    int sms = 0, smem = 0;
    const int rc = device_limits(w->device, &sms, &smem);
    if (rc) return rc;
    const cudaError_t e = a.layer[0].n_px ? launch_tc16(w->dt, a, std::min(a.n_items, sms), st) : launch_tc(w->dt, patch, a, std::min(a.n_items, sms), st);
    return e == cudaSuccess ? ALCS_OK : cuda_fail(e);
}

int tc_run(const alcs_packed* w, const TcPrep& t, const TcProblem& p, cudaStream_t st)
{
    TcArgs<kTcMaxLayers> a;
    a.n_layers = 1;
    int rc = tc_fill(w, t, p, &a.layer[0]);
    if (!rc) rc = tc_finish(w, a, p.kh > 0);
    return rc ? rc : tc_launch(w, a, p.kh > 0, st);
}

// The width, and the number of parts the channels are split into, that take the least time: rounds of items over
// the SMs, and for split columns the partial sums' way through memory and one more launch (5 us, then 2.8 TB/s).
// Small batches leave most SMs idle otherwise: one 7 x 7 image of 512 channels is a chain of 72 chunks.
double tc_conv2d_choose(const alcs_packed* w, const TcProblem& p, int sms, int* n_out, int* splits_out)
{
    const long long hw = (long long)p.oh * p.ow;
    const int taps = p.kh * p.kw;
    *n_out = 0;
    *splits_out = 1;
    if (!tc_fits(w, taps, p.n, (long long)p.h_in * p.w_in, hw)) return 0;
    const int blocks = (w->cin / taps + 15) / 16;
    const long long px = (p.n * hw + kTcM - 1) / kTcM;
    const TcForms forms = tc_forms(w);
    double best = 0;
    for (int want = kTcMaxN; want >= 16; want -= 16) {
        const int want_tiles = (w->cout + want - 1) / want, v = ((w->cout + want_tiles - 1) / want_tiles + 15) / 16 * 16;
        if (!tc_patch_fits(w, p, v)) continue;
        const int tiles = (w->cout + v - 1) / v;
        for (int s = 1; s <= std::min(8, blocks); ++s) {
            const int part = (blocks + s - 1) / s;
            if ((blocks + part - 1) / part != s) continue;
            const double bytes = (double)s * tiles * v * p.n * hw * 4;
            if (s > 1 && (bytes > (32 << 20) || (double)p.n * hw * w->cout > 1e9)) break;
            if (!tc_form_free(w, forms, {v, p.kh, p.kw, s})) continue;
            const long long items = px * tiles * s;
            const double us = kPatchRamp + kPatchFirst * std::min(part * taps, 4) +
                              (double)((items + sms - 1) / sms) * tc_tile_us(w, p, v, part * taps, false, false) + (s > 1 ? 5.2 + bytes / 2.8e6 : 0.0);
            if (*n_out == 0 || us < best * 0.95) { *n_out = v; *splits_out = s; best = us; }
        }
    }
    return best;
}

int tc_conv2d(const alcs_packed* w, const TcProblem& p, int n, int splits, cudaStream_t st)
{
    const long long hw = (long long)p.oh * p.ow;
    int sms = 0, smem = 0;
    int rc = device_limits(w->device, &sms, &smem);
    if (rc) return rc;
    TcForm t;
    rc = tc_prepare(w, {n, p.kh, p.kw, splits}, st, &t);
    if (rc) return rc;
    if (splits == 1) return tc_run(w, *t, p, st);
    const int tiles = t->n_tiles / splits;
    void* part = nullptr;
    rc = scratch_alloc(w->device, (size_t)t->n_tiles * n * p.n * hw * 4, st, &part);
    if (rc) return rc;
    TcProblem q = p;
    q.y = part;
    q.bias = nullptr;
    q.flags = 0;
    TcArgs<kTcMaxLayers> a;
    a.n_layers = 1;
    rc = tc_fill(w, *t, q, &a.layer[0]);
    a.layer[0].cout = t->n_tiles * n;       // every part of a tile writes rows of its own
    if (!rc) rc = tc_finish(w, a, true);
    if (!rc) rc = tc_launch(w, a, true, st);
    if (!rc) {
        TcReduce r;
        r.part = static_cast<const float*>(part); r.y = static_cast<float*>(p.y); r.bias = p.bias;
        r.n = p.n; r.splits = splits; r.tiles = tiles; r.cout = w->cout; r.relu = (p.flags & ALCS_RELU) ? 1 : 0;
        r.hw = tc_div((int)hw); r.width = tc_div(n);
        r.total = (long long)p.n * w->cout * hw;
        const cudaError_t e = launch_tc_reduce(r, sms, st);
        if (e != cudaSuccess) rc = cuda_fail(e);
    }
    scratch_free(part, st);
    return rc;
}

// 32-bit arithmetic of the kernel: element offsets into X, byte offsets inside the images one tile touches.  fp32 weights that
// are not finite cannot be split into parts that add up to them.
bool tc_fits(const alcs_packed* w, int taps, long long n, long long hw_in, long long hw)
{
    return n * hw_in * (w->cin / taps) < (1ll << 31) - 4096 && ((long long)kTcM / std::max(1ll, hw) + 2) * hw * w->cout * 4 < (1ll << 32) &&
           w->cin < (1 << 20) && n * hw <= (1ll << 30) && (w->finite || w->dt != ALCS_F32);
}

}  // namespace alcs
