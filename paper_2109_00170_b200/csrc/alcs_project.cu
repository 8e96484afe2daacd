// Latency model (paper, Section 3.3) and projection with bisection (Section 3.4, Algorithm 1).
//
// Host part: the linear interpolation over a layer's measured (non-zero count, run time) pairs and
// the network sum.  Algorithm 1 runs on the device from end to end, in one stream and with one wait at the
// end: the ranking key of every group of g adjacent filters (its squared L2 norm), the ranking of all
// groups of all layers (a radix sort from the CUDA toolkit's CUB, a library primitive), per-bucket layer
// histograms of the ranked list, the search over the length of the kept prefix (one thread block, five
// bisection steps per round), and the mask and the projected tensors from the key of the last kept group.
#include <cuda_runtime.h>

#include <cub/device/device_radix_sort.cuh>

#include <algorithm>
#include <cstdint>
#include <mutex>
#include <vector>

#include "alcs_internal.h"

namespace alcs {
void set_cuda_error_text(const char* s);
}

namespace {

#define ALCS_CUDA(call)                                        \
    do {                                                       \
        cudaError_t e_ = (call);                               \
        if (e_ != cudaSuccess) {                               \
            alcs::set_cuda_error_text(cudaGetErrorString(e_)); \
            (void)cudaGetLastError();                          \
            return ALCS_ERR_CUDA;                              \
        }                                                      \
    } while (0)

// Eq. for T^(s): t_1 + sum_i delta_i alpha_i min(k_{i+1} - k_i, s - k_i), evaluated term by term.
double interpolate(const alcs_latency_table& tab, int64_t s)
{
    double total = tab.t[0];
    for (int i = 0; i + 1 < tab.n_knots; ++i) {
        const double delta = s >= tab.k[i] ? 1.0 : 0.0;
        const double width = (double)tab.k[i + 1] - (double)tab.k[i];
        const double alpha = (tab.t[i + 1] - tab.t[i]) / width;
        total += delta * alpha * std::min(width, (double)s - (double)tab.k[i]);
    }
    return total;
}

int check_table(const alcs_latency_table* tab)
{
    if (!tab || tab->n_knots < 2 || !tab->k || !tab->t) return ALCS_ERR_INVALID_ARG;
    for (int i = 0; i + 1 < tab->n_knots; ++i)
        if (tab->k[i + 1] <= tab->k[i]) return ALCS_ERR_INVALID_ARG;
    return ALCS_OK;
}

// Layers of one launch of the per-group kernels.
constexpr int kLayersPerLaunch = 64;
struct LayerTable {
    int n_layers, g;
    long long total;                        // groups in this launch
    const float* u[kLayersPerLaunch];
    float* out[kLayersPerLaunch];           // may be null
    int cout[kLayersPerLaunch], cols[kLayersPerLaunch];
    long long off[kLayersPerLaunch + 1];    // first group of each layer, counted over all layers of the call
};

// Layer of group i (binary search over the layers' group offsets).
__device__ __forceinline__ int layer_of_group(const long long* off, int n_layers, long long i)
{
    int lo = 0, hi = n_layers - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (off[mid] <= i) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// key[group] = sum over the g filters of the group of the squared element: fp32, one rounded
// multiply and one rounded add per element, filters in ascending order (no fused multiply-add, so
// that the ranking is reproducible bit for bit).  Group (r, c) of a [cout][cols] layer covers
// elements (r*g + j, c); a missing filter of a ragged last group counts as zero.  Also writes the
// identity permutation that the sort carries along.  One launch for (up to 64) layers: reads the weights
// once, at the memory's rate for large networks; small ones are a launch's latency.
__global__ void group_keys_kernel(const __grid_constant__ LayerTable t, unsigned* __restrict__ keys, unsigned* __restrict__ idx)
{
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < t.total; i += (long long)gridDim.x * blockDim.x) {
        const long long id = t.off[0] + i;
        const int l = layer_of_group(t.off, t.n_layers, id);
        const int cols = t.cols[l];
        const unsigned in = (unsigned)(id - t.off[l]);
        const int r = in / (unsigned)cols, c = in - r * cols;
        const float* p = t.u[l] + (size_t)r * t.g * cols + c;
        const int nj = min(t.g, t.cout[l] - r * t.g);
        float acc = 0.0f;
#pragma unroll 8
        for (int j = 0; j < nj; ++j) {
            const float v = __ldg(p + (size_t)j * cols);
            acc = __fadd_rn(acc, __fmul_rn(v, v));
        }
        keys[id] = __float_as_uint(acc);      // non-negative floats order like their bit patterns
        idx[id] = (unsigned)id;
    }
}

// The result: a group is kept if it ranks before the n_keep-th, i.e. if its key is larger than that of the last
// kept group, or equal and its number not larger (the sort is stable).  u_out = u where kept, +0 elsewhere.
__global__ void apply_kernel(const __grid_constant__ LayerTable t, const unsigned* __restrict__ keys, const unsigned* __restrict__ ranked_keys,
                             const unsigned* __restrict__ ranked_idx, const long long* __restrict__ n_keep, uint8_t* __restrict__ mask)
{
    const long long n = *n_keep;
    const unsigned last_key = n > 0 ? ranked_keys[n - 1] : 0u, last_id = n > 0 ? ranked_idx[n - 1] : 0u;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < t.total; i += (long long)gridDim.x * blockDim.x) {
        const long long id = t.off[0] + i;
        const unsigned k = keys[id];
        const bool keep = n > 0 && (k > last_key || (k == last_key && (unsigned)id <= last_id));
        mask[id] = keep ? 1 : 0;
        const int l = layer_of_group(t.off, t.n_layers, id);
        if (!t.out[l]) continue;
        const int cols = t.cols[l];
        const unsigned in = (unsigned)(id - t.off[l]);
        const int r = in / (unsigned)cols, c = in - r * cols;
        const size_t at = (size_t)r * t.g * cols + c;
        const int nj = min(t.g, t.cout[l] - r * t.g);
#pragma unroll 4
        for (int j = 0; j < nj; ++j) t.out[l][at + (size_t)j * cols] = keep ? t.u[l][at + (size_t)j * cols] : 0.0f;
    }
}

constexpr int kMaxLayers = 4096;
constexpr long long kRankBucket = 1024;

// layer_of[i] = layer of the i-th ranked group; hist[b][l] = how many of the ranked entries
// b*kRankBucket .. (b+1)*kRankBucket - 1 belong to layer l (one thread block per bucket).
__global__ void ranked_layers_kernel(const unsigned* __restrict__ idx, long long total, const long long* __restrict__ off, int n_layers,
                                     unsigned short* __restrict__ layer_of, unsigned* __restrict__ hist)
{
    extern __shared__ unsigned int h[];
    for (int i = threadIdx.x; i < n_layers; i += blockDim.x) h[i] = 0;
    __syncthreads();
    const long long b0 = (long long)blockIdx.x * kRankBucket;
    const long long b1 = b0 + kRankBucket < total ? b0 + kRankBucket : total;
    for (long long i = b0 + threadIdx.x; i < b1; i += blockDim.x) {
        const int l = layer_of_group(off, n_layers, idx[i]);
        layer_of[i] = (unsigned short)l;
        atomicAdd(&h[l], 1u);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < n_layers; i += blockDim.x) hist[(size_t)blockIdx.x * n_layers + i] = h[i];
}

// hist[b][l] becomes the number of entries of layer l in the buckets before b (one thread block per layer, 1024
// buckets per round: a warp per layer took 16 us for 767 buckets).
__global__ void __launch_bounds__(1024) prefix_kernel(unsigned* __restrict__ hist, long long n_buckets, int n_layers)
{
    __shared__ unsigned sums[32];
    const int l = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned before = 0;
    for (long long b0 = 0; b0 < n_buckets; b0 += 1024) {
        const long long b = b0 + threadIdx.x;
        const unsigned v = b < n_buckets ? hist[(size_t)b * n_layers + l] : 0u;
        unsigned s = v;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const unsigned o = __shfl_up_sync(0xffffffffu, s, d);
            if (lane >= d) s += o;
        }
        if (lane == 31) sums[warp] = s;
        __syncthreads();
        unsigned w = sums[lane];
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const unsigned o = __shfl_up_sync(0xffffffffu, w, d);
            if (lane >= d) w += o;
        }
        const unsigned mine = warp ? __shfl_sync(0xffffffffu, w, warp - 1) : 0u;
        if (b < n_buckets) hist[(size_t)b * n_layers + l] = before + mine + s - v;
        before += __shfl_sync(0xffffffffu, w, 31);
        __syncthreads();
    }
}

// What the search returns; written to page-locked host memory.
struct SearchResult {
    long long n_keep, lo, hi;
    int iters;
    double latency;
};

struct SearchArgs {
    const unsigned short* layer_of;
    const unsigned* prefix;             // [bucket][layer]
    const int* first_knot;              // [n_layers + 1]
    const long long* k;                 // knots of all layers
    const double* t;
    const double* alpha;                // slope of the interval that starts at a knot
    long long total;
    int n_layers, g, depth;
    double tau, t_budget, eps;
    long long* n_keep;                  // device
    SearchResult* result;               // host
    long long* kept;                    // host, [n_layers]
};

// T(W) of "the n best-ranked groups kept", by one warp: per-layer counts from the bucket's prefix and a walk over
// at most one bucket, then Eq. for T^(s) term by term and the sum over the layers in order, every operation
// rounded as the host's (no fused multiply-add).
__device__ double latency_of_top(const SearchArgs& a, long long n, unsigned* counts, double* terms, int lane)
{
    const long long bk = n / kRankBucket < (a.total + kRankBucket - 1) / kRankBucket ? n / kRankBucket : (a.total + kRankBucket - 1) / kRankBucket - 1;
    __syncwarp();
    for (int l = lane; l < a.n_layers; l += 32) counts[l] = a.prefix[(size_t)bk * a.n_layers + l];
    __syncwarp();
    for (long long i = bk * kRankBucket + lane; i < n; i += 32) atomicAdd(&counts[a.layer_of[i]], 1u);
    __syncwarp();
    double t = a.tau;
    for (int l0 = 0; l0 < a.n_layers; l0 += 32) {
        const int l = l0 + lane;
        if (l < a.n_layers) {
            const long long s = (long long)counts[l] * a.g;
            const int f = a.first_knot[l], e = a.first_knot[l + 1] - 1;
            double sum = a.t[f];
            for (int i = f; i < e; ++i) {
                const double delta = s >= a.k[i] ? 1.0 : 0.0;
                const double width = __dsub_rn((double)a.k[i + 1], (double)a.k[i]);
                const double in = __dsub_rn((double)s, (double)a.k[i]);
                sum = __dadd_rn(sum, __dmul_rn(__dmul_rn(delta, a.alpha[i]), in < width ? in : width));
            }
            terms[lane] = sum;
        }
        __syncwarp();
        for (int i = 0; i < min(32, a.n_layers - l0); ++i) t = __dadd_rn(t, terms[i]);
        __syncwarp();
    }
    return t;
}

// Search (Section 3.4, Algorithm 1): the bracket [lo, hi] of prefix lengths is halved until the latencies of its
// two ends are within eps of each other or it has width 1.  A round evaluates every prefix length the next
// `depth` steps may ask for (2^depth - 1, a warp each), then the steps are taken one by one as printed:
// a step costs a fifth of a round trip through the ranked list instead of a whole one.
__global__ void __launch_bounds__(1024) search_kernel(const __grid_constant__ SearchArgs a)
{
    extern __shared__ __align__(16) unsigned char shared[];
    __shared__ double node[32];
    __shared__ long long bracket[2];
    __shared__ double ends[2];
    __shared__ int state[2];                // iterations, finished
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    double* const terms = reinterpret_cast<double*>(shared) + warp * 32;
    unsigned* const counts = reinterpret_cast<unsigned*>(shared + (blockDim.x >> 5) * 256) + (size_t)warp * a.n_layers;
    if (warp < 2) {
        const double t = latency_of_top(a, warp ? a.total : 0, counts, terms, lane);
        if (lane == 0) { ends[warp] = t; bracket[warp] = warp ? a.total : 0; }
    }
    if (threadIdx.x == 0) state[0] = state[1] = 0;
    __syncthreads();
    for (;;) {
        if (threadIdx.x == 0) state[1] = !(ends[1] - ends[0] > a.eps && bracket[1] - bracket[0] > 1);
        __syncthreads();
        if (state[1]) break;
        const int id = warp + 1;            // node of the tree of possible steps: 1 is the next one, 2i / 2i + 1 follow "lower half" / "upper half"
        if (id < 1 << a.depth) {
            long long lo = bracket[0], hi = bracket[1];
            for (int bit = 30 - __clz(id); bit >= 0; --bit) {
                const long long mid = (lo + hi) / 2;
                if ((id >> bit) & 1) lo = mid; else hi = mid;
            }
            const double t = hi - lo > 1 ? latency_of_top(a, (lo + hi) / 2, counts, terms, lane) : 0.0;
            if (lane == 0) node[id] = t;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            long long lo = bracket[0], hi = bracket[1];
            double t_lo = ends[0], t_hi = ends[1];
            int id2 = 1, iters = state[0];
            for (int d = 0; d < a.depth && t_hi - t_lo > a.eps && hi - lo > 1; ++d) {
                const long long mid = (lo + hi) / 2;
                const double t = node[id2];
                if (t < a.t_budget) { t_lo = t; lo = mid; id2 = 2 * id2 + 1; } else { t_hi = t; hi = mid; id2 = 2 * id2; }
                ++iters;
            }
            bracket[0] = lo; bracket[1] = hi;
            ends[0] = t_lo; ends[1] = t_hi;
            state[0] = iters;
        }
        __syncthreads();
    }
    if (warp == 0) {
        const long long n = (bracket[0] + bracket[1]) / 2;
        const double t = latency_of_top(a, n, counts, terms, lane);
        for (int l = lane; l < a.n_layers; l += 32) a.kept[l] = counts[l];
        if (lane == 0) {
            *a.n_keep = n;
            *a.result = {n, bracket[0], bracket[1], state[0], t};
        }
    }
}

// Page-locked staging of alcs_project_bisection (tables in, result out), shared by all calls: one call at a time.
std::mutex g_staging_mu;
void* g_staging = nullptr;
size_t g_staging_bytes = 0;

// Device memory of the calls: a pool of the library's own per device, which keeps up to kPoolKeep bytes between
// calls (the device's default pool gives everything back at the first synchronisation, and a call then spends
// more time in the driver than on the GPU).
constexpr unsigned long long kPoolKeep = 64ull << 20;
std::mutex g_pool_mu;
cudaMemPool_t g_pools[64] = {};

cudaError_t pool_of(int dev, cudaMemPool_t* out)
{
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lk(g_pool_mu);
    if (!g_pools[dev]) {
        cudaMemPoolProps props = {};
        props.allocType = cudaMemAllocationTypePinned;
        props.location.type = cudaMemLocationTypeDevice;
        props.location.id = dev;
        cudaMemPool_t pool = nullptr;
        cudaError_t e = cudaMemPoolCreate(&pool, &props);
        unsigned long long keep = kPoolKeep;
        if (e == cudaSuccess) e = cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep);
        if (e != cudaSuccess) return e;
        g_pools[dev] = pool;
    }
    *out = g_pools[dev];
    return cudaSuccess;
}

}  // namespace

namespace alcs {

int scratch_alloc(int device, size_t bytes, void* cuda_stream, void** out)
{
    cudaMemPool_t mem = nullptr;
    ALCS_CUDA(pool_of(device, &mem));
    if (cudaMallocFromPoolAsync(out, bytes, mem, static_cast<cudaStream_t>(cuda_stream)) != cudaSuccess) {
        (void)cudaGetLastError();
        return ALCS_ERR_ALLOC;
    }
    return ALCS_OK;
}

void scratch_free(void* p, void* cuda_stream) { cudaFreeAsync(p, static_cast<cudaStream_t>(cuda_stream)); }

}  // namespace alcs

extern "C" {

ALCS_API int alcs_layer_latency(const alcs_latency_table* tab, int64_t s, double* out)
{
    if (!out) return ALCS_ERR_INVALID_ARG;
    const int rc = check_table(tab);
    if (rc) return rc;
    *out = interpolate(*tab, s);
    return ALCS_OK;
}

ALCS_API int alcs_network_latency(double tau, const alcs_latency_table* tabs, int n_layers, const int64_t* s, double* out)
{
    if (!out || n_layers < 0 || (n_layers && (!tabs || !s))) return ALCS_ERR_INVALID_ARG;
    double total = tau;
    for (int l = 0; l < n_layers; ++l) {
        const int rc = check_table(&tabs[l]);
        if (rc) return rc;
        total += interpolate(tabs[l], s[l]);
    }
    *out = total;
    return ALCS_OK;
}

ALCS_API int alcs_project_bisection(const float* const* u_tilde, const int* cout, const int* cols, int n_layers, int g,
                                    const alcs_latency_table* tabs, double tau, double t_budget, double eps,
                                    uint8_t* mask_out, float* const* u_out, int64_t* kept_per_layer,
                                    alcs_projection_result* result, void* cuda_stream)
{
    if (!u_tilde || !cout || !cols || !tabs || !mask_out || n_layers <= 0 || g < 1 || g > 64) return ALCS_ERR_INVALID_ARG;
    if (n_layers > kMaxLayers) return ALCS_ERR_UNSUPPORTED;
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    std::vector<long long> off(n_layers + 1, 0);
    for (int l = 0; l < n_layers; ++l) {
        if (!u_tilde[l] || cout[l] <= 0 || cols[l] <= 0) return ALCS_ERR_INVALID_ARG;
        const int rc = check_table(&tabs[l]);
        if (rc) return rc;
        off[l + 1] = off[l] + (long long)((cout[l] + g - 1) / g) * cols[l];
    }
    const long long total = off[n_layers];
    if (total >= (1ll << 31)) return ALCS_ERR_SHAPE;        // the sort takes a 32-bit signed item count
    int dev = 0, sms = 0;
    ALCS_CUDA(cudaGetDevice(&dev));
    ALCS_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    auto blocks_for = [&](long long n) {
        return (unsigned)std::max<long long>(1, std::min<long long>((n + 255) / 256, (long long)sms * 16));
    };
    auto up = [](size_t b) { return (b + 255) / 256 * 256; };

    // Host tables: group offsets, knots, slopes.
    size_t knots = 0;
    for (int l = 0; l < n_layers; ++l) knots += tabs[l].n_knots;
    const size_t h_first = up((n_layers + 1) * 8), h_k = h_first + up((n_layers + 1) * 4), h_t = h_k + up(knots * 8), h_alpha = h_t + up(knots * 8);
    const size_t h_tables = h_alpha + up(knots * 8), h_result = h_tables, h_kept = h_result + up(sizeof(SearchResult));
    const size_t host_bytes = h_kept + up((size_t)n_layers * 8);
    std::unique_lock<std::mutex> staging_lock(g_staging_mu);
    if (g_staging_bytes < host_bytes) {
        if (g_staging) cudaFreeHost(g_staging);
        g_staging = nullptr;
        g_staging_bytes = 0;
        if (cudaMallocHost(&g_staging, host_bytes) != cudaSuccess) {
            (void)cudaGetLastError();
            return ALCS_ERR_ALLOC;
        }
        g_staging_bytes = host_bytes;
    }
    unsigned char* const host = static_cast<unsigned char*>(g_staging);
    std::copy(off.begin(), off.end(), reinterpret_cast<long long*>(host));
    {
        int* first = reinterpret_cast<int*>(host + h_first);
        long long* k = reinterpret_cast<long long*>(host + h_k);
        double *t = reinterpret_cast<double*>(host + h_t), *alpha = reinterpret_cast<double*>(host + h_alpha);
        int at = 0;
        for (int l = 0; l < n_layers; ++l) {
            first[l] = at;
            for (int i = 0; i < tabs[l].n_knots; ++i, ++at) {
                k[at] = tabs[l].k[i];
                t[at] = tabs[l].t[i];
                alpha[at] = i + 1 < tabs[l].n_knots ? (tabs[l].t[i + 1] - tabs[l].t[i]) / ((double)tabs[l].k[i + 1] - (double)tabs[l].k[i]) : 0.0;
            }
        }
        first[n_layers] = at;
    }

    // One stream-ordered allocation for everything.
    const long long n_buckets = std::max(1ll, (total + kRankBucket - 1) / kRankBucket);
    size_t sort_bytes = 0;
    ALCS_CUDA(cub::DeviceRadixSort::SortPairsDescending(nullptr, sort_bytes, (unsigned*)nullptr, (unsigned*)nullptr,
                                                       (unsigned*)nullptr, (unsigned*)nullptr, (int)total, 0, 32, st));
    const size_t b_keys = up((size_t)total * 4), b_lay = up((size_t)total * 2), b_hist = up((size_t)n_buckets * n_layers * 4);
    const size_t bytes = 4 * b_keys + b_lay + b_hist + h_tables + 256 + up(sort_bytes);
    unsigned char* pool = nullptr;
    if (const int rc = alcs::scratch_alloc(dev, bytes, st, reinterpret_cast<void**>(&pool))) return rc;
    // (an error on the way out: nothing may still write to the staging memory when the lock goes)
    struct Release {
        unsigned char* p; cudaStream_t s; bool waited;
        ~Release() { cudaFreeAsync(p, s); if (!waited) cudaStreamSynchronize(s); }
    } release{pool, st, false};
    unsigned* keys = (unsigned*)pool;
    unsigned* idx = (unsigned*)(pool + b_keys);
    unsigned* keys2 = (unsigned*)(pool + 2 * b_keys);
    unsigned* idx2 = (unsigned*)(pool + 3 * b_keys);
    unsigned short* layer_of = (unsigned short*)(pool + 4 * b_keys);
    unsigned* hist = (unsigned*)(pool + 4 * b_keys + b_lay);
    unsigned char* tables = pool + 4 * b_keys + b_lay + b_hist;
    long long* d_keep = (long long*)(tables + h_tables);
    void* sort_tmp = tables + h_tables + 256;

    // Ranking (Algorithm 1: the groups of all layers sorted together by norm, largest first).  The radix
    // sort is stable, so equal keys stay in (layer, group) order.  Then, for the ranked list, the layer
    // of every entry and, per bucket of kRankBucket consecutive ranks, how many entries each layer has
    // before it: the latency of "the N best-ranked groups kept" depends on N through those counts only.
    ALCS_CUDA(cudaMemcpyAsync(tables, host, h_tables, cudaMemcpyHostToDevice, st));
    std::vector<LayerTable> launches((n_layers + kLayersPerLaunch - 1) / kLayersPerLaunch);
    for (size_t i = 0; i < launches.size(); ++i) {
        LayerTable& t = launches[i];
        const int l0 = (int)i * kLayersPerLaunch;
        t.n_layers = std::min(kLayersPerLaunch, n_layers - l0);
        t.g = g;
        for (int l = 0; l < t.n_layers; ++l) {
            t.u[l] = u_tilde[l0 + l];
            t.out[l] = u_out ? u_out[l0 + l] : nullptr;
            t.cout[l] = cout[l0 + l];
            t.cols[l] = cols[l0 + l];
            t.off[l] = off[l0 + l];
        }
        t.off[t.n_layers] = off[l0 + t.n_layers];
        t.total = t.off[t.n_layers] - t.off[0];
        group_keys_kernel<<<blocks_for(t.total), 256, 0, st>>>(t, keys, idx);
    }
    ALCS_CUDA(cudaGetLastError());
    ALCS_CUDA(cub::DeviceRadixSort::SortPairsDescending(sort_tmp, sort_bytes, keys, keys2, idx, idx2, (int)total, 0, 32, st));
    ranked_layers_kernel<<<(unsigned)n_buckets, 256, n_layers * 4, st>>>(idx2, total, (const long long*)tables, n_layers, layer_of, hist);
    prefix_kernel<<<(unsigned)n_layers, 1024, 0, st>>>(hist, n_buckets, n_layers);
    ALCS_CUDA(cudaGetLastError());

    SearchArgs a;
    a.layer_of = layer_of; a.prefix = hist;
    a.first_knot = (const int*)(tables + h_first); a.k = (const long long*)(tables + h_k);
    a.t = (const double*)(tables + h_t); a.alpha = (const double*)(tables + h_alpha);
    a.total = total; a.n_layers = n_layers; a.g = g;
    a.tau = tau; a.t_budget = t_budget; a.eps = eps;
    a.n_keep = d_keep;
    a.result = reinterpret_cast<SearchResult*>(host + h_result);
    a.kept = reinterpret_cast<long long*>(host + h_kept);
    // as many warps as have room for their counts, in full levels of the tree of steps
    const size_t per_warp = 256 + (size_t)n_layers * 4;
    a.depth = 5;
    while (a.depth > 1 && ((1u << a.depth) - 1) * per_warp > 40 * 1024) --a.depth;
    const unsigned warps = std::max(2u, (1u << a.depth) - 1);
    search_kernel<<<1, warps * 32, warps * per_warp, st>>>(a);
    ALCS_CUDA(cudaGetLastError());
    for (const LayerTable& t : launches) apply_kernel<<<blocks_for(t.total), 256, 0, st>>>(t, keys, keys2, idx2, d_keep, mask_out);
    ALCS_CUDA(cudaGetLastError());
    ALCS_CUDA(cudaStreamSynchronize(st));
    release.waited = true;
    const SearchResult& r = *a.result;
    if (kept_per_layer)
        for (int l = 0; l < n_layers; ++l) kept_per_layer[l] = (int64_t)a.kept[l];
    if (result) {
        result->n_keep = r.n_keep; result->n0 = r.lo; result->n1 = r.hi; result->iters = r.iters; result->latency = r.latency;
        result->n_groups = total;
    }
    return ALCS_OK;
}

}  // extern "C"
