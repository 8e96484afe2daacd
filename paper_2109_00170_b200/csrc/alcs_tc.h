// The tensor-core path of the convolutions (fifth-generation tensor cores, tcgen05): launch arguments
// shared by the kernel (alcs_tc.cu) and the host code that prepares it.
#ifndef ALCS_TC_H_
#define ALCS_TC_H_

#include <cuda_runtime.h>

#include <cstdint>

namespace alcs {

constexpr int kTcM = 128;            // pixels per tile = rows of one MMA (TMEM lanes)
constexpr int kTcMaxN = 128;         // output channels per tile
constexpr int kTcKC32 = 64, kTcKC16 = 128;      // input columns per pipeline step (chunk): fp32, 16 bits
constexpr int tc_kc(int dt) { return dt == 0 ? kTcKC32 : kTcKC16; }
constexpr int kTcHeaderBytes = 3072;     // shared memory in front of the weight stages
constexpr int kTcMaxLayers = 16;     // layers one launch can take

// One channel tile of a layer: the `n` output channels one work item computes.
struct TcTile {
    unsigned b16;      // start of its weight tiles, in 16-byte units from TcLayer::b
    int k16;           // 16-column steps (0: the tile keeps nothing, output = bias)
    int kstart;        // start of its column list; patch staging: its first block of 16 channels
};

// Division of 0 <= n < 2^31 by a fixed d >= 1 as a multiplication: with 2^(s-1) < d <= 2^s and
// mul = floor(2^(31+s) / d) + 1 the error of n * mul / 2^(31+s) is below n / 2^(31+s) < 1 / d.
struct TcDiv {
    unsigned mul, shift;
    int d;
};
inline TcDiv tc_div(int d)
{
    unsigned s = 0;
    while ((1ull << s) < (unsigned long long)d) ++s;
    return {(unsigned)((1ull << (31 + s)) / (unsigned)d + 1), 31 + s, d};
}

// The layer's packed weights as they are stored, for the outputs that the tensor cores cannot give (see recompute).
struct TcSparse {
    const int* row_ptr;
    const int* col_idx;
    const void* vals;
    int g, cout, splits;
};

struct TcLayer {
    const void* x;
    void* y;
    const float* bias;
    const void* res;
    const unsigned char* b;      // weight tiles, in the layout the MMA reads from shared memory
    const TcTile* tiles;         // null: every tile takes k16 steps, the tiles' weights one after the other
    int k16;
    const int* cols;             // input channel per entry of the tile's column list (null: all channels in order)
    const int* chan;             // output channel of row i of the tiles (null: i itself; -1: padding)
    const TcSparse* sparse;      // device memory
    int* err;
    int first_item;              // items of this layer start here
    TcDiv n_tiles, px_tiles;     // channel tiles, pixel tiles
    int tile_major;              // item order: 0 = channel tiles of one pixel tile together, 1 = pixel tiles together
    int n;                       // output channels per tile (a multiple of 16)
    int q;                       // output pixels, all images
    TcDiv hw;                    // output pixels per image
    int cin, cout;
    int hw_in, w_in, h_in;       // input image
    TcDiv ow;
    int stride, pad;
    // Patch staging (k x k kernels, strides): columns run [block of 16 channels][tap = r * kw + s][channel]; a ring slot
    // holds `blocks` blocks of the input rows a tile needs, `pitch` elements per channel
    int kh, kw;
    TcDiv taps, kwd;
    TcDiv w_vec;                 // copies per image row
    int oh, row_step;            // input rows are taken every row_step
    int blocks, pitch;
    int vec_bytes;               // bytes of one copy of X: 16, 8, 4; 0: element by element; kTcRaw: see alcs_tc16.cu
    // alcs_tc16.cu: pixels of the MMA (ppt rounded up to a multiple of 32; 0: the other kernel); bytes of one store, and of one load of the
    // residual; kTcRaw: bytes of a chunk's rows, between the runs of a row, between rows
    int n_px, y_vec, res_vec, raw_bytes, raw_pitch, raw_row;
    int ppt;                     // pixels per tile: kTcM (alcs_tc16.cu: up to kTc16Pixels), or those of ...
    int images;                  // ... this many whole images, staged as runs of memory (0: not so)
    int n_img;
    int relu, y32;               // y32: fp32 output of 16-bit operands
};

template <int L>
struct TcArgs {
    int n_layers, n_items;
    const int* sched;            // null: thread block b takes items b, b + grid, ...; else its items are sched[b], sched[b + grid], ... until -1
    int stages;                  // weight stages in shared memory
    int stage_bytes;
    int slots, slot_bytes;       // patch staging: X ring; alcs_tc16.cu: slot_bytes of weights in front of a stage's X
    int raw_slots, raw_bytes;    // alcs_tc16.cu: rows fetched as they are
    TcLayer layer[L];
};

// alcs_tc16.cu: a stage holds kTc16Chunk columns of the weights and of X; kTc16Fixed bytes of shared memory
// in front of the stages.
constexpr int kTc16Chunk = 64, kTc16Header = 1024, kTc16Staging = 32 * 128, kTc16Fixed = kTc16Header + 16 * kTc16Staging;
constexpr int kTc16Pixels = 256;     // at most, per tile; half of it where a tile's columns take several accumulators
constexpr int kTc16Group = 16;       // 16-column steps per accumulator
constexpr int kTcRaw = 1;            // X is fetched by 16-byte words and picked apart in shared memory
constexpr int kTc16RawMost = 48 * 1024;        // bytes of a chunk's rows
constexpr int kTc16Raw = kTc16Pixels / 2;      // most pixels per tile then
constexpr int tc16_weight_bytes(int n) { return kTc16Chunk * n * 2; }
constexpr int tc16_stage_bytes(int n, int px) { return tc16_weight_bytes(n) + (px + 63) / 64 * (64 * kTc16Chunk * 2); }
cudaError_t launch_tc16(int dt, const TcArgs<kTcMaxLayers>& a, int blocks, cudaStream_t st);
cudaError_t prepare_tc16(int dt);

// Sum of the partial results of a layer whose columns were split: part[image][tile][split][n][hw] over the splits in
// order, bias, ReLU.
struct TcReduce {
    const float* part;
    float* y;
    const float* bias;
    int n, splits, tiles, cout, relu;
    TcDiv hw, width;             // width: channels per tile
    long long total;             // outputs
};
cudaError_t launch_tc_reduce(const TcReduce& a, int sms, cudaStream_t st);

// Launch a (n_layers <= kTcMaxLayers; one launch with elements of type dt) on `blocks` thread
// blocks; patch: all layers by patch staging.
cudaError_t launch_tc(int dt, bool patch, const TcArgs<kTcMaxLayers>& a, int blocks, cudaStream_t st);
cudaError_t prepare_tc(int dt);      // once per device: shared-memory attribute
constexpr int tc_planes(int dt) { return dt == 0 ? 3 : 1; }      // 16-bit planes an operand is split into
// ring of X chunks: 4 of 128 pixels x 64 columns in fp32, x 128 columns in 16 bits
constexpr int kTcRingBytes = 4 * kTcM * 64 * 4;
constexpr int tc_stage_bytes(int dt, int n) { return tc_planes(dt) * tc_kc(dt) * n * 2; }

}  // namespace alcs

#endif  // ALCS_TC_H_
