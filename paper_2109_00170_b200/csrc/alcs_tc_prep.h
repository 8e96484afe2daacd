// Host side of the tensor-core path (alcs_tc_prep.cu): channel tiles, expanded weights, launch arguments.
#ifndef ALCS_TC_PREP_H_
#define ALCS_TC_PREP_H_

#include <array>
#include <memory>
#include <vector>

#include "alcs_internal.h"
#include "alcs_tc.h"

namespace alcs {

// What the expanded weights depend on: channels per tile and, for patch staging (kh > 0), the kernel size, by
// which the columns are reordered.
struct TcKey {
    int n, kh, kw;
    int splits = 1;      // patch staging: parts the channel blocks are split into, a tile of its own each
    std::array<int, 4> id() const { return {n, kh, kw, splits}; }
};

struct TcPrep {
    int n = 0, n_tiles = 0;      // channels per tile; tiles, parts counted
    int splits = 1;
    std::vector<int> k16;        // steps of each tile
    int k16_max = 0, k16_min = 0;
    bool uploaded = false;
    // device; one allocation, `b` first
    unsigned char* b = nullptr;
    TcTile* tiles = nullptr;
    int* cols = nullptr;         // null: every tile takes all columns
    int* chan = nullptr;         // null: identity
    TcSparse* sparse = nullptr;
};

// The problem a launch solves (one layer), everything but the weights.
struct TcProblem {
    const void* x; void* y; const float* bias; const void* res;
    int n, oh, ow, h_in, w_in, stride, pad, kh, kw;      // kh = 0: no patch staging
    unsigned flags;
    int pixels = 0;      // pixels per tile on alcs_tc16.cu; 0: on alcs_tc.cu
};

using TcForm = std::shared_ptr<TcPrep>;
int tc_prepare(const alcs_packed* w, const TcKey& key, cudaStream_t st, TcForm* out);
TcForm tc_find(const alcs_packed* w, const TcKey& key);        // already prepared, or null; caller holds w->mu
const TcPrep* tc_any_pointwise(const alcs_packed* w);          // a prepared form for pointwise layers, or null; caller holds w->mu
// Release the pointwise forms that are not among `before` (keys), in no cached plan and in no stack.
using TcForms = std::vector<std::array<int, 4>>;
TcForms tc_forms(const alcs_packed* w);
// What a call that asks for no kernel may spend on expanded weights (6 bytes per dense weight in fp32, 2 in 16 bits): matrices of
// at most kTcMaxWeights, and kTcMaxForms forms per kernel size, beyond which a further batch size takes one that is there.
constexpr long long kTcMaxWeights = 1ll << 26;
constexpr int kTcMaxForms = 4;
bool tc_form_free(const alcs_packed* w, const TcForms& forms, const TcKey& key);       // may `key` be chosen?
void tc_release(const alcs_packed* w, const TcForms& before);
int tc_fill(const alcs_packed* w, const TcPrep& t, const TcProblem& p, TcLayer* out);
// Estimates, in microseconds, from the shape and the weights alone.
double tc_tile_us(const alcs_packed* w, const TcProblem& p, int n, int k16, bool list, bool sorted);
std::vector<double> tc_tiles_us(const alcs_packed* w, const TcProblem& p, int n);        // of every channel tile, as tc_prepare would make them
double tc_merged_item_us(int dt, int n, int k16);
bool tc16_direct(const alcs_packed* w, const TcProblem& p);       // alcs_tc16.cu copies the rows of X to where they are multiplied
// alcs_tc16.cu (16-bit operands, stride 1): of an item; of a layer on its own with the pixels per tile that take the least, or (cap) with the
// most that are no more than `cap`; those.
double tc16_item_us(const alcs_packed* w, const TcProblem& p, int n, int k16, int pixels);
double tc16_layer_us(const alcs_packed* w, const TcProblem& p, int n, int sms, int cap, int* pixels);
int tc16_capped(const alcs_packed* w, const TcProblem& p, int k16_max, int cap);
std::vector<int> tc_tile_steps(const alcs_packed* w, const TcProblem& p, int n);        // of every channel tile, as tc_prepare would make them
double tc_layer_us(const alcs_packed* w, const TcProblem& p, int n, int sms);
int tc_finish(const alcs_packed* w, TcArgs<kTcMaxLayers>& a, bool patch);
int tc_launch(const alcs_packed* w, const TcArgs<kTcMaxLayers>& a, bool patch, cudaStream_t st);
int tc_run(const alcs_packed* w, const TcPrep& t, const TcProblem& p, cudaStream_t st);      // one layer, prepared
// Channels per tile and parts of the columns for a k x k layer (n = 0: not for this kernel), and the time they take.
double tc_conv2d_choose(const alcs_packed* w, const TcProblem& p, int sms, int* n, int* splits);
int tc_conv2d(const alcs_packed* w, const TcProblem& p, int n, int splits, cudaStream_t st);
bool tc_whole_images(const alcs_packed* w, const TcProblem& p);     // are X's chunks staged as runs of whole images?
bool tc_patch_fits(const alcs_packed* w, const TcProblem& p, int n);     // can the problem be run by patch staging, n channels per tile?
bool tc_fits(const alcs_packed* w, int taps, long long n, long long hw_in, long long hw);       // taps: of the kernel, 1 for pointwise layers

}  // namespace alcs

#endif  // ALCS_TC_PREP_H_
