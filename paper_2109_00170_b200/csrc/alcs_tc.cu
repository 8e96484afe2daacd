// Convolution on the fifth-generation tensor cores (tcgen05), sm_100a: fp32 operands, k x k kernels, strides, and those 16-bit
// layers at stride 1 that alcs_tc16.cu is not expected to be faster at (small images staged whole, most rows of odd length, layers
// of few pixels: half of the layers of random shape).
//
// A work item is (128 output pixels) x (n output channels).  The item's pruned weights are expanded
// to a dense [columns][n] tile (columns that no row of the tile keeps are left out), so that the item
// is a plain contraction
//     D[128 pixels][n] += A[128 pixels][64 columns] * B[64 columns][n]
// per chunk of 64 columns, with D and A in tensor memory and B in shared memory.
//
// fp32 operands are split exactly into three bfloat16 parts (8 + 8 + 8 significant bits) and six of
// the nine partial products are formed, which leaves out terms below 2^-24 of a product; they are
// summed smallest first into a fresh accumulator per chunk, and the chunk sums are added in fp32
// (round to nearest) in registers.  The tensor core truncates when it adds to its fp32 accumulator;
// with four full-size additions per chunk the result is closer to the exact sum than a chain of fp32
// FMAs (relative error 7e-8 against 2.3e-7 at 512 columns, 30 % of them kept).
// 16-bit operands are used as they are, 256 columns per accumulator.
//
// Roles (32 warps, one thread block per SM, persistent over items):
//   warps 27-30  producers: copy chunks of X ([64 columns][128 pixels]) into a ring in shared memory, several
//                chunks ahead; 16-byte copies where images allow it, single elements otherwise (any image
//                size, stride, channel list or tap offset costs only address arithmetic)
//   warps 0-15   converters: a lane is a pixel, a warp takes 16 of a chunk's columns; split the values and write them to tensor memory as
//                the A operand (double-buffered)
//   warps 24-25  issue the MMAs: in fp32 the chunks, which have an accumulator each, in turn, so that one waits for
//                its next chunk while the other's instructions run; in 16 bits the first alone
//   warp 26      copies the weight tiles (bulk copies into a ring)
//   warps 16-23  epilogue: add the chunk sums up, then bias, residual, ReLU and stores, while the next
//                item is already being multiplied (two accumulators)
#include "alcs_tc.cuh"

namespace alcs {
namespace {

constexpr int kConvWarps = 16, kEpiWarps = 8, kProdWarps = 4;
constexpr int kMmaWarp = kConvWarps + kEpiWarps, kLoadWarp = kMmaWarp + 2, kProdWarp0 = kMmaWarp + 3;
constexpr int kThreads = 1024;      // eight warpgroups (one warp idle)
// Registers per thread: 1024 threads start with 64; the epilogue, which holds 64 sums, takes from the
// others: 4 * 40 + 2 * 128 + 2 * 48 <= 8 * 64.
constexpr int kConvRegs = 40, kEpiRegs = 128, kProdRegs = 48;
// Shared memory: barriers and the TMEM address; the bias of the items being stored (two copies of 128 words per
// half of the epilogue); weight stages; X ring.
constexpr int kBarBytes = kTcHeaderBytes, kEpiOff = 1024, kEpiBytes = 512;
static_assert(kEpiOff + 4 * kEpiBytes <= kBarBytes, "header");
constexpr int kMaxStages = 8;
constexpr int kMaxTcSmem = 227 * 1024;
// Subtract from each of two fp32 values what its upper 16 bits stand for (exact).
__device__ __forceinline__ void cut2(unsigned& u0, unsigned& u1)
{
    asm("{\n\t.reg .b32 h0, h1;\n\t.reg .b64 x, h;\n\tand.b32 h0, %0, 0xffff0000;\n\tand.b32 h1, %1, 0xffff0000;\n\t"
        "mov.b64 x, {%0, %1};\n\tmov.b64 h, {h0, h1};\n\tsub.rn.f32x2 x, x, h;\n\tmov.b64 {%0, %1}, x;\n\t}"
        : "+r"(u0), "+r"(u1));
}

// Three bfloat16 parts of two fp32 values, packed two to a word: x = part 0 + part 1 + part 2 exactly.
// Cutting off the low bits (instead of rounding) needs no conversion instructions and cannot overflow;
// the weights' parts are rounded, so the partial products that are left out have no common sign.
__device__ __forceinline__ void split2(float x0, float x1, unsigned& p0, unsigned& p1, unsigned& p2)
{
    unsigned u0 = __float_as_uint(x0), u1 = __float_as_uint(x1);
    p0 = __byte_perm(u0, u1, 0x7632);
    cut2(u0, u1);
    p1 = __byte_perm(u0, u1, 0x7632);
    cut2(u0, u1);
    p2 = __byte_perm(u0, u1, 0x7632);
}

// Where a producer warp finds the pixels of one item.
template <typename XT>
struct Source {
    using raw = typename Elem<XT>::raw;
    static constexpr int kRow = kTcM * (int)sizeof(raw);      // bytes of a column of a chunk in shared memory
    const raw* x;
    const int* cols;
    int off[4];                    // element offset of this lane's first column entry: [0] alone for vector copies
    int hw_in, cin, vb;
    int img0, n_img = 0, hw;       // whole images (TcLayer::images): first, how many, pixels

    __device__ __forceinline__ int pixel(const TcLayer& y, int q) const
    {
        const int img = div_of(q, y.hw);
        return img * cin * hw_in + (q - img * y.hw.d);
    }

    __device__ __forceinline__ void open(const TcLayer& y, const TcTile& t, int pt, int lane)
    {
        x = static_cast<const raw*>(y.x);
        hw_in = y.hw_in;
        cin = y.cin;
        vb = y.vec_bytes;
        cols = y.cols ? y.cols + t.kstart : nullptr;
        // (pixels past the end repeat the last ones and are not stored)
        if (y.images) {
            img0 = pt * y.images;
            n_img = min(y.images, y.n_img - img0);
            hw = y.hw.d;
        } else if (vb) {
            const int ppl = vb / (int)sizeof(raw);      // pixels per copy; a column's 128 pixels take 128 / ppl copies
            off[0] = pixel(y, min(pt * y.ppt + (lane * ppl & (kTcM - 1)), y.q - ppl));
            if (vb == 4) off[1] = pixel(y, min(pt * y.ppt + 64 + (lane * ppl & 63), y.q - ppl));
        } else {
#pragma unroll
            for (int j = 0; j < 4; ++j) off[j] = pixel(y, min(pt * y.ppt + j * 32 + lane, y.q - 1));
        }
    }

    // Element offsets of columns k .. k + 3 (past the last channel they meet zero weights: any valid one will do).
    __device__ __forceinline__ int4 cols4(int k) const
    {
        int4 c;
        if (cols) {
            c = __ldg(reinterpret_cast<const int4*>(cols + k));
        } else {
            c = make_int4(k, k + 1, k + 2, k + 3);
            if (k + 4 > cin) c = make_int4(min(c.x, cin - 1), min(c.y, cin - 1), min(c.z, cin - 1), min(c.w, cin - 1));
        }
        return make_int4(c.x * hw_in, c.y * hw_in, c.z * hw_in, c.w * hw_in);
    }

    // Copy the chunk that starts at column k0 (kk columns, a multiple of 16) into `slot`; one arrival per lane on `bar`.
    __device__ __forceinline__ void chunk(unsigned slot, int k0, int kk, int lane, unsigned bar) const
    {
        if (n_img) {
            // whole small images: the chunk's columns of an image are one run of memory
            if (lane == 0) {
                const unsigned bytes = (unsigned)(kk * hw) * (unsigned)sizeof(raw);
                asm volatile("mbarrier.expect_tx.relaxed.cta.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(bytes * n_img) : "memory");
#pragma unroll 1
                for (int i = 0; i < n_img; ++i)
                    bulk_load(slot + i * bytes, x + ((size_t)(img0 + i) * cin + k0) * hw, bytes, bar);
            }
            __syncwarp();
            bar_arrive(bar);
            return;
        }
        slot += lane * (vb == 0 ? (int)sizeof(raw) : vb);
#pragma unroll 1
        for (int k = 0; k < kk; k += 4, slot += 4 * kRow) {
                const int4 c = cols4(k0 + k);
                const int at[4] = {c.x, c.y, c.z, c.w};
                if (vb == 16) {
                    if constexpr (sizeof(raw) == 4) {
#pragma unroll
                        for (int i = 0; i < 4; ++i) cp_async16(slot + i * kRow, x + (at[i] + off[0]));
                    } else {        // two columns per instruction
#pragma unroll
                        for (int i = 0; i < 4; i += 2) cp_async16(slot + i * kRow, x + ((lane < 16 ? at[i] : at[i + 1]) + off[0]));
                    }
                } else if constexpr (sizeof(raw) == 4) {
#pragma unroll
                    for (int i = 0; i < 4; ++i)
#pragma unroll
                        for (int j = 0; j < 4; ++j) cp_async_small<4>(slot + i * kRow + j * 128, x + (at[i] + off[j]), 4);
                } else if (vb == 8) {
#pragma unroll
                    for (int i = 0; i < 4; ++i) cp_async_small<8>(slot + i * kRow, x + (at[i] + off[0]), 8);
                } else if (vb == 4) {
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        cp_async_small<4>(slot + i * kRow, x + (at[i] + off[0]), 4);
                        cp_async_small<4>(slot + i * kRow + 128, x + (at[i] + off[1]), 4);
                    }
                } else {            // rows that start on odd element boundaries: through registers
                    raw v[4][4];
#pragma unroll
                    for (int i = 0; i < 4; ++i)
#pragma unroll
                        for (int j = 0; j < 4; ++j) v[i][j] = ld_x(x + (at[i] + off[j]));
#pragma unroll
                    for (int i = 0; i < 4; ++i)
#pragma unroll
                        for (int j = 0; j < 4; ++j) st_slot(slot + i * kRow + j * 64, v[i][j]);
                }
        }
        if (sizeof(raw) == 2 && vb == 0) bar_arrive(bar);
        else cp_async_arrive(bar);
    }
};

// The input rows a tile of consecutive output pixels needs, by patch staging: the tile touches images img0 .. ; of
// each, rows first .. of every channel lie one after the other in the slot.
struct Patch {
    int img0, n_img;
    int y0, first0, rows0;         // of the first image (y0: its first output row here)
    int rows, rows_last;           // of a whole image, and of the last one (if it is not the first)

    __device__ __forceinline__ Patch(const TcLayer& y, int pt)
    {
        const int q0 = pt * y.ppt, q1 = min(q0 + kTcM, y.q) - 1;
        img0 = div_of(q0, y.hw);
        n_img = div_of(q1, y.hw) - img0 + 1;
        y0 = div_of(q0 - img0 * y.hw.d, y.ow);
        const int y1 = div_of(q1 - (img0 + n_img - 1) * y.hw.d, y.ow);
        first0 = max(0, y0 * y.stride - y.pad);
        rows0 = count(y, first0, n_img > 1 ? y.oh - 1 : y1);
        rows = count(y, 0, y.oh - 1);
        rows_last = count(y, 0, y1);
    }
    // input rows from `first` to the last one that output row `last` needs
    static __device__ __forceinline__ int count(const TcLayer& y, int first, int last)
    {
        const int n = min(y.h_in - 1, last * y.stride - y.pad + y.kh - 1) - first;
        return max(0, y.row_step == 1 ? n + 1 : last - first / y.stride + 1);
    }
};

// Copy one slot of patches: channels c0 .. c0 + nc, all images of the tile.
template <typename XT>
__device__ __forceinline__ void copy_patch(const TcLayer& y, const Patch& t, unsigned slot, int c0, int nc, int lane, unsigned bar)
{
    using raw = typename Elem<XT>::raw;
    const int vb = y.vec_bytes, epv = vb / (int)sizeof(raw);
    const raw* const x = static_cast<const raw*>(y.x);
    const unsigned pitch = y.pitch * (unsigned)sizeof(raw);
#pragma unroll 1
    for (int i = 0; i < t.n_img; ++i) {
        const int rows = i == 0 ? t.rows0 : i + 1 == t.n_img ? t.rows_last : t.rows;
        const raw* const src = x + (((t.img0 + i) * y.cin + c0) * y.hw_in + (i == 0 ? t.first0 : 0) * y.w_in);
        const int pieces = rows * y.w_vec.d;
#pragma unroll 1
        for (int p = lane; p < pieces; p += 32) {
            int at = p * epv;
            if (y.row_step != 1) {
                const int r = div_of(p, y.w_vec);
                at += r * (y.row_step - 1) * y.w_in;
            }
            const raw* from = src + at;
            unsigned to = slot + p * vb;
            if constexpr (sizeof(raw) == 2)
                if (vb == 2) {      // (an X that starts on an odd element)
#pragma unroll 1
                    for (int c = 0; c < nc; ++c) st_slot(to + c * pitch, ld_x(from + (size_t)c * y.hw_in));
                    continue;
                }
#pragma unroll 4
            for (int c = 0; c < nc; ++c) {
                if (vb == 16) cp_async16(to, from);
                else if (vb == 8) cp_async_small<8>(to, from, 8);
                else cp_async_small<4>(to, from, 4);
                to += pitch;
                from += y.hw_in;
            }
        }
        slot += rows * y.w_in * (unsigned)sizeof(raw);
    }
    if (sizeof(raw) == 2 && vb == 2) bar_arrive(bar);
    else cp_async_arrive(bar);
}

__device__ __forceinline__ void ld_slot(unsigned addr, float& v) { asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(addr)); }
__device__ __forceinline__ void ld_slot(unsigned addr, unsigned short& v) { asm volatile("ld.shared.u16 %0, [%1];" : "=h"(v) : "r"(addr)); }

// The end of an item, 32 rows at a time: bias, residual, ReLU, one rounding, stores.  A warp stores 32 consecutive
// pixels of one channel per instruction.  `lane_off` is the byte offset of this lane's pixel from `out` (and from
// `res`, if there is one), which are the same for the whole warp, so that an address is one 32-bit addition.
// floor: 0 with ReLU, else NaN (fmaxf then returns the other operand); pitch: bytes from one channel to the next.
// any = false: rows row0 .. row0 + rows are channels row0 .. , and out points at row0; otherwise every row's channel
// is looked up and out points at channel 0.
template <typename YT>
__device__ __forceinline__ void store32(float (&v)[32], const TcLayer& y, char* out, const char* res, unsigned lane_off, unsigned pitch, float floor,
                                        unsigned bias, int row0, int rows, bool live, bool any)
{
#pragma unroll
    for (int j = 0; j < 32; j += 4) {
        float b[4];
        asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(b[0]), "=f"(b[1]), "=f"(b[2]), "=f"(b[3]) : "r"(bias + j * 4));
#pragma unroll
        for (int k = 0; k < 4; ++k) v[j + k] += b[k];
    }
    if (!any) {
        if (!live) return;
        if (res) {      // all loads, then all additions: one round trip to L2 per 32 rows
            YT r[32];
#pragma unroll
            for (int j = 0; j < 32; ++j) r[j] = __ldg(reinterpret_cast<const YT*>(res + (lane_off + (j < rows ? j : 0) * pitch)));
#pragma unroll
            for (int j = 0; j < 32; ++j) v[j] += (float)r[j];
        }
#pragma unroll
        for (int j = 0; j < 32; j += 8) {
            if (j >= rows) break;
            if (j + 8 <= rows) {
#pragma unroll
                for (int k = 0; k < 8; ++k) put(reinterpret_cast<YT*>(out + (lane_off + (j + k) * pitch)), fmaxf(v[j + k], floor));
            } else {
#pragma unroll
                for (int k = 0; k < 7; ++k)
                    if (j + k < rows) put(reinterpret_cast<YT*>(out + (lane_off + (j + k) * pitch)), fmaxf(v[j + k], floor));
            }
        }
        return;
    }
#pragma unroll
    for (int j = 0; j < 32; j += 8) {
        if (j >= rows) break;
        int c[8];
        float r[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) c[k] = channel_of(y, row0 + j + k);
#pragma unroll
        for (int k = 0; k < 8; ++k) r[k] = res && live && c[k] >= 0 ? (float)__ldg(reinterpret_cast<const YT*>(res + (lane_off + c[k] * pitch))) : 0.0f;
#pragma unroll
        for (int k = 0; k < 8; ++k)
            if (live && c[k] >= 0) put(reinterpret_cast<YT*>(out + (lane_off + c[k] * pitch)), fmaxf(v[j + k] + r[k], floor));
    }
}

// An item whose tile keeps no block: bias and residual alone, four channels at a time (one at a time, each waited for its
// loads: 230 us for 60 -> 644 channels, 56 x 56, batch 22, fp16, 1 % kept, most of whose tiles are empty).
template <typename YT>
__device__ __forceinline__ void store_bias(const TcLayer& y, char* out, const char* res, unsigned lane_off, int row0, int rows, bool live)
{
    const unsigned pitch = (unsigned)y.hw.d * (unsigned)sizeof(YT);
#pragma unroll 1
    for (int j = 0; j < rows; j += 4) {
        int c[4];
        float v[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) c[k] = live && j + k < rows ? channel_of(y, row0 + j + k) : -1;
#pragma unroll
        for (int k = 0; k < 4; ++k) v[k] = y.bias && c[k] >= 0 ? __ldg(y.bias + c[k]) : 0.0f;
        if (res) {
            YT r[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) r[k] = __ldg(reinterpret_cast<const YT*>(res + (live ? lane_off + max(c[k], 0) * pitch : 0)));
#pragma unroll
            for (int k = 0; k < 4; ++k) v[k] += (float)r[k];
        }
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (c[k] >= 0) put(reinterpret_cast<YT*>(out + (lane_off + c[k] * pitch)), y.relu ? fmaxf(v[k], 0.0f) : v[k]);
    }
}

// GENERAL: layers with a residual, sorted rows or fp32 output of 16-bit operands among them.  What they add to the
// epilogue is a third of the kernel's code, and the roles' loops compete for the instruction caches as it is.
template <typename XT, bool PATCH, bool GENERAL, int L>
__global__ void __launch_bounds__(kThreads, 1) tc_kernel(const __grid_constant__ TcArgs<L> a)
{
    using E = Elem<XT>;
    using raw = typename E::raw;
    constexpr int P = E::planes;
    constexpr bool kEarly = P == 3 && (PATCH || L == 1);       // converters read a chunk's values before its buffer is free
    extern __shared__ __align__(1024) unsigned char smem[];
    const unsigned s0 = smem_u32(smem);
    const unsigned a_full = s0, a_empty = s0 + 32, d_full = s0 + 64, d_empty = s0 + 80, x_full = s0 + 128, x_empty = s0 + 192;
    const unsigned b_full = s0 + 256, b_empty = s0 + 320, turn = s0 + 384, tmem_slot = s0 + 400, drained = s0 + 408;
    const unsigned not_finite = s0 + 424;      // layers whose items had sums that are not finite, a bit each
    const unsigned stage0 = s0 + kBarBytes, ring0 = stage0 + a.stages * a.stage_bytes;
    constexpr int NA = E::abufs, KC = P == 3 ? kTcKC32 : kTcKC16, NS = KC / 16, AB = KC / 2 * P;      // AB: TMEM columns of a chunk of A
    // every producer owns a slot
    const unsigned S = PATCH ? (unsigned)a.slots : (unsigned)kProdWarps, kSlot = PATCH ? (unsigned)a.slot_bytes : KC * kTcM * (unsigned)sizeof(raw);
    static_assert(kProdWarps * KC * kTcM * (int)sizeof(raw) == kTcRingBytes && NA * AB <= 256, "ring and A buffers");
    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;

    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (warp == kMmaWarp) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(tmem_slot) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    } else if (warp == kLoadWarp && lane == 0) {
#pragma unroll 1
        for (int i = 0; i < NA; ++i) {
            bar_init(a_full + 8 * i, kConvWarps);
            bar_init(a_empty + 8 * i, 1);
        }
#pragma unroll 1
        for (int i = 0; i < 2; ++i) {
            bar_init(turn + 8 * i, 1);
            bar_init(drained + 8 * i, 1);
            bar_init(d_full + 8 * i, 1);
            bar_init(d_empty + 8 * i, kEpiWarps);
        }
#pragma unroll 1
        for (int i = 0; i < kMaxStages; ++i) {
            bar_init(b_full + 8 * i, 1);
            bar_init(b_empty + 8 * i, 1);
        }
#pragma unroll 1
        for (int i = 0; i < kProdWarps; ++i) {
            bar_init(x_full + 8 * i, 32);
            bar_init(x_empty + 8 * i, kConvWarps);
        }
        asm volatile("st.shared.u32 [%0], 0;" ::"r"(not_finite) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    tc_before();
    __syncthreads();
    tc_after();
    unsigned tmem;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(tmem) : "r"(tmem_slot));
    // tensor memory: D in columns [0, 256), two accumulators of up to 128; A behind, NA buffers
    const unsigned tmem_a = tmem + 256;
    bool ok = true;

    if (warp < kConvWarps) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kConvRegs));
        const unsigned quad = (unsigned)(warp & 3);
        const int s0_ = warp >> 2, row = quad * 32 + lane;       // a warp takes every fourth 16-column step
        unsigned i = 0, slot = 0, xph = 0, buf = 0, aph = 1;
        bool opened = false;            // PATCH: whether the slot in use has been waited for
        Cursor<L> cur(a);
#pragma unroll 1
        while (ok && cur.step()) {
            const TcLayer& y = cur.of();
            const int images = PATCH ? 0 : y.images;
            int hw = kTcM, img = 0, px = row;
            // PATCH: this pixel's window in the patch, which taps of it lie inside the image, and the walk over the steps
            int block = 0, tap = s0_, in_slot = 0;
            unsigned mask = 0;
            if constexpr (PATCH) {
                const Patch t(y, cur.pt());
                const int q = min(cur.pt() * y.ppt + row, y.q - 1);
                img = div_of(q, y.hw);
                const int p = q - img * y.hw.d, oy = div_of(p, y.ow), ox = p - oy * y.ow.d;
                const int ih = oy * y.stride - y.pad, iw = ox * y.stride - y.pad, seg = img - t.img0;
                unsigned bits = 0;
#pragma unroll 1
                for (int s = 0; s < y.kw; ++s) bits |= ((unsigned)(iw + s) < (unsigned)y.w_in ? 1u : 0u) << s;
#pragma unroll 1
                for (int r = 0; r < y.kh; ++r)
                    if ((unsigned)(ih + r) < (unsigned)y.h_in) mask |= bits << (r * y.kw);
                const int line = y.row_step == 1 ? ih - (seg ? 0 : t.first0) : oy - (seg ? 0 : t.y0);
                px = ((seg ? t.rows0 + (seg - 1) * t.rows : 0) + line) * y.w_in + iw;
            } else if (images) {
                hw = y.hw.d;
                img = min(div_of(row, y.hw), images - 1);
                px = min(row - img * hw, hw - 1);
            }
#pragma unroll 1
            for (int k16 = cur.t.k16; k16 > 0; k16 -= NS, ++i) {
                const unsigned my_a = tmem_a + (quad << 21) + buf * AB;      // lanes 32 * quad ...
                const int ns = min(NS, k16);
                if (i == 0) asm volatile("griddepcontrol.wait;" ::: "memory");
                // Read the values of step s of the chunk.
                auto load = [&](int s, raw (&v)[16]) {
                    if constexpr (PATCH) {
                        while (tap >= y.taps.d) { tap -= y.taps.d; ++block; ++in_slot; }
                        // on to the slot that holds the block; every slot is waited for and given back in turn
                        while (in_slot >= y.blocks || !opened) {
                            if (in_slot >= y.blocks) {
                                in_slot -= y.blocks;
                                if (!opened) ok = ok && bar_wait(x_full + 8 * slot, xph);
                                __syncwarp();
                                if (lane == 0) bar_arrive(x_empty + 8 * slot);
                                if (++slot == S) { slot = 0; xph ^= 1u; }
                                opened = false;
                            } else {
                                ok = ok && bar_wait(x_full + 8 * slot, xph);
                                opened = true;
                            }
                        }
                        ok = __all_sync(0xffffffffu, ok);
                        if (!ok) return;
                        const int r = div_of(tap, y.kwd), nv = y.cin - (cur.t.kstart + block) * 16;
                        const bool in = (mask >> tap) & 1u;
                        const int pitch = y.pitch * (int)sizeof(raw);
                        const unsigned at = ring0 + slot * kSlot + in_slot * 16 * pitch + (px + r * y.w_in + (tap - r * y.kw)) * (int)sizeof(raw);
#pragma unroll
                        for (int j = 0; j < 16; ++j) {
                            v[j] = raw(0);
                            if (in && j < nv) ld_slot(at + j * pitch, v[j]);
                        }
                        tap += 4;
                    } else if (images) {
                        const unsigned at = ring0 + slot * kSlot + ((img * ns + s) * 16 * hw + px) * (unsigned)sizeof(raw);
#pragma unroll
                        for (int j = 0; j < 16; ++j) ld_slot(at + j * hw * (unsigned)sizeof(raw), v[j]);
                    } else {
                        const unsigned at = ring0 + slot * kSlot + (s * 16 * kTcM + px) * (unsigned)sizeof(raw);
#pragma unroll
                        for (int j = 0; j < 16; ++j) ld_slot(at + j * kTcM * (unsigned)sizeof(raw), v[j]);
                    }
                };
                auto store = [&](int s, const raw (&v)[16]) {
#pragma unroll
                    for (int h = 0; h < 8; h += 4) {
                        unsigned w[P][4];
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            const raw x0 = v[2 * (h + j)], x1 = v[2 * (h + j) + 1];
                            if constexpr (P == 3) split2(x0, x1, w[0][j], w[1][j], w[2][j]);
                            else w[0][j] = (unsigned)x0 | ((unsigned)x1 << 16);
                        }
#pragma unroll
                        for (int p = 0; p < P; ++p) tmem_st4(my_a + p * (KC / 2) + s * 8 + h, w[p]);
                    }
                };
                auto give_back = [&] {
                    __syncwarp();
                    if (lane == 0) bar_arrive(x_empty + 8 * slot);
                    if (++slot == S) { slot = 0; xph ^= 1u; }
                };
                if constexpr (kEarly) {
                    // The values are read, and their slot is given back, while the buffer they go to is still being multiplied: what is
                    // left between the end of that and the next multiplication is the split and its stores (917 cycles a chunk
                    // instead of 1,390; 3x3 layers of ResNet-18, batch 32: 354 -> 341 us; pointwise layers gain 1 %, about the noise.
                    // In merged launches, whose items are short, it is 3 % slower.)
                    raw v[16];
                    if (!PATCH) ok = __all_sync(0xffffffffu, bar_wait(x_full + 8 * slot, xph));
                    if (ok && s0_ < ns) load(s0_, v);
                    if (!ok) break;
                    if (!PATCH) {
#pragma unroll
                        for (int j = 0; j < 16; ++j) asm volatile("" : "+f"(v[j]));      // (all read)
                        give_back();
                    }
                    ok = __all_sync(0xffffffffu, bar_wait(a_empty + 8 * buf, aph));
                    if (!ok) break;
                    tc_after();
                    if (s0_ < ns) store(s0_, v);
                } else {
                    ok = (PATCH || bar_wait(x_full + 8 * slot, xph)) && bar_wait(a_empty + 8 * buf, aph);
                    ok = __all_sync(0xffffffffu, ok);
                    if (!ok) break;
                    tc_after();
#pragma unroll 1
                    for (int s = s0_; s < ns; s += 4) {
                        raw v[16];
                        load(s, v);
                        if (!ok) break;
                        store(s, v);
                    }
                    if (!ok) break;
                    if (!PATCH) give_back();
                }
                asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
                tc_before();
                __syncwarp();
                if (lane == 0) bar_arrive(a_full + 8 * buf);
                if (++buf == NA) { buf = 0; aph ^= 1u; }
            }
            if constexpr (PATCH) {      // give back the slots that are left of the item
                if (!ok) break;
                const int n_blocks = cur.t.k16 ? div_of(cur.t.k16, y.taps) : 0;
#pragma unroll 1
                for (int b = block - in_slot; b < n_blocks; b += y.blocks) {
                    if (!opened) ok = ok && __all_sync(0xffffffffu, bar_wait(x_full + 8 * slot, xph));
                    __syncwarp();
                    if (lane == 0) bar_arrive(x_empty + 8 * slot);
                    if (++slot == S) { slot = 0; xph ^= 1u; }
                    opened = false;
                }
            }
        }
    } else if (warp < kConvWarps + kEpiWarps) {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kEpiRegs));
        const unsigned quad = (unsigned)(warp & 3);
        // An item of one chunk sum is stored by the four warps that own its accumulator, so that consecutive items
        // overlap; the sums of the others are added up by all eight warps, half of the channels each.
        const int e = (warp - kConvWarps) >> 2;
        unsigned n_grp = 0, bias = s0 + kEpiOff + e * (2 * kEpiBytes);
        int key = -1, key_layer = -1;       // whose bias is in shared memory
        asm volatile("griddepcontrol.wait;" ::: "memory");
        Cursor<L> cur(a);
#pragma unroll 1
        while (ok && cur.step()) {
            const TcLayer& y = cur.of();
            const int groups = (cur.t.k16 + NS * E::group - 1) / (NS * E::group);
            const bool whole = groups <= 1;
            if (whole && (groups ? (int)(n_grp & 1u) : 0) != e) {
                n_grp += groups;
                continue;
            }
            const int nr = whole ? y.n : y.n >> 1, part = whole ? 0 : e * nr, row0 = cur.nt() * y.n + part;
            // the bias of these rows goes through shared memory; consecutive items of one channel tile share it
            const int want = row0 * 2 + whole;
            const bool fresh = groups && (want != key || cur.layer != key_layer);
            float b[4];
            if (fresh) {
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int r = row0 + i * 32 + lane, c = !y.bias || i * 32 + lane >= nr ? -1 : y.chan ? __ldg(y.chan + r) : r;
                    b[i] = c >= 0 && c < y.cout ? __ldg(y.bias + c) : 0.0f;
                }
                key = want;
                key_layer = cur.layer;
            }
            const int row = (int)quad * 32 + lane, q0 = cur.pt() * y.ppt, q = q0 + row;
            const bool live = row < y.ppt && q < y.q;
            const int img0 = div_of(q0, y.hw), img = div_of(live ? q : q0, y.hw), p = (live ? q : q0) - img * y.hw.d;
            const bool wide = sizeof(XT) == 4 || (GENERAL && y.y32), any = GENERAL && y.chan;
            const unsigned ye = wide ? 4 : sizeof(XT), pitch = (unsigned)y.hw.d * ye;
            const float floor = y.relu ? 0.0f : __int_as_float(0x7fffffff);
            const int out_rows = any ? nr : min(nr, y.cout - row0);       // (may be negative: nothing to store)
            const unsigned lane_off = ((unsigned)(img - img0) * (unsigned)y.cout * (unsigned)y.hw.d + (unsigned)p) * ye;
            const size_t item_off = ((size_t)img0 * y.cout + (any ? 0 : row0)) * y.hw.d * ye;
            char* const out = static_cast<char*>(y.y) + item_off;
            const char* const res = GENERAL && y.res ? static_cast<const char*>(y.res) + item_off : nullptr;
            if (groups == 0) {      // nothing kept: the sum is zero, and there is no accumulator to read it from
                const char* r = GENERAL && y.res ? static_cast<const char*>(y.res) + (size_t)img0 * y.cout * y.hw.d * ye : nullptr;
                char* o = static_cast<char*>(y.y) + (size_t)img0 * y.cout * y.hw.d * ye;
                if (GENERAL && sizeof(XT) == 2 && wide) store_bias<float>(y, o, r, lane_off, row0, nr, live);
                else store_bias<XT>(y, o, r, lane_off, row0, nr, live);
                __syncwarp();
                continue;
            }
            if (res && live) {      // what the end of the item will add: on its way while the item is multiplied
#pragma unroll 1
                for (int k = 0; k < nr; ++k) {
                    const int c = any ? channel_of(y, row0 + k) : row0 + k < y.cout ? k : -1;
                    if (c >= 0) asm volatile("prefetch.global.L2 [%0];" ::"l"(res + (lane_off + (unsigned)c * (unsigned)y.hw.d * ye)));
                }
            }
            __syncwarp();
            float lo[32], hi[32];               // rows 0 .. 31 and 32 .. 63
            if (!whole) {
#pragma unroll
                for (int j = 0; j < 32; ++j) lo[j] = hi[j] = 0.0f;
            }
            const unsigned src = tmem + (quad << 21) + part;
#pragma unroll 1
            for (int g = 0; g < groups; ++g, ++n_grp) {
                const unsigned d = n_grp & 1u;
                ok = __all_sync(0xffffffffu, bar_wait(d_full + 8 * d, (n_grp >> 1) & 1u));
                if (!ok) break;
                tc_after();
                if (whole) break;               // (stored from where it is)
                const unsigned from = src + d * 128;
#pragma unroll
                for (int j = 0; j < 64; j += 16) {
                    if (j >= nr) break;
                    float t[16];
                    tmem_ld16(from + j, t);         // (rows past nr: other columns of the accumulators, never stored)
                    tmem_wait_ld(t);
#pragma unroll
                    for (int k = 0; k < 16; ++k) (j < 32 ? lo : hi)[(j & 31) + k] += t[k];
                }
                tc_before();
                __syncwarp();
                if (lane == 0) bar_arrive(d_empty + 8 * d);
            }
            if (!ok) break;
            if (fresh) {
                // The four warps of a half write the same values.  Whoever has seen the item's last accumulator full knows
                // that all have stored the item that they stored before the last one, whose copy this is: an accumulator
                // is full only after the one two before it has been drained, and nobody drains for an item before the
                // item before it is stored.
                bias ^= kEpiBytes;
#pragma unroll
                for (int i = 0; i < 4; ++i) asm volatile("st.shared.f32 [%0], %1;" ::"r"(bias + (i * 32 + lane) * 4), "f"(b[i]) : "memory");
                __syncwarp();
            }
            const unsigned d = n_grp & 1u;
            if (whole) tmem_ld32(src + d * 128, lo);
#pragma unroll 1
            for (int h = 0; h < out_rows; h += 32) {
                if (whole) tmem_wait_ld(lo);
                // (an input that is not finite reaches every channel of the tile, so one of them tells; rows that are no
                // output may hold whatever lay in shared memory)
                if (h == 0 && live && special<float>(lo[0])) asm volatile("red.shared.or.b32 [%0], %1;" ::"r"(not_finite), "r"(1u << (L > 1 ? cur.layer : 0)) : "memory");
                const unsigned off = lane_off + (any ? 0 : (unsigned)h * pitch);
                const int rows = min(32, out_rows - h);
                if (GENERAL && sizeof(XT) == 2 && wide) store32<float>(lo, y, out, res, off, pitch, floor, bias + h * 4, row0 + h, rows, live, any);
                else store32<XT>(lo, y, out, res, off, pitch, floor, bias + h * 4, row0 + h, rows, live, any);
                __syncwarp();
                if (whole && h + 32 < out_rows) {
                    tmem_ld32(src + d * 128 + h + 32, lo);
                } else {
#pragma unroll
                    for (int j = 0; j < 32; ++j) lo[j] = hi[j];
                }
            }
            if (whole) {
                tc_before();
                __syncwarp();
                if (lane == 0) {        // (once more for the half that has no part in it)
                    bar_arrive(d_empty + 8 * d);
                    bar_arrive(d_empty + 8 * d);
                }
                ++n_grp;
            }
        }
        // (whichever warp stored an output, all have)
        asm volatile("bar.sync 1, %0;" ::"n"(kEpiWarps * 32) : "memory");
        unsigned layers;
        asm volatile("ld.shared.u32 %0, [%1];" : "=r"(layers) : "r"(not_finite));
        if (layers) recompute<XT, PATCH, GENERAL, L>(a, layers, (int)quad, e, lane);
    } else {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kProdRegs));
        constexpr int kIssuers = E::group == 1 ? 2 : 1;
        if (warp >= kMmaWarp && warp < kMmaWarp + kIssuers && elect_one()) {
            const unsigned me = warp - kMmaWarp;
            unsigned n_chunk = 0, n_grp = 0, stage = 0, ph = 0, buf = 0, aph = 0;
            Cursor<L> cur(a);
#pragma unroll 1
            while (ok && cur.step()) {
                const int k16 = cur.t.k16, n = cur.of().n;
                const unsigned idesc = (1u << 4) | ((unsigned)E::fmt << 7) | ((unsigned)E::fmt << 10) | ((unsigned)(n >> 3) << 17) |
                                       ((unsigned)(kTcM >> 4) << 24);
                // shared-memory descriptor of B: K-major, no swizzle; 8 columns x n channels are n * 16
                // contiguous bytes, so neighbouring column groups are n * 16 and channel groups 128 bytes apart
                const unsigned long long desc0 = ((unsigned long long)n << 16) | (8ull << 32) | (1ull << 46);
                const unsigned step = 2u * n;      // in 16-byte units
                const int nch = (k16 + NS - 1) / NS;
#pragma unroll 1
                for (int c = 0; c < nch; ++c, ++n_chunk) {
                    const bool first = c % E::group == 0, last = (c + 1) % E::group == 0 || c + 1 == nch;
                    if (kIssuers == 1 || (n_chunk & 1u) == me) {
                        const int ns = min(NS, k16 - NS * c);
                        const unsigned d = n_grp & 1u;
                        if (n_chunk == me) asm volatile("griddepcontrol.wait;" ::: "memory");
                        ok = (!first || bar_wait(d_empty + 8 * d, ((n_grp >> 1) & 1u) ^ 1u)) && bar_wait(b_full + 8 * stage, ph) &&
                             bar_wait(a_full + 8 * buf, aph);
                        // all a chunk needs is there: when the other issuer's chunk has been issued, this one follows it
                        // without a gap, and whatever surrounds it here costs the tensor cores nothing
                        if (kIssuers == 2) ok = ok && bar_wait(turn + 8 * me, ((n_chunk >> 1) & 1u) ^ (me ^ 1u));
                        if (!ok) break;
                        tc_after();
                        const unsigned dst = tmem + d * 128, at = tmem_a + buf * AB, plane = step * ns;
                        const unsigned long long bt = desc0 | ((stage0 + stage * a.stage_bytes) >> 4);
                        if constexpr (P == 3) {
                            const int pa[5] = {2, 0, 1, 1, 0}, pb[5] = {0, 2, 1, 0, 1};
#pragma unroll 1
                            for (int s = 0; s < ns; ++s)
#pragma unroll
                                for (int m = 0; m < 5; ++m)
                                    mma_f16(dst, at + pa[m] * (KC / 2) + s * 8, bt + pb[m] * plane + s * step, idesc, (s | m) != 0);
#pragma unroll 1
                            for (int s = 0; s < ns; ++s) mma_f16(dst, at + s * 8, bt + s * step, idesc, 1u);
                        } else {
#pragma unroll 1
                            for (int s = 0; s < ns; ++s) mma_f16(dst, at + s * 8, bt + s * step, idesc, !(first && s == 0));
                        }
                        if (kIssuers == 2) bar_arrive(turn + 8 * (me ^ 1u));
                        mma_commit(a_empty + 8 * buf);
                        mma_commit(b_empty + 8 * stage);
                        if (last) mma_commit(d_full + 8 * d);
                    }
                    n_grp += last;
                    if (++buf == NA) { buf = 0; aph ^= 1u; }
                    if (++stage == (unsigned)a.stages) { stage = 0; ph ^= 1u; }
                }
            }
            if (!ok) {      // gave up: see the MMAs in flight end before tensor memory is given back
                mma_commit(drained + 8 * me);
                (void)bar_wait(drained + 8 * me, 0);
            }
        }
        if (warp >= kProdWarp0 && warp < kProdWarp0 + (int)S) {
            asm volatile("griddepcontrol.wait;" ::: "memory");
            // every producer copies whole chunks, the block's chunks in turn
            unsigned n = 0, mine = warp - kProdWarp0;
            int bulk_phase = -1;        // of its slot, if the last copy there was a bulk one
            Cursor<L> cur(a);
#pragma unroll 1
            while (ok && cur.step()) {
                const TcLayer& y = cur.of();
                const int k16 = cur.t.k16;
                if constexpr (PATCH) {
                    const int n_blocks = k16 ? div_of(k16, y.taps) : 0;
                    const unsigned end = n + (n_blocks + y.blocks - 1) / y.blocks;
                    const Patch t(y, cur.pt());
#pragma unroll 1
                    for (; mine < end; mine += S) {
                        const unsigned slot = mine % S;
                        const int c0 = (cur.t.kstart + (int)(mine - n) * y.blocks) * 16;
                        ok = __all_sync(0xffffffffu, bar_wait(x_empty + 8 * slot, ((mine / S) & 1u) ^ 1u));
                        if (!ok) break;
                        copy_patch<XT>(y, t, ring0 + slot * kSlot, c0, min(y.blocks * 16, y.cin - c0), lane, x_full + 8 * slot);
                    }
                    n = end;
                } else {
                    Source<XT> src;
                    const unsigned end = n + (k16 + NS - 1) / NS;
                    if (mine < end) src.open(y, cur.t, cur.pt(), lane);
#pragma unroll 1
                    for (; mine < end; mine += S) {
                        const unsigned slot = mine % S;
                        const int k = (mine - n) * NS;
                        ok = __all_sync(0xffffffffu, bar_wait(x_empty + 8 * slot, ((mine / S) & 1u) ^ 1u));
                        if (!ok) break;
                        src.chunk(ring0 + slot * kSlot, k * 16, min(NS, k16 - k) * 16, lane, x_full + 8 * slot);
                        bulk_phase = src.n_img ? (int)((mine / S) & 1u) : -1;
                    }
                    n = end;
                }
            }
            // whoever waits for them may have given up: see the copies in flight land before shared memory goes away
            asm volatile("cp.async.wait_all;" ::: "memory");
            if (!PATCH && bulk_phase >= 0) (void)bar_wait(x_full + 8 * (warp - kProdWarp0), bulk_phase);
        }
        if (warp == kLoadWarp && elect_one()) {
            unsigned stage = 0, ph = 0, used = 0;
            Cursor<L> cur(a);
#pragma unroll 1
            while (ok && cur.step()) {
                const TcLayer& y = cur.of();
                const TcTile t = cur.t;
                const unsigned char* src = y.b + (y.tiles ? (size_t)t.b16 * 16 : (size_t)cur.nt() * y.k16 * (32 * P) * y.n);
#pragma unroll 1
                for (int k = 0; k < t.k16 && ok; k += NS) {
                    const unsigned bytes = (unsigned)(min(NS, t.k16 - k) * 16 * y.n * 2 * P);
                    // (the weights do not depend on the kernel before this one: the first copies run ahead of its end)
                    if (used == (unsigned)a.stages) asm volatile("griddepcontrol.wait;" ::: "memory");
                    ok = bar_wait(b_empty + 8 * stage, ph ^ 1u);
                    if (!ok) break;
                    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(b_full + 8 * stage), "r"(bytes) : "memory");
                    bulk_load(stage0 + stage * a.stage_bytes, src, bytes, b_full + 8 * stage);
                    src += bytes;
                    ++used;
                    if (++stage == (unsigned)a.stages) { stage = 0; ph ^= 1u; }
                }
            }
            // whoever waits for them may have given up: see the copies in flight land before shared memory goes away
#pragma unroll 1
            for (unsigned i = 0; i < min(used, (unsigned)a.stages); ++i) {
                const unsigned at = (stage + a.stages - 1 - i) % a.stages;
                (void)bar_wait(b_full + 8 * at, at < stage ? ph : ph ^ 1u);
            }
        }
    }
    if (!ok)
#pragma unroll 1
        for (int l = 0; l < a.n_layers; ++l) atomicExch(a.layer[l].err, warp == kLoadWarp || warp >= kProdWarp0 ? 2 : 1);
    tc_before();
    __syncthreads();
    if (warp == kMmaWarp) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem));
}

// Memory-bound and short: one output per thread and step, consecutive threads on consecutive pixels.
__global__ void __launch_bounds__(256) tc_reduce_kernel(const __grid_constant__ TcReduce a)
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int hw = a.hw.d, n = a.width.d;
    for (int i = blockIdx.x * 256 + threadIdx.x; i < (int)a.total; i += gridDim.x * 256) {
        const int row = div_of(i, a.hw), p = i - row * hw;       // row = image * cout + channel
        const int img = row / a.cout, c = row - img * a.cout;
        const int tile = div_of(c, a.width), r = c - tile * n;
        const float* q = a.part + (((size_t)img * a.tiles + tile) * a.splits * n + r) * hw + p;
        float v = 0.0f;
#pragma unroll 4
        for (int s = 0; s < a.splits; ++s) v += __ldcg(q + (size_t)s * n * hw);
        if (a.bias) v += __ldg(a.bias + c);
        a.y[i] = a.relu ? fmaxf(v, 0.0f) : v;
    }
}

template <typename XT, bool PATCH, bool GENERAL, int L>
cudaError_t launch(const TcArgs<L>& a, int blocks, cudaStream_t st)
{
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3((unsigned)blocks);
    lc.blockDim = dim3(kThreads);
    lc.dynamicSmemBytes = kBarBytes + (size_t)a.stages * a.stage_bytes + (PATCH ? (size_t)a.slots * a.slot_bytes : kTcRingBytes);
    lc.stream = st;
    // programmatic dependent launch: set-up overlaps the tail of the kernel before it on the stream
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    lc.attrs = attr;
    lc.numAttrs = 1;
    return cudaLaunchKernelEx(&lc, tc_kernel<XT, PATCH, GENERAL, L>, a);
}

template <typename XT>
cudaError_t launch_any(bool patch, const TcArgs<kTcMaxLayers>& a, int blocks, cudaStream_t st)
{
    bool general = false;
    for (int i = 0; i < a.n_layers; ++i) general = general || a.layer[i].res || a.layer[i].chan || (sizeof(XT) == 2 && a.layer[i].y32);
    if (a.n_layers > 1) {
        if (patch) return cudaErrorInvalidValue;      // (such layers are not merged)
        return general ? launch<XT, false, true, kTcMaxLayers>(a, blocks, st) : launch<XT, false, false, kTcMaxLayers>(a, blocks, st);
    }
    TcArgs<1> one;      // (a launch's arguments are copied by the driver: few layers, few bytes)
    one.n_layers = 1; one.n_items = a.n_items; one.sched = nullptr; one.stages = a.stages; one.stage_bytes = a.stage_bytes;
    one.slots = a.slots; one.slot_bytes = a.slot_bytes;
    one.layer[0] = a.layer[0];
    if (patch) return general ? launch<XT, true, true, 1>(one, blocks, st) : launch<XT, true, false, 1>(one, blocks, st);
    return general ? launch<XT, false, true, 1>(one, blocks, st) : launch<XT, false, false, 1>(one, blocks, st);
}

template <typename XT>
cudaError_t prepare()
{
    const void* const fn[] = {(const void*)tc_kernel<XT, false, false, 1>, (const void*)tc_kernel<XT, false, true, 1>,
                              (const void*)tc_kernel<XT, false, false, kTcMaxLayers>, (const void*)tc_kernel<XT, false, true, kTcMaxLayers>,
                              (const void*)tc_kernel<XT, true, false, 1>, (const void*)tc_kernel<XT, true, true, 1>};
    for (const void* f : fn) {
        const cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxTcSmem);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace

cudaError_t launch_tc(int dt, bool patch, const TcArgs<kTcMaxLayers>& a, int blocks, cudaStream_t st)
{
    return dt == 0 ? launch_any<float>(patch, a, blocks, st) : dt == 1 ? launch_any<__half>(patch, a, blocks, st) : launch_any<__nv_bfloat16>(patch, a, blocks, st);
}

cudaError_t launch_tc_reduce(const TcReduce& a, int sms, cudaStream_t st)
{
    cudaLaunchConfig_t lc = {};
    const long long blocks = (a.total + 255) / 256;
    lc.gridDim = dim3((unsigned)(blocks < 8ll * sms ? blocks : 8ll * sms));
    lc.blockDim = dim3(256);
    lc.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    lc.attrs = attr;
    lc.numAttrs = 1;
    return cudaLaunchKernelEx(&lc, tc_reduce_kernel, a);
}

cudaError_t prepare_tc(int dt) { return dt == 0 ? prepare<float>() : dt == 1 ? prepare<__half>() : prepare<__nv_bfloat16>(); }

}  // namespace alcs
