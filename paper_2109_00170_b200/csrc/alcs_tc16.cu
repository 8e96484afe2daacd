// Pointwise convolution of 16-bit operands on the fifth-generation tensor cores (tcgen05), sm_100a.
//
// A work item is (up to 128 output channels) x (up to 256 output pixels).  As in the fp32 kernel the item's pruned weights
// are expanded to a dense tile; here the weights are the A operand and the pixels the B operand,
//     D[128 channels][pixels] += A[128 channels][64 columns] * B[64 columns][pixels]      per chunk of 64 columns,
// both read from shared memory as they were copied there: X keeps its order (rows of consecutive pixels, "MN-major"), so
// nothing is converted and no thread touches X between its copy and the multiplication.  A lane of D is a channel and its
// columns are consecutive pixels, so a thread packs two results to a word, and a warp stores whole 16-byte pieces of rows
// through a small transposing tile in shared memory.
// (With pixels as the A operand, as in alcs_tc.cu, 16 warps pack X from shared memory into tensor memory and every store instruction
// writes 64 bytes.  Measured, that kernel -> this one: 156 -> 118 channels @112x112, batch 28: 65 -> 39 us, 4.8 TB/s; 155 -> 39
// @56x56, batch 56: 28 -> 21 us; 380 -> 172 @14x14, batch 4, residual: 13.3 -> 9.2 us; ResNet-50's pointwise layers in one launch, 128x128
// input, batch 23: 47 -> 24 us, 192x192, batch 26: 90 -> 59 us.)
//
// What bounds it: the stores of an item (64 KB for 128 channels x 256 pixels take an SM 1.7 us when all SMs store), which is why two
// halves of the epilogue take items in turn, and the latency of a chunk's copies (0.4 us for 64 columns; 2.2 where rows have
// to be picked apart).
//
// 256 columns per accumulator, as the tensor core cuts off when it adds to its fp32 accumulator; longer sums are added up in
// registers with round to nearest.
//
// Registers: 64 per thread at launch (see kEpiRegs), of which the compiler spills 42 bytes (66 in merged launches); nothing says that
// it costs time, and no split of the block's registers among the roles leaves more for all of them.
//
// Roles (32 warps, one thread block per SM, persistent over items):
//   warps 0-15   epilogue: bias, residual, activation, stores, while the next item is multiplied (two accumulators); a warp takes
//                32 channels and a half or a quarter of the pixels
//   warps 16-23  producers: bring X into the ring, eight channels of a chunk each.  Images of an even number of pixels are copied
//                (16 or 8 bytes at a time) if four pixels fit a copy; else they take the pixels from what ...
//   warps 24-27  ... these have fetched: the 16-byte words that hold a chunk's rows
//   warp 28      issues the MMAs
//   warp 29      copies the weight tiles (bulk copies)
#include "alcs_tc.cuh"

namespace alcs {
namespace {

constexpr int kEpiWarps = 16, kProdWarps = 8, kRawWarps = 4, kProdWarp0 = kEpiWarps, kRawWarp0 = kProdWarp0 + kProdWarps;
constexpr int kMmaWarp = kRawWarp0 + kRawWarps, kLoadWarp = kMmaWarp + 1;
constexpr int kThreads = 1024;       // eight warpgroups (two warps idle)
// Registers per thread: 1024 threads start with 64; the epilogue, which holds 32 sums, takes from the others: 4 * 80 + 4 * 48 = 8 * 64.
constexpr int kEpiRegs = 80, kOtherRegs = 48;
static_assert(4 * kEpiRegs + 4 * kOtherRegs <= 8 * 64, "registers");
constexpr int kChunk = kTc16Chunk;   // columns per ring stage
constexpr int kRows = kChunk / kProdWarps;       // of them, a producer warp's
static_assert(kRows == 8, "a producer warp fills one row group of the swizzle");
constexpr int kAtom = 64, kAtomBytes = kChunk * kAtom * 2;     // pixels that lie together (128 bytes, the swizzle's width), for all columns of a chunk
constexpr int kGroup = 256 / kChunk;             // chunks per accumulator
constexpr int kStagingBytes = kTc16Staging;          // a warp's: 32 channels x 128 bytes

__device__ __forceinline__ void mma_ss(unsigned d, unsigned long long a, unsigned long long b, unsigned idesc, unsigned acc)
{
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\ttcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
                 ::"r"(d), "l"(a), "l"(b), "r"(idesc), "r"(acc) : "memory");
}
__device__ __forceinline__ void fence_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void sts(unsigned a, unsigned v) { asm volatile("st.shared.b32 [%0], %1;" ::"r"(a), "r"(v) : "memory"); }

// Pieces of V bytes between shared and global memory.
template <int V> struct Piece;
template <> struct Piece<16> {
    uint4 v;
    __device__ void lds(unsigned a) { asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a)); }
    __device__ void sts(unsigned a) const { asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(a), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory"); }
    __device__ void ldg(const char* p) { v = __ldg(reinterpret_cast<const uint4*>(p)); }
    __device__ void stg(char* p) const { *reinterpret_cast<uint4*>(p) = v; }
};
template <> struct Piece<8> {
    uint2 v;
    __device__ void lds(unsigned a) { asm volatile("ld.shared.v2.b32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(a)); }
    __device__ void sts(unsigned a) const { asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(a), "r"(v.x), "r"(v.y) : "memory"); }
    __device__ void ldg(const char* p) { v = __ldg(reinterpret_cast<const uint2*>(p)); }
    __device__ void stg(char* p) const { *reinterpret_cast<uint2*>(p) = v; }
};
template <> struct Piece<4> {
    unsigned v;
    __device__ void lds(unsigned a) { asm volatile("ld.shared.b32 %0, [%1];" : "=r"(v) : "r"(a)); }
    __device__ void sts(unsigned a) const { asm volatile("st.shared.b32 [%0], %1;" ::"r"(a), "r"(v) : "memory"); }
    __device__ void ldg(const char* p) { v = __ldg(reinterpret_cast<const unsigned*>(p)); }
    __device__ void stg(char* p) const { *reinterpret_cast<unsigned*>(p) = v; }
};
template <> struct Piece<2> {
    unsigned short v;
    __device__ void lds(unsigned a) { asm volatile("ld.shared.u16 %0, [%1];" : "=h"(v) : "r"(a)); }
    __device__ void sts(unsigned a) const { asm volatile("st.shared.u16 [%0], %1;" ::"r"(a), "h"(v) : "memory"); }
    __device__ void ldg(const char* p) { v = __ldg(reinterpret_cast<const unsigned short*>(p)); }
    __device__ void stg(char* p) const { *reinterpret_cast<unsigned short*>(p) = v; }
};

// Offset of pixel q, channel 0.
__device__ __forceinline__ int input_of(const TcLayer& y, int q)
{
    const int img = div_of(q, y.hw);
    return img * y.cin * y.hw_in + q - img * y.hw.d;
}

// A producer warp's view of one item: where its lanes find the pixels.  A row of an atom (64 pixels of one channel) takes
// 128 / V lanes that copy V bytes each; one by one, a lane has two neighbouring pixels.  Pixels past the end repeat the last ones
// and are not stored, columns past the last channel meet zero weights: any valid one will do.
struct Rows {
    const unsigned short* x;
    const int* cols;
    int hw_in, cin, mode, atoms;
    int off[4];          // copies: [atom], -1: not wanted; fetched rows: [atom][pixel] place in a row << 4 | byte of a 16-byte word

    __device__ __forceinline__ void open(const TcLayer& y, const TcTile& t, int pt, int lane)
    {
        x = static_cast<const unsigned short*>(y.x);
        hw_in = y.hw_in;
        cin = y.cin;
        mode = y.vec_bytes;
        cols = y.cols ? y.cols + t.kstart : nullptr;
        atoms = (y.n_px + kAtom - 1) / kAtom;
        const int q0 = pt * y.ppt;
        if (mode != kTcRaw) {
            const int ppl = mode / 2, at = (lane * ppl) & (kAtom - 1);
#pragma unroll
            for (int a = 0; a < 4; ++a) off[a] = a * kAtom + at < y.ppt ? input_of(y, min(q0 + a * kAtom + at, y.q - ppl)) : -1;
        } else {
            static_assert(kTc16Raw <= 2 * kAtom, "two atoms");
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int q = min(q0 + min((i >> 1) * kAtom + 2 * lane + (i & 1), y.ppt - 1), y.q - 1);
                const Run r(y, q, q0);
                off[i] = (r.index * y.raw_pitch + (input_of(y, q) - r.first) * 2) << 4 | (int)(((uintptr_t)x + 2u * (unsigned)r.first) & 15u);
            }
        }
    }
    // A tile's pixels as runs of consecutive elements of X (per channel), one per image.
    struct Run {
        int index, first, last;      // number in the tile; offsets of the first and last element, channel 0
        __device__ __forceinline__ Run(const TcLayer& y, int q, int q0)        // the run that pixel q belongs to
        {
            const int n = div_of(q, y.hw);
            index = n - div_of(q0, y.hw);
            first = input_of(y, max(n * y.hw.d, q0));
            last = input_of(y, min(min((n + 1) * y.hw.d, q0 + y.ppt), y.q) - 1);
        }
    };
    __device__ __forceinline__ int channel(int k) const { return (cols ? __ldg(cols + k) : min(k, cin - 1)) * hw_in; }

    // Copy columns k .. k + 7 to the rows that start at `to`.
    template <int V>
    __device__ __forceinline__ void copy(unsigned to, int k, int lane) const
    {
        constexpr int per_row = 128 / V, rows = 32 / per_row;
        const int sub = lane / per_row, at = lane % per_row * V;
#pragma unroll
        for (int c0 = 0; c0 < kRows; c0 += rows) {
            const int c = c0 + sub;
            const unsigned short* const src = x + channel(k + c);
            const unsigned dst = to + c * 128 + (((at >> 4) ^ c) << 4) + (at & 15);
#pragma unroll
            for (int a = 0; a < 4; ++a)
                if (off[a] >= 0) {
                    if constexpr (V == 16) cp_async16(dst + a * kAtomBytes, src + off[a]);
                    else cp_async_small<V>(dst + a * kAtomBytes, src + off[a], V);
                }
        }
    }
    // The same from what was fetched to `raw` as it is.
    __device__ __forceinline__ void pick(unsigned to, unsigned raw, int raw_row, int k, int lane) const
    {
#pragma unroll
        for (int a = 0; a < 2; ++a) {
            if (a >= atoms) break;
            const int o0 = off[2 * a], o1 = off[2 * a + 1];
            unsigned short lo[kRows], hi[kRows];
#pragma unroll
            for (int c = 0; c < kRows; ++c) {
                const int shift = channel(k + c) * 2;
                const unsigned r = raw + c * raw_row;
                asm volatile("ld.shared.u16 %0, [%1];" : "=h"(lo[c]) : "r"(r + (o0 >> 4) + ((o0 + shift) & 15)));
                asm volatile("ld.shared.u16 %0, [%1];" : "=h"(hi[c]) : "r"(r + (o1 >> 4) + ((o1 + shift) & 15)));
            }
#pragma unroll
            for (int c = 0; c < kRows; ++c) sts(to + a * kAtomBytes + c * 128 + (((lane >> 2) ^ c) << 4) + (lane & 3) * 4, (unsigned)lo[c] | ((unsigned)hi[c] << 16));
        }
    }
};

// (a predicate, not a branch: the copies of several rows are then prepared side by side)
__device__ __forceinline__ void cp_async16_if(bool p, unsigned dst, const void* src)
{
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %2, 0;\n\t@p cp.async.cg.shared.global [%0], [%1], 16;\n\t}" ::"r"(dst), "l"(src), "r"((unsigned)p) : "memory");
}

// A fetching warp's view of one item.  The 16-byte words of X that hold a channel's runs go, each to its byte, to a row of
// raw_pitch bytes per run: a lane takes the words lane and lane + 32 of every row.  A word that reaches beyond X (its first
// and last one may) is read by elements.  Offsets are bytes from the 16-byte word X starts in, in 32 bits: four warps, one
// to a scheduler, do this, and every dependent instruction is five cycles of theirs.
struct Fetch {
    const char* base;
    const int* cols;
    unsigned start, span;                    // where X starts; its bytes
    unsigned first[2], bytes[2], word[2];    // of the run: byte offset (channel 0), bytes (0: none); the word's byte in it

    __device__ __forceinline__ Fetch(const TcLayer& y, const TcTile& t, int pt, int lane)
    {
        start = (unsigned)(uintptr_t)y.x & 15u;
        base = static_cast<const char*>(y.x) - start;
        span = 2u * (unsigned)(y.n_img * y.cin * y.hw_in);
        cols = y.cols ? y.cols + t.kstart : nullptr;
        const int q0 = pt * y.ppt, q1 = min(q0 + y.ppt, y.q), per_run = y.raw_pitch >> 4, n0 = div_of(q0, y.hw);
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const int w = lane + 32 * i, run = w / per_run, q = max((n0 + run) * y.hw.d, q0);
            first[i] = bytes[i] = word[i] = 0;
            if (q >= q1) continue;
            const Rows::Run r(y, q, q0);
            first[i] = start + 2u * (unsigned)r.first;
            bytes[i] = (r.last - r.first + 1) * 2;
            word[i] = (w - run * per_run) * 16;
        }
    }
    // Fetch 16 rows; did this lane store elements itself?
    __device__ __forceinline__ bool rows(const TcLayer& y, unsigned to, int k, int lane) const
    {
        to += lane * 16;
        bool stored = false;
#pragma unroll 1
        for (int r0 = 0; r0 < kChunk / kRawWarps; r0 += 4) {
            unsigned at[4][2];
            bool edge = false;
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const unsigned row = 2u * (unsigned)((cols ? __ldg(cols + k + r0 + r) : min(k + r0 + r, y.cin - 1)) * y.hw_in);
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    const unsigned from = row + first[i], w = (from & ~15u) + word[i];
                    const bool wanted = bytes[i] && w < from + bytes[i], inside = w - start <= span - 16u && span >= 16u;
                    cp_async16_if(wanted && inside, to + (r0 + r) * y.raw_row + i * 512, base + w);
                    at[r][i] = wanted && !inside ? w : 0xffffffffu;
                    edge = edge || (wanted && !inside);
                }
            }
            stored = stored || edge;
            if (edge)
#pragma unroll
                for (int r = 0; r < 4; ++r)
#pragma unroll
                    for (int i = 0; i < 2; ++i)
#pragma unroll 1
                        for (unsigned b = at[r][i]; at[r][i] != 0xffffffffu && b < at[r][i] + 16; b += 2)
                            if (b - start < span) {
                                const unsigned short v = ld_x(reinterpret_cast<const unsigned short*>(base + b));
                                asm volatile("st.shared.u16 [%0], %1;" ::"r"(to + (r0 + r) * y.raw_row + i * 512 + (b - at[r][i])), "h"(v) : "memory");
                            }
        }
        return stored;
    }
};

// A warp's 32 channels x `row_bytes` (64 or 128) of the item's output, between its staging tile and global memory, in pieces of V bytes.
// Piece j of row r lies at j ^ (r & 7), so that both a lane per row and consecutive lanes along a row are free of bank conflicts.
// `chan` is this lane's row's channel; q0 .. end: pixels; e: bytes per element.
template <int V, bool LOAD>
__device__ __forceinline__ void rows_io(const TcLayer& y, char* base, unsigned staging, int chan, int q0, int end, int row_bytes, int e, int lane)
{
    const int per_row = row_bytes / V, lanes = min(per_row, 32), step = 32 / lanes;       // powers of two
    const unsigned pitch = (unsigned)(y.hw.d * e);
    const int shift = e == 4 ? 2 : 1;
    constexpr int U = LOAD ? 2 : 4;      // pieces in flight per lane (four loads of the residual would spill)
#pragma unroll 1
    for (int first = 0; first < per_row; first += 32) {
        const int at = (first + (lane & (lanes - 1))) * V, q = q0 + (at >> shift);
        const bool live = q < end;
        const int img = div_of(live ? q : 0, y.hw), p = (live ? q : 0) - img * y.hw.d;
        char* const g = base + ((size_t)img * y.cout * y.hw.d + p) * e;
        int r = lane / lanes;
#pragma unroll 1
        for (int i0 = 0; i0 < lanes; i0 += U, r += U * step) {       // (4 <= lanes)
            Piece<V> v[U];
            int c[U];
#pragma unroll
            for (int i = 0; i < U; ++i) {
                const int at_row = r + i * step;
                c[i] = __shfl_sync(0xffffffffu, chan, at_row);
                if (!live) c[i] = -1;
                if (LOAD) {
                    if (c[i] >= 0) v[i].ldg(g + (unsigned)c[i] * pitch);
                } else {
                    v[i].lds(staging + at_row * 128 + (((at >> 4) ^ (at_row & 7)) << 4) + (at & 15));
                }
            }
#pragma unroll
            for (int i = 0; i < U; ++i) {
                if (c[i] < 0) continue;
                const int at_row = r + i * step;
                if (LOAD) v[i].sts(staging + at_row * 128 + (((at >> 4) ^ (at_row & 7)) << 4) + (at & 15));
                else v[i].stg(g + (unsigned)c[i] * pitch);
            }
        }
    }
}

template <bool LOAD>
__device__ __forceinline__ void rows_any(const TcLayer& y, int vec, char* base, unsigned staging, int chan, int q0, int end, int row_bytes, int e, int lane)
{
    if (vec == 16) rows_io<16, LOAD>(y, base, staging, chan, q0, end, row_bytes, e, lane);
    else if (vec == 8) rows_io<8, LOAD>(y, base, staging, chan, q0, end, row_bytes, e, lane);
    else if (vec == 4) rows_io<4, LOAD>(y, base, staging, chan, q0, end, row_bytes, e, lane);
    else rows_io<2, LOAD>(y, base, staging, chan, q0, end, row_bytes, e, lane);
}

__device__ __forceinline__ unsigned pack2(float a, float b, const __half*) { const __half2 h = __floats2half2_rn(a, b); return *reinterpret_cast<const unsigned*>(&h); }
__device__ __forceinline__ unsigned pack2(float a, float b, const __nv_bfloat16*) { const __nv_bfloat162 h = __floats2bfloat162_rn(a, b); return *reinterpret_cast<const unsigned*>(&h); }
__device__ __forceinline__ float2 unpack2(unsigned v, const __half*) { return __half22float2(*reinterpret_cast<const __half2*>(&v)); }
__device__ __forceinline__ float2 unpack2(unsigned v, const __nv_bfloat16*) { return make_float2(__uint_as_float(v << 16), __uint_as_float(v & 0xffff0000u)); }

__device__ __forceinline__ void add2(float& a, float& b, float c)       // two additions
{
    asm("{\n\t.reg .b64 x, y;\n\tmov.b64 x, {%0, %1};\n\tmov.b64 y, {%2, %2};\n\tadd.rn.f32x2 x, x, y;\n\tmov.b64 {%0, %1}, x;\n\t}" : "+f"(a), "+f"(b) : "f"(c));
}
__device__ __forceinline__ unsigned relu2(unsigned v, const __half*) { unsigned r; asm("max.f16x2 %0, %1, %2;" : "=r"(r) : "r"(v), "r"(0u)); return r; }
__device__ __forceinline__ unsigned relu2(unsigned v, const __nv_bfloat16*) { unsigned r; asm("max.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(v), "r"(0u)); return r; }

// 32 pixels of this lane's channel: bias, residual (in the staging tile already), activation, one rounding, into the staging tile.
// piece0: the first of the row's 16-byte pieces they take.  (Rounding keeps the sign, so the activation can come behind it.)
template <typename XT>
__device__ __forceinline__ void finish32(float (&v)[32], unsigned row, int lane, int piece0, bool wide, bool res, float bias, bool relu)
{
    const XT* const tag = nullptr;
#pragma unroll
    for (int j = 0; j < 32; j += 2) add2(v[j], v[j + 1], bias);
    if (wide) {
        const float floor = relu ? 0.0f : __int_as_float(0x7fffffff);        // (fmaxf returns the operand that is a number)
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const unsigned s = row + ((j ^ (lane & 7)) << 4);
            Piece<16> p;
            if (res) {
                p.lds(s);
                v[4 * j] += __uint_as_float(p.v.x); v[4 * j + 1] += __uint_as_float(p.v.y);
                v[4 * j + 2] += __uint_as_float(p.v.z); v[4 * j + 3] += __uint_as_float(p.v.w);
            }
            p.v = make_uint4(__float_as_uint(fmaxf(v[4 * j], floor)), __float_as_uint(fmaxf(v[4 * j + 1], floor)),
                             __float_as_uint(fmaxf(v[4 * j + 2], floor)), __float_as_uint(fmaxf(v[4 * j + 3], floor)));
            p.sts(s);
        }
        return;
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const unsigned s = row + (((piece0 + j) ^ (lane & 7)) << 4);
        Piece<16> p;
        if (res) {
            p.lds(s);
            const unsigned w[4] = {p.v.x, p.v.y, p.v.z, p.v.w};
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const float2 r = unpack2(w[k], tag);
                v[8 * j + 2 * k] += r.x;
                v[8 * j + 2 * k + 1] += r.y;
            }
        }
        unsigned w[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            w[k] = pack2(v[8 * j + 2 * k], v[8 * j + 2 * k + 1], tag);
            if (relu) w[k] = relu2(w[k], tag);
        }
        p.v = make_uint4(w[0], w[1], w[2], w[3]);
        p.sts(s);
    }
}

template <typename XT, int L>
__global__ void __launch_bounds__(kThreads, 1) tc16_kernel(const __grid_constant__ TcArgs<L> a)
{
    extern __shared__ __align__(1024) unsigned char smem[];
    const unsigned s0 = smem_u32(smem);
    const unsigned full = s0, empty = s0 + 64, d_full = s0 + 128, d_empty = s0 + 144, tmem_slot = s0 + 160, drained = s0 + 168;
    const unsigned not_finite = s0 + 176;      // layers whose items had sums that are not finite, a bit each
    const unsigned raw_full = s0 + 192, raw_empty = s0 + 224;
    const unsigned staging0 = s0 + kTc16Header, stage0 = staging0 + kEpiWarps * kStagingBytes;
    const unsigned S = a.stages, R = a.raw_slots, raw0 = stage0 + S * a.stage_bytes;
    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;

    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (warp == kMmaWarp) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(tmem_slot) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    } else if (warp == kLoadWarp && lane == 0) {
#pragma unroll 1
        for (unsigned i = 0; i < S; ++i) {
            bar_init(full + 8 * i, kProdWarps * 32 + 1);
            bar_init(empty + 8 * i, 1);
        }
#pragma unroll 1
        for (int i = 0; i < 2; ++i) {
            bar_init(d_full + 8 * i, 1);
            bar_init(d_empty + 8 * i, kEpiWarps);
        }
#pragma unroll 1
        for (unsigned i = 0; i < R; ++i) {
            bar_init(raw_full + 8 * i, kRawWarps * 32);
            bar_init(raw_empty + 8 * i, kProdWarps);
        }
        bar_init(drained, 1);
        asm volatile("st.shared.u32 [%0], 0;" ::"r"(not_finite) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    tc_before();
    __syncthreads();
    tc_after();
    unsigned tmem;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(tmem) : "r"(tmem_slot));
    bool ok = true;

    if (warp < kEpiWarps) {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kEpiRegs));
        const int quad = warp & 3, quarter = warp >> 2;
        // Items of one accumulator are taken by the two halves of the warps in turn, so that one half's stores, which wait for memory,
        // run beside the other's arithmetic; the sums of longer ones are added up by all warps, and so is a block's only item.
        const bool alone = a.n_items <= (int)gridDim.x;
        const unsigned staging = staging0 + warp * kStagingBytes, my_row = staging + lane * 128;
        unsigned n_grp = 0;
        asm volatile("griddepcontrol.wait;" ::: "memory");
        Cursor<L, true> cur(a);
#pragma unroll 1
        while (ok && cur.step()) {
            const TcLayer& y = cur.of();
            const int groups = (cur.t.k16 + kTc16Group - 1) / kTc16Group;
            const bool whole = groups <= 1 && !alone;
            if (whole && (quarter >> 1) != (int)(groups ? n_grp & 1u : 0)) {
                n_grp += groups;
                continue;
            }
            const int row = quad * 32 + lane, nt = cur.nt(), q0 = cur.pt() * y.ppt, q1 = min(q0 + y.ppt, y.q);
            int chan = row < y.n ? y.chan ? __ldg(y.chan + nt * y.n + row) : nt * y.n + row : -1;
            if (chan >= y.cout) chan = -1;
            const float bias = y.bias && chan >= 0 ? __ldg(y.bias + chan) : 0.0f;
            const bool wide = y.y32, res = y.res != nullptr;
            const int e = wide ? 4 : 2;
            // this warp's pixels: a half or a quarter of the item's, in blocks of 32; a round of the staging tile takes 128 bytes of a row
            const int parts = whole ? 2 : 4, part = quarter & (parts - 1);
            const int blocks = y.n_px / 32, b0 = part * blocks / parts, per_round = wide ? 1 : 2;
            const int end = quad * 32 < y.n ? min((part + 1) * blocks / parts, (q1 - q0 + 31) / 32) : b0;
            char* const out = static_cast<char*>(y.y);
            char* const rsd = const_cast<char*>(static_cast<const char*>(y.res));
            if (res && b0 < end) {      // what the end of the item will add: on its way while the item is multiplied
                rows_any<true>(y, y.res_vec, rsd, staging, chan, q0 + b0 * 32, q1, min(per_round, end - b0) * 32 * e, e, lane);
                if (chan >= 0)
#pragma unroll 1
                    for (int b = b0 + per_round; b < end; b += per_round) {
                        const int q = q0 + b * 32, img = div_of(q, y.hw);
                        asm volatile("prefetch.global.L2 [%0];" ::"l"(rsd + (((size_t)img * y.cout + chan) * y.hw.d + (q - img * y.hw.d)) * e));
                    }
            }
            float v[32];               // sums of block b0, the only one where an item has several accumulators (128 pixels at most)
            const unsigned src = tmem + ((unsigned)quad << 21);
            unsigned d = n_grp & 1u;
            auto release = [&] {
                tc_before();
                __syncwarp();
                if (lane == 0) {
                    bar_arrive(d_empty + 8 * d);
                    if (whole) bar_arrive(d_empty + 8 * d);        // (for a warp of the half that has no part in it)
                }
            };
#pragma unroll
            for (int j = 0; j < 32; ++j) v[j] = 0.0f;
            if (groups > 1) {
#pragma unroll 1
                for (int g = 0; g < groups; ++g, ++n_grp) {
                    d = n_grp & 1u;
                    ok = __all_sync(0xffffffffu, bar_wait(d_full + 8 * d, (n_grp >> 1) & 1u));
                    if (!ok) break;
                    tc_after();
                    if (b0 < end) {
#pragma unroll
                        for (int j = 0; j < 32; j += 16) {
                            float t[16];
                            tmem_ld16(src + d * 256 + b0 * 32 + j, t);
                            tmem_wait_ld(t);
#pragma unroll
                            for (int k = 0; k < 16; ++k) v[j + k] += t[k];
                        }
                    }
                    release();
                }
            } else if (groups == 1) {
                ok = __all_sync(0xffffffffu, bar_wait(d_full + 8 * d, (n_grp >> 1) & 1u));
                tc_after();
                if (ok && b0 >= end) release();
            }
            if (!ok) break;
#pragma unroll 1
            for (int b = b0; b < end; b += per_round) {
                const int now = min(per_round, end - b);
                if (b > b0) {
                    __syncwarp();           // (the stores of the round before have read the tile)
                    if (res) rows_any<true>(y, y.res_vec, rsd, staging, chan, q0 + b * 32, q1, now * 32 * e, e, lane);
#pragma unroll
                    for (int j = 0; j < 32; ++j) v[j] = 0.0f;       // (several rounds: no sums in registers)
                }
                __syncwarp();
#pragma unroll 1
                for (int h = 0; h < now; ++h) {
                    if (groups == 1) {
                        tmem_ld32(src + d * 256 + (b + h) * 32, v);
                        tmem_wait_ld(v);
                        if (b + h + 1 == end) release();
                    } else if (h) {
#pragma unroll
                        for (int j = 0; j < 32; ++j) v[j] = 0.0f;       // (a tile that keeps nothing)
                    }
                    if (quad == 0 && groups) {      // (an input that is not finite reaches every channel of the tile, so one of them tells)
                        float t[2] = {0.0f, 0.0f};
#pragma unroll
                        for (int j = 0; j < 32; ++j) t[j & 1] = fmaf(v[j], 0.0f, t[j & 1]);
                        const float s = t[0] + t[1];
                        if (lane == 0 && s != s) asm volatile("red.shared.or.b32 [%0], %1;" ::"r"(not_finite), "r"(1u << (L > 1 ? cur.layer : 0)) : "memory");
                    }
                    finish32<XT>(v, my_row, lane, h * 4, wide, res, bias, y.relu != 0);
                }
                __syncwarp();
                rows_any<false>(y, y.y_vec, out, staging, chan, q0 + b * 32, q1, now * 32 * e, e, lane);
            }
            __syncwarp();
            n_grp += groups == 1;
        }
        // (whichever warp stored an output, all have)
        asm volatile("bar.sync 1, %0;" ::"n"(kEpiWarps * 32) : "memory");
        unsigned layers;
        asm volatile("ld.shared.u32 %0, [%1];" : "=r"(layers) : "r"(not_finite));
        if (layers && warp < 8) recompute<XT, false, true, L>(a, layers, quad, quarter, lane);
    } else {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kOtherRegs));
        if (warp >= kProdWarp0 && warp < kProdWarp0 + kProdWarps) {
            const int pw = warp - kProdWarp0;
            unsigned stage = 0, ph = 1, slot = 0, raw_ph = 0;
            asm volatile("griddepcontrol.wait;" ::: "memory");
            Cursor<L, true> cur(a);
#pragma unroll 1
            while (ok && cur.step()) {
                const TcLayer& y = cur.of();
                Rows rows;
                rows.open(y, cur.t, cur.pt(), lane);
#pragma unroll 1
                for (int k0 = 0; k0 < cur.t.k16 * 16; k0 += kChunk) {
                    ok = __all_sync(0xffffffffu, bar_wait(empty + 8 * stage, ph));
                    if (!ok) break;
                    const unsigned to = stage0 + stage * a.stage_bytes + a.slot_bytes + pw * (kRows * 128);
                    const int k = k0 + pw * kRows;
                    if (rows.mode == kTcRaw) {
                        ok = __all_sync(0xffffffffu, bar_wait(raw_full + 8 * slot, raw_ph));
                        if (!ok) break;
                        if (k < cur.t.k16 * 16) rows.pick(to, raw0 + slot * a.raw_bytes + pw * kRows * y.raw_row, y.raw_row, k, lane);
                        fence_async();
                        bar_arrive(full + 8 * stage);
                        __syncwarp();
                        if (lane == 0) bar_arrive(raw_empty + 8 * slot);
                        if (++slot == R) { slot = 0; raw_ph ^= 1u; }
                    } else if (k >= cur.t.k16 * 16) {
                        bar_arrive(full + 8 * stage);
                    } else {
                        if (rows.mode == 16) rows.copy<16>(to, k, lane);
                        else rows.copy<8>(to, k, lane);
                        cp_async_arrive(full + 8 * stage);
                    }
                    if (++stage == S) { stage = 0; ph ^= 1u; }
                }
            }
            // whoever waits for them may have given up: see the copies in flight land before shared memory goes away
            asm volatile("cp.async.wait_all;" ::: "memory");
        } else if (warp >= kRawWarp0 && warp < kRawWarp0 + kRawWarps && R) {
            const int k_mine = (warp - kRawWarp0) * (kChunk / kRawWarps);
            unsigned slot = 0, ph = 1;
            asm volatile("griddepcontrol.wait;" ::: "memory");
            Cursor<L, true> cur(a);
#pragma unroll 1
            while (ok && cur.step()) {
                const TcLayer& y = cur.of();
                if (y.vec_bytes != kTcRaw) continue;
                const Fetch f(y, cur.t, cur.pt(), lane);
#pragma unroll 1
                for (int k0 = 0; k0 < cur.t.k16 * 16; k0 += kChunk) {
                    ok = __all_sync(0xffffffffu, bar_wait(raw_empty + 8 * slot, ph));
                    if (!ok) break;
                    const bool stored = k0 + k_mine < cur.t.k16 * 16 && f.rows(y, raw0 + slot * a.raw_bytes + k_mine * y.raw_row, k0 + k_mine, lane);
                    if (stored) {
                        // The arrival of copies says nothing of a thread's own stores; an ordinary one orders both, once the copies are done.
                        asm volatile("cp.async.wait_all;" ::: "memory");
                        bar_arrive(raw_full + 8 * slot);
                    } else {
                        cp_async_arrive(raw_full + 8 * slot);
                    }
                    if (++slot == R) { slot = 0; ph ^= 1u; }
                }
            }
            asm volatile("cp.async.wait_all;" ::: "memory");
        } else if (warp == kMmaWarp) {
            if (elect_one()) {
                unsigned n_grp = 0, stage = 0, ph = 0;
                bool first_wait = true;
                Cursor<L, true> cur(a);
#pragma unroll 1
                while (ok && cur.step()) {
                    const int k16 = cur.t.k16, n = cur.of().n, pixels = cur.of().n_px;
                    constexpr unsigned fmt = Elem<XT>::fmt;
                    const unsigned idesc = (1u << 4) | (fmt << 7) | (fmt << 10) | (1u << 16) | ((unsigned)(pixels >> 3) << 17) | ((unsigned)(128 >> 4) << 24);
                    // A, the weights: K-major, no swizzle; 8 columns x n channels are n * 16 contiguous bytes, so neighbouring column
                    // groups are n * 16 and channel groups 128 bytes apart.  (Rows past n: whatever follows, never stored.)
                    const unsigned long long da = ((unsigned long long)n << 16) | (8ull << 32) | (1ull << 46);
                    // B, the pixels: MN-major, 128-byte swizzle; atoms of 64 pixels kAtomBytes, groups of 8 columns 1024 bytes apart
                    const unsigned long long db = ((unsigned long long)(kAtomBytes >> 4) << 16) | ((1024ull >> 4) << 32) | (1ull << 46) | (2ull << 61);
                    const int nch = (k16 * 16 + kChunk - 1) / kChunk;
#pragma unroll 1
                    for (int c = 0; c < nch; ++c) {
                        const bool first = c % kGroup == 0, last = (c + 1) % kGroup == 0 || c + 1 == nch;
                        const unsigned d = n_grp & 1u;
                        if (first_wait) asm volatile("griddepcontrol.wait;" ::: "memory");
                        first_wait = false;
                        ok = (!first || bar_wait(d_empty + 8 * d, ((n_grp >> 1) & 1u) ^ 1u)) && bar_wait(full + 8 * stage, ph);
                        if (!ok) break;
                        tc_after();
                        fence_async();
                        const unsigned base = stage0 + stage * a.stage_bytes, dst = tmem + d * 256;
                        const unsigned long long at = da | (base >> 4), bt = db | ((base + a.slot_bytes) >> 4);
                        const int ns = min(kChunk / 16, k16 - c * (kChunk / 16));
#pragma unroll 1
                        for (int s = 0; s < ns; ++s) mma_ss(dst, at + (unsigned)(2 * n * s), bt + (unsigned)(128 * s), idesc, !(first && s == 0));
                        mma_commit(empty + 8 * stage);
                        if (last) mma_commit(d_full + 8 * d);
                        n_grp += last;
                        if (++stage == S) { stage = 0; ph ^= 1u; }
                    }
                }
                if (!ok) {      // gave up: see the MMAs in flight end before tensor memory is given back
                    mma_commit(drained);
                    (void)bar_wait(drained, 0);
                }
            }
        } else if (warp == kLoadWarp) {
            if (elect_one()) {
                unsigned stage = 0, ph = 1, used = 0;
                Cursor<L, true> cur(a);
#pragma unroll 1
                while (ok && cur.step()) {
                    const TcLayer& y = cur.of();
                    const TcTile t = cur.t;
                    const unsigned char* src = y.b + (y.tiles ? (size_t)t.b16 * 16 : (size_t)cur.nt() * y.k16 * 32 * y.n);
#pragma unroll 1
                    for (int k = 0; k < t.k16 && ok; k += kChunk / 16) {
                        const unsigned bytes = (unsigned)(min(kChunk / 16, t.k16 - k) * 32 * y.n);
                        // (the weights do not depend on the kernel before this one: the first copies run ahead of its end)
                        if (used == S) asm volatile("griddepcontrol.wait;" ::: "memory");
                        ok = bar_wait(empty + 8 * stage, ph);
                        if (!ok) break;
                        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(full + 8 * stage), "r"(bytes) : "memory");
                        bulk_load(stage0 + stage * a.stage_bytes, src, bytes, full + 8 * stage);
                        src += bytes;
                        ++used;
                        if (++stage == S) { stage = 0; ph ^= 1u; }
                    }
                }
                asm volatile("griddepcontrol.wait;" ::: "memory");
                // whoever waits for them may have given up: see the copies in flight land before shared memory goes away (the phase
                // ends with the producers' copies; where those gave up, too, the wait runs out long after the bulk copy has landed)
#pragma unroll 1
                for (unsigned i = 0; i < min(used, S); ++i) {
                    const unsigned at = (stage + S - 1 - i) % S;
                    (void)bar_wait(full + 8 * at, at < stage ? ph ^ 1u : ph);
                }
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

template <typename XT, int L>
cudaError_t launch(const TcArgs<L>& a, int blocks, cudaStream_t st)
{
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3((unsigned)blocks);
    lc.blockDim = dim3(kThreads);
    lc.dynamicSmemBytes = kTc16Header + kEpiWarps * kStagingBytes + (size_t)a.stages * a.stage_bytes + (size_t)a.raw_slots * a.raw_bytes;
    lc.stream = st;
    // programmatic dependent launch: set-up overlaps the tail of the kernel before it on the stream
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    lc.attrs = attr;
    lc.numAttrs = 1;
    return cudaLaunchKernelEx(&lc, tc16_kernel<XT, L>, a);
}

template <typename XT>
cudaError_t launch_any(const TcArgs<kTcMaxLayers>& a, int blocks, cudaStream_t st)
{
    if (a.n_layers > 1) return launch<XT, kTcMaxLayers>(a, blocks, st);
    TcArgs<1> one;      // (a launch's arguments are copied by the driver: few layers, few bytes)
    one.n_layers = 1; one.n_items = a.n_items; one.sched = nullptr; one.stages = a.stages; one.stage_bytes = a.stage_bytes;
    one.slots = a.slots; one.slot_bytes = a.slot_bytes; one.raw_slots = a.raw_slots; one.raw_bytes = a.raw_bytes;
    one.layer[0] = a.layer[0];
    return launch<XT, 1>(one, blocks, st);
}

}  // namespace

cudaError_t launch_tc16(int dt, const TcArgs<kTcMaxLayers>& a, int blocks, cudaStream_t st)
{
    return dt == 1 ? launch_any<__half>(a, blocks, st) : launch_any<__nv_bfloat16>(a, blocks, st);
}

cudaError_t prepare_tc16(int dt)
{
    const void* const fn[2][2] = {{(const void*)tc16_kernel<__half, 1>, (const void*)tc16_kernel<__half, kTcMaxLayers>},
                                  {(const void*)tc16_kernel<__nv_bfloat16, 1>, (const void*)tc16_kernel<__nv_bfloat16, kTcMaxLayers>}};
    for (const void* f : fn[dt == 2]) {
        const cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace alcs
