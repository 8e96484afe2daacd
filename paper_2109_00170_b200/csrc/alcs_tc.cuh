// Device code shared by the two tcgen05 kernels (alcs_tc.cu; alcs_tc16.cu: 16-bit operands at stride 1): barriers and
// tensor-core instructions, the walk over a block's items, and outputs that the tensor cores cannot give.
#ifndef ALCS_TC_CUH_
#define ALCS_TC_CUH_

#include "alcs_tc.h"

#include <cuda_bf16.h>
#include <cuda_fp16.h>

namespace alcs {
namespace {

// A bounded wait gives up after this many polls, about a second (the limit of the library's other kernels).  It is
// only ever started behind griddepcontrol.wait, so that the time a predecessor still runs does not count against it.
constexpr unsigned kPolls = 1u << 21;

__device__ __forceinline__ unsigned smem_u32(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void bar_init(unsigned bar, unsigned count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void bar_arrive(unsigned bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool bar_wait(unsigned bar, unsigned parity)
{
#pragma unroll 1
    for (unsigned i = 0; i < kPolls; ++i) {
        unsigned ok;
        asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                     : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
        if (ok) return true;
    }
    return false;
}
__device__ __forceinline__ bool elect_one()
{
    unsigned ok;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(ok));
    return ok != 0;
}
__device__ __forceinline__ void tc_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ void mma_f16(unsigned d, unsigned a, unsigned long long b, unsigned idesc, unsigned acc)
{
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\ttcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
                 ::"r"(d), "r"(a), "l"(b), "r"(idesc), "r"(acc) : "memory");
}
__device__ __forceinline__ void mma_commit(unsigned bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tmem_st4(unsigned addr, const unsigned (&v)[4])
{
    asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]) : "memory");
}
__device__ __forceinline__ void tmem_ld16(unsigned addr, float* v)
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
                 : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7]),
                   "=f"(v[8]), "=f"(v[9]), "=f"(v[10]), "=f"(v[11]), "=f"(v[12]), "=f"(v[13]), "=f"(v[14]), "=f"(v[15]) : "r"(addr));
}

__device__ __forceinline__ void tmem_ld32(unsigned addr, float (&v)[32])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
                 "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
                 : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7]),
                   "=f"(v[8]), "=f"(v[9]), "=f"(v[10]), "=f"(v[11]), "=f"(v[12]), "=f"(v[13]), "=f"(v[14]), "=f"(v[15]),
                   "=f"(v[16]), "=f"(v[17]), "=f"(v[18]), "=f"(v[19]), "=f"(v[20]), "=f"(v[21]), "=f"(v[22]), "=f"(v[23]),
                   "=f"(v[24]), "=f"(v[25]), "=f"(v[26]), "=f"(v[27]), "=f"(v[28]), "=f"(v[29]), "=f"(v[30]), "=f"(v[31])
                 : "r"(addr));
}

// One element of X: read once per item, so it takes no room in L1.
__device__ __forceinline__ unsigned short ld_x(const unsigned short* p)
{
    unsigned short v;
    asm volatile("ld.global.nc.L1::no_allocate.u16 %0, [%1];" : "=h"(v) : "l"(p));
    return v;
}

// Wait for loads from tensor memory; the values may not be touched before (they are tied to the wait here).
template <int N>
__device__ __forceinline__ void tmem_wait_ld(float (&v)[N])
{
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < N; ++i) asm volatile("" : "+f"(v[i]));
}

template <typename XT> struct Elem;
template <> struct Elem<float> {
    using raw = float;
    static constexpr int planes = 3, fmt = 1;
    static constexpr int group = 1;       // chunks per accumulator
    static constexpr int abufs = 2;       // chunks in tensor memory
};
template <> struct Elem<__half> {
    using raw = unsigned short;
    static constexpr int planes = 1, fmt = 0, group = 2, abufs = 3;
};
template <> struct Elem<__nv_bfloat16> {
    using raw = unsigned short;
    static constexpr int planes = 1, fmt = 1, group = 2, abufs = 3;
};

__device__ __forceinline__ int div_of(int n, const TcDiv& d) { return (int)((unsigned long long)(unsigned)n * d.mul >> d.shift); }

// A role's walk over the block's items.  Where the tiles differ, what the next item needs from the tile table
// is loaded one item ahead.  AHEAD: from the list of items two ahead, so that no step waits for memory; of use to short items
// (the other kernel's merged launches lose 1 % by it: a register and a load more in every role).
template <int L, bool AHEAD = false>
struct Cursor {
    const TcArgs<L>& a;
    int item, next_item, after = -1, at, layer = 0, next_layer = 0;
    TcTile t, next;

    __device__ __forceinline__ explicit Cursor(const TcArgs<L>& a_) : a(a_), at(blockIdx.x)
    {
        next_item = L > 1 && a.sched ? __ldg(a.sched + at) : at;
        if (AHEAD && L > 1 && a.sched) after = __ldg(a.sched + at + gridDim.x);
        peek();
    }
    __device__ __forceinline__ const TcLayer& of() const { return a.layer[L > 1 ? layer : 0]; }
    __device__ __forceinline__ const TcLayer& next_of() const { return a.layer[L > 1 ? next_layer : 0]; }
    __device__ __forceinline__ bool has_next() const { return (unsigned)next_item < (unsigned)a.n_items; }
    static __device__ __forceinline__ int channel_tile(const TcLayer& y, int i)
    {
        if (y.tile_major) return div_of(i - y.first_item, y.px_tiles);
        const int r = i - y.first_item;
        return r - div_of(r, y.n_tiles) * y.n_tiles.d;
    }
    __device__ __forceinline__ int nt() const { return channel_tile(of(), item); }
    __device__ __forceinline__ int next_nt() const { return channel_tile(next_of(), next_item); }
    __device__ __forceinline__ int pt() const
    {
        const TcLayer& y = of();
        const int r = item - y.first_item;
        return y.tile_major ? r - div_of(r, y.px_tiles) * y.px_tiles.d : div_of(r, y.n_tiles);
    }
    __device__ __forceinline__ void peek()
    {
        if (!has_next()) return;
        if (L > 1) {
            next_layer = 0;
#pragma unroll 1
            while (next_layer + 1 < a.n_layers && next_item >= a.layer[next_layer + 1].first_item) ++next_layer;
        }
        const TcLayer& y = next_of();
        if (y.tiles) {
            const TcTile* p = y.tiles + next_nt();
            next.b16 = __ldg(&p->b16);
            next.k16 = __ldg(&p->k16);
            next.kstart = __ldg(&p->kstart);
        } else {
            next.k16 = y.k16;
            next.kstart = 0;
        }
    }
    __device__ __forceinline__ bool step()
    {
        if (!has_next()) return false;
        item = next_item;
        at += gridDim.x;
        if (AHEAD && L > 1 && a.sched) {        // (the list ends with a row of -1)
            next_item = after;
            if (has_next()) after = __ldg(a.sched + at + gridDim.x);
        } else {
            next_item = L > 1 && a.sched ? __ldg(a.sched + at) : at;
        }
        layer = next_layer;
        t = next;
        peek();
        return true;
    }
};

__device__ __forceinline__ void cp_async16(unsigned dst, const void* src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
template <int B>
__device__ __forceinline__ void cp_async_small(unsigned dst, const void* src, unsigned bytes)      // bytes = B, or 0: write zeros
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;" ::"r"(dst), "l"(src), "n"(B), "r"(bytes) : "memory");
}

__device__ __forceinline__ void st_slot(unsigned addr, unsigned short v) { asm volatile("st.shared.u16 [%0], %1;" ::"r"(addr), "h"(v) : "memory"); }

__device__ __forceinline__ void cp_async_arrive(unsigned bar)      // one arrival once this thread's copies so far have landed
{
    asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ void bulk_load(unsigned dst, const void* src, unsigned bytes, unsigned bar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst), "l"(src), "r"(bytes), "r"(bar)
                 : "memory");
}

__device__ __forceinline__ void put(float* p, float v) { *p = v; }
__device__ __forceinline__ void put(__half* p, float v) { *p = __float2half_rn(v); }
__device__ __forceinline__ void put(__nv_bfloat16* p, float v) { *p = __float2bfloat16_rn(v); }

// Output channel of row r of the channel tiles (-1: none).
__device__ __forceinline__ int channel_of(const TcLayer& y, int r) { return y.chan ? __ldg(y.chan + r) : r < y.cout ? r : -1; }

template <typename XT> __device__ __forceinline__ bool special(typename Elem<XT>::raw v);      // infinite or not a number?
template <> __device__ __forceinline__ bool special<float>(float v) { return (__float_as_uint(v) & 0x7f800000u) == 0x7f800000u; }
template <> __device__ __forceinline__ bool special<__half>(unsigned short v) { return (v & 0x7c00u) == 0x7c00u; }
template <> __device__ __forceinline__ bool special<__nv_bfloat16>(unsigned short v) { return (v & 0x7f80u) == 0x7f80u; }

template <typename XT> __device__ __forceinline__ float value(typename Elem<XT>::raw v);
template <> __device__ __forceinline__ float value<float>(float v) { return v; }
template <> __device__ __forceinline__ float value<__half>(unsigned short v) { return __half2float(__ushort_as_half(v)); }
template <> __device__ __forceinline__ float value<__nv_bfloat16>(unsigned short v) { return __uint_as_float((unsigned)v << 16); }

// Where output pixel q reads X: the value of (channel, tap) is at base + channel * hw_in + r * w_in + s, inside the image
// for taps whose (iy + r, ix + s) is.  (Not PATCH: one tap.)
template <bool PATCH>
struct Window {
    int img, p, iy, ix;
    size_t base;
    __device__ __forceinline__ Window(const TcLayer& y, int q)
    {
        img = div_of(q, y.hw);
        p = q - img * y.hw.d;
        const int oy = PATCH ? div_of(p, y.ow) : 0;
        iy = PATCH ? oy * y.stride - y.pad : 0;
        ix = PATCH ? (p - oy * y.ow.d) * y.stride - y.pad : p;
        base = (size_t)img * y.cin * y.hw_in;
    }
    __device__ __forceinline__ bool inside(const TcLayer& y, int r, int s) const
    {
        return !PATCH || ((unsigned)(iy + r) < (unsigned)y.h_in && (unsigned)(ix + s) < (unsigned)y.w_in);
    }
    __device__ __forceinline__ size_t at(const TcLayer& y, int c, int r, int s) const
    {
        return base + (size_t)c * y.hw_in + (PATCH ? (iy + r) * y.w_in + ix + s : ix);
    }
};

// The block's items once more, for pixels with an infinite or NaN input.  The expanded weights multiply such a value with the
// zeros of dropped blocks, too, and its parts do not add up to it: the whole tile is NaN there (which is how the
// epilogue notices).  Here the pixel's outputs are computed from the storage format, which touches kept blocks alone,
// and stored over what the epilogue stored.  At the end of the block, where no bounded wait of another role can run
// out meanwhile.  Slow, one pixel per warp at a time, and of use only to outputs that are then mostly not finite.
template <typename XT, bool PATCH, bool GENERAL, int L>
__device__ __forceinline__ void recompute(const TcArgs<L>& a, unsigned layers, int quad, int half, int lane)
{
    using raw = typename Elem<XT>::raw;
    Cursor<L> cur(a);
#pragma unroll 1
    while (cur.step()) {
        const TcLayer& y = cur.of();
        if (!(layers >> (L > 1 ? cur.layer : 0) & 1u) || cur.t.k16 == 0) continue;
        const raw* const x = static_cast<const raw*>(y.x);
        // channels of the item: all, or those of its part
        const int c0 = PATCH ? cur.t.kstart * 16 : 0, c1 = PATCH ? min(y.cin, c0 + div_of(cur.t.k16, y.taps) * 16) : y.cin;
#pragma unroll 1
        for (int row0 = quad * 32; row0 < y.ppt; row0 += kTcM) {
            const int row = row0 + lane, q0 = cur.pt() * y.ppt;
            bool bad = false;
            if (row < y.ppt && q0 + row < y.q) {
                const Window<PATCH> w(y, q0 + row);
#pragma unroll 1
                for (int r = 0; r < (PATCH ? y.kh : 1); ++r)
#pragma unroll 1
                    for (int s = 0; s < (PATCH ? y.kw : 1); ++s)
                        if (w.inside(y, r, s))
#pragma unroll 8
                            for (int c = c0; c < c1; ++c) bad |= special<XT>(__ldg(x + w.at(y, c, r, s)));
            }
            unsigned todo = __ballot_sync(0xffffffffu, bad);
            if (!todo) continue;
            const TcSparse sp = *y.sparse;
            const int nt = cur.nt(), tile = nt / sp.splits;
            const bool wide = sizeof(XT) == 4 || (GENERAL && y.y32);
#pragma unroll 1
            for (; todo; todo &= todo - 1) {
                const Window<PATCH> w(y, q0 + row0 + __ffs(todo) - 1);
#pragma unroll 1
                for (int j = half * 32 + lane; j < y.n; j += 64) {
                    const int c = GENERAL && y.chan ? __ldg(y.chan + nt * y.n + j) : tile * y.n + j;
                    if (c < 0 || c >= sp.cout) continue;
                    const int r = c / sp.g, in_block = c - r * sp.g;
                    float sum = 0.0f;
#pragma unroll 2
                    for (int k = __ldg(sp.row_ptr + r), end = __ldg(sp.row_ptr + r + 1); k < end; ++k) {
                        const int col = __ldg(sp.col_idx + k), ch = PATCH ? div_of(col, y.taps) : col, tap = PATCH ? col - ch * y.taps.d : 0;
                        const int tr = PATCH ? div_of(tap, y.kwd) : 0, ts = PATCH ? tap - tr * y.kwd.d : 0;
                        if (PATCH && (ch < c0 || ch >= c1 || !w.inside(y, tr, ts))) continue;
                        sum = fmaf(value<XT>(__ldg(x + w.at(y, ch, tr, ts))), value<XT>(__ldg(static_cast<const raw*>(sp.vals) + (size_t)k * sp.g + in_block)), sum);
                    }
                    const int o = sp.splits > 1 ? nt * y.n + j : c;       // (parts write rows of their own)
                    const size_t at = ((size_t)w.img * y.cout + o) * y.hw.d + w.p;
                    if (y.bias) sum += __ldg(y.bias + c);
                    if (GENERAL && y.res) sum += wide ? __ldg(static_cast<const float*>(y.res) + at) : (float)__ldg(static_cast<const XT*>(y.res) + at);
                    if (y.relu) sum = fmaxf(sum, 0.0f);
                    if (wide) static_cast<float*>(y.y)[at] = sum;
                    else put(static_cast<XT*>(y.y) + at, sum);
                }
            }
        }
    }
}

}  // namespace
}  // namespace alcs

#endif  // ALCS_TC_CUH_
