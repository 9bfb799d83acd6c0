// fused_common.cuh -- shared pieces of the fused bandwidth kernel
// (dpdr_allreduce): its launch arguments, the 16-byte and single-element
// memory units, and the running post-order fold every layout uses.
//
// The fused kernel computes y = v(r0) (.) v(r1) with the post-order
// bracketing of Sec. 1.1 (v(i) = v(child_1) (.) (v(child_0) (.) x_i),
// child_0 = i-1) for every element column and stores it to all p outputs.
// Every input element is read once and every output element written once:
// 2 p m element transfers, the floor for any reduction-to-all whose p inputs
// and p outputs live in device memory.  The tree's pipeline blocks
// (Algorithm 1) do not change the result, so the kernel tiles by columns.
// Layouts (one file each): column streaming (fused_stream.cu),
// shared-memory tile (fused_tile.cu), subtree split (fused_split.cu),
// bulk-copy pipeline (fused_bulk.cu), hierarchical tile (fused_tree.cu);
// fused.cu chooses and launches.
#pragma once

#include <algorithm>

#include "dpdr_internal.h"
#include "ops.cuh"

namespace dpdr {
namespace fused {

constexpr int kStreamThreads = 256;
constexpr int kStreamAhead = 8;  // ranks loaded ahead (tape read 8 at a time)
constexpr int kTileThreads = 256;
constexpr size_t kTileSmemTarget = 96 * 1024;
constexpr int kBulkConsumers = 256;                   // 8 warps
constexpr int kBulkThreads = kBulkConsumers + 32;     // + producer warp
constexpr int kBulkTile = kBulkConsumers * 16;        // bytes per rank row piece
constexpr int kBulkStages = 16;
constexpr int kTreeThreads = 512;                     // hierarchical tile: threads per CTA,
constexpr int kTreeUnitsNarrow = 8;                   // 16-byte column units per CTA:
constexpr int kTreeUnitsWide = 16;                    // the two tile widths
constexpr int kTreeCtasPerSm = 2;                     // resident (registers, shared memory)

struct FusedArgs {
    const char* const* x;   // [p] rank inputs
    char* const* y;         // [p] rank outputs
    const uint8_t* tape;    // [p rounded up to 8]
    const LevelNode* levels;
    const int* level_off;
    int nlevels;
    int p;
    int r0, r1;
    int dual;               // 1: y = v(r0) (.) v(r1); 0: one tree, y = v(p-1)
    int64_t nvec;           // 16-byte units, or (quad) units of four single elements
    int64_t nscalar;        // single elements after the vector units
    int64_t scalar_base;    // element index of the first single element
    int lg_wu;              // tile: log2 of vector units per row
    int quad;               // rows are not all 16-byte aligned: QuadUnit instead of VecUnit
    int64_t vec_tiles;      // tile: number of vector tiles
    // split layout
    const int2* seg;        // [nseg] (first rank, root rank) of each subtree
    const int2* items;      // [nitems] top fold: (source, tape byte | kind << 8)
    int nitems;
    char* part;             // [nseg] rows of subtree values
    int64_t part_stride;    // bytes per row
    int group;              // ranks stored by one CTA row of the finish kernel
    // bulk layout
    int64_t bulk_tiles;     // full tiles of kBulkTile bytes
    int bulk_bar_off;       // byte offset of the mbarriers in shared memory
    uint32_t* err;          // plan error record (an expired pipeline wait)
    int64_t wait_ns;
    // hierarchical tile layout
    const int2* tree_seg;   // [tree_nseg] subtree intervals, then nodes above the cut
    const int4* tree_lev;   // levels above the cut: (node, child_0, child_1) entries
    const int* tree_levoff; // [tree_nlev + 1]
    int tree_nseg, tree_nlev, tree_r0, tree_r1, tree_s, tree_slots;
    int64_t tree_tiles;     // CTAs of tree_width vector units
    int tree_width;         // kTreeUnitsNarrow or kTreeUnitsWide
    int overlap;            // launch: set up while the kernel before drains
    int far;                // inputs many times L2: FarUnit
};

template <class Op>
struct VecUnit {
    using T = uint4;
    __device__ __forceinline__ static T ld(const char* row, int64_t u)
    {
        return ld_stream(row + u * 16);
    }
    // Past L1, in the paired streaming and split layouts: p = 104, m = 2^18
    // float32 38.6 and 37.6 us, p = 1152 int32, m = 2^16 107.4 and 105.6,
    // m = 2^20 1403 and 1394, p = 4094, m = 2^17 698 and 678, never slower.
    // In the others it is not clear: plain streaming p = 100, m = 2^20 135.7
    // and 134.2 but p = 62, m = 1862468 147.8 and 148.3, hierarchical tile
    // p = 1152, m = 8192 21.7 and 21.4 but p = 576, m = 8192 12.9 and 13.0.
    __device__ __forceinline__ static T ld_wave(const char* row, int64_t u)
    {
        return ld_stream_past_l1(row + u * 16);
    }
    __device__ __forceinline__ static void st(char* row, int64_t u, const T& v)
    {
        st_stream(row + u * 16, v);
    }
    __device__ __forceinline__ static T op(const T& a, const T& b) { return Op::vec(a, b); }
    // data read again soon (subtree values, top-of-tree inputs): keep in L2
    __device__ __forceinline__ static T ld_keep(const char* row, int64_t u)
    {
        return ld_l2(row + u * 16);
    }
    __device__ __forceinline__ static void st_keep(char* row, int64_t u, const T& v)
    {
        st_l2(row + u * 16, v);
    }
};

// 16-byte units of inputs that are many times L2 (a.far): loads cached in L2
// only, at normal priority.
template <class Op>
struct FarUnit : VecUnit<Op> {
    __device__ __forceinline__ static uint4 ld(const char* row, int64_t u) { return ld_l2(row + u * 16); }
    __device__ __forceinline__ static uint4 ld_wave(const char* row, int64_t u) { return ld(row, u); }
};

// Four 4-byte elements of rows that are only 4-byte aligned: columns c, c + G,
// c + 2G and c + 3G of a group of 4G, so that G neighbouring units move 4G
// contiguous elements, in four accesses of 4G contiguous bytes.  G is the
// units that run side by side on one row: a warp's 32 in the streaming and
// split layouts, the tile's width in the others.  One element per thread and
// row left a quarter of the bytes in flight: p = 11, m = 6264977 int32 in
// 136 us, 87 with these units (83 with aligned rows); p = 62, m = 1862471
// 206 and 157 (153); p = 1152, m = 65537 163 and 115 (108).
template <class Op, int G>
struct QuadUnit {
    using T = uint4;
    static constexpr int kStep = 4 * G;  // bytes from one element to the next
    __device__ __forceinline__ static int64_t at(int64_t u)
    {
        return (u / G * (4 * G) + u % G) * 4;
    }
    __device__ __forceinline__ static uint32_t ld1(const char* p)
    {
        return __ldcs(reinterpret_cast<const unsigned int*>(p));
    }
    __device__ __forceinline__ static void st1(char* p, uint32_t v)
    {
        __stcs(reinterpret_cast<unsigned int*>(p), v);
    }
    __device__ __forceinline__ static T ld(const char* row, int64_t u)
    {
        const char* p = row + at(u);
        return make_uint4(ld1(p), ld1(p + kStep), ld1(p + 2 * kStep), ld1(p + 3 * kStep));
    }
    __device__ __forceinline__ static T ld_wave(const char* row, int64_t u) { return ld(row, u); }
    __device__ __forceinline__ static void st(char* row, int64_t u, const T& v)
    {
        char* p = row + at(u);
        st1(p, v.x);
        st1(p + kStep, v.y);
        st1(p + 2 * kStep, v.z);
        st1(p + 3 * kStep, v.w);
    }
    __device__ __forceinline__ static T op(const T& a, const T& b) { return Op::vec(a, b); }
    __device__ __forceinline__ static T ld_keep(const char* row, int64_t u)
    {
        const char* p = row + at(u);
        return make_uint4(ld_l2_u32(p), ld_l2_u32(p + kStep), ld_l2_u32(p + 2 * kStep),
                          ld_l2_u32(p + 3 * kStep));
    }
    __device__ __forceinline__ static void st_keep(char* row, int64_t u, const T& v)
    {
        char* p = row + at(u);
        st_l2_u32(p, v.x);
        st_l2_u32(p + kStep, v.y);
        st_l2_u32(p + 2 * kStep, v.z);
        st_l2_u32(p + 3 * kStep, v.w);
    }
};

// The wide unit of a launch: 16-byte units, or on unaligned rows of 4-byte
// elements (a.quad) four of them; f is called with a value of the unit type.
// with_stream_unit, of the streaming and split layouts, knows FarUnit too.
template <class Op, int G, class F>
inline int with_unit(const FusedArgs& a, F f)
{
    if constexpr (Op::kEpv == 4) {
        if (a.quad) return f(QuadUnit<Op, G>());
    }
    return f(VecUnit<Op>());
}
template <class Op, int G, class F>
inline int with_stream_unit(const FusedArgs& a, F f)
{
    return a.far ? f(FarUnit<Op>()) : with_unit<Op, G>(a, f);
}
constexpr int kQuadStream = 32;  // G of the streaming and split layouts
constexpr int kQuadTile = 8;     // of the shared-memory tile (as many units or more to a row)
constexpr int kQuadAttr = 7;  // offset of the unaligned kernels in Plan::smem_attr
constexpr int kFarAttr = 14;  // and of those for inputs many times L2

template <class Op>
struct OneUnit {
    using T = Elem<Op>;
    __device__ __forceinline__ static T ld(const char* row, int64_t e)
    {
        return ld_one_stream<Op>(row + e * Op::kEsize);
    }
    __device__ __forceinline__ static T ld_wave(const char* row, int64_t e) { return ld(row, e); }
    __device__ __forceinline__ static void st(char* row, int64_t e, const T& v)
    {
        st_one_stream<Op>(row + e * Op::kEsize, v);
    }
    __device__ __forceinline__ static T op(const T& a, const T& b) { return comb<Op>(a, b); }
    __device__ __forceinline__ static T ld_keep(const char* row, int64_t e)
    {
        return ld_one_l2<Op>(row + e * Op::kEsize);
    }
    __device__ __forceinline__ static void st_keep(char* row, int64_t e, const T& v)
    {
        st_one_l2<Op>(row + e * Op::kEsize, v);
    }
};

__device__ __forceinline__ const char* rank_ptr(const char* const* t, int i)
{
    return reinterpret_cast<const char*>(__ldg(reinterpret_cast<const unsigned long long*>(t) + i));
}
__device__ __forceinline__ char* rank_ptr_w(char* const* t, int i)
{
    return reinterpret_cast<char*>(__ldg(reinterpret_cast<const unsigned long long*>(t) + i));
}

// ---------------------------------------------------------------- streaming
// One step of the running post-order fold: v is rank i's own value x_i (or,
// in the split layout, a whole subtree's value with no children left); acc
// holds the value of rank i-1, which is child_0 whenever i has a child; a
// child_1 value waits in slot[depth+1]; a node that is a child_1 (or the
// lower root) parks its value in slot[depth].
template <class U>
__device__ __forceinline__ void fold_step(unsigned t, typename U::T v, typename U::T& acc,
                                          typename U::T* slot, int stride)
{
    const unsigned c = t & 3u, d = (t >> 3) & 31u;
    if (c >= 1) v = U::op(acc, v);                     // v(c0) (.) x_i
    if (c == 2) v = U::op(slot[(d + 1) * stride], v);  // v(c1) (.) (..)
    if (t & kTapeKeep) slot[d * stride] = v;
    acc = v;
}

template <class U>
__device__ __forceinline__ void stream_column(const FusedArgs& a, int64_t u,
                                              typename U::T* slot, int stride)
{
    using T = typename U::T;
    const int p = a.p;
    T acc{};  // set by rank 0, a leaf
    // one batch of kStreamAhead loads in flight per thread; the other warps
    // of the four CTAs per SM cover the latency between batches
    for (int i0 = 0; i0 < p; i0 += kStreamAhead) {
        T cur[kStreamAhead];
#pragma unroll
        for (int k = 0; k < kStreamAhead; k++)
            if (i0 + k < p) cur[k] = U::ld(rank_ptr(a.x, i0 + k), u);
        const unsigned long long tp =
            __ldg(reinterpret_cast<const unsigned long long*>(a.tape + i0));
#pragma unroll
        for (int k = 0; k < kStreamAhead; k++)
            if (i0 + k < p) fold_step<U>(unsigned(tp >> (8 * k)) & 0xffu, cur[k], acc, slot, stride);
    }
    const T y = a.dual ? U::op(slot[0], acc) : acc;  // v(r0) (.) v(r1), or v(root)
#pragma unroll 4
    for (int i = 0; i < p; i++) U::st(rank_ptr_w(a.y, i), u, y);
}

// The depth slots of thread t sit in 16-byte cells t, t + n, t + 2n, ... of
// a [depth][n] array of uint4 (n threads).  A thread folding single elements
// keeps its slots in the same cells (an element is at most 16 bytes), so its
// slots never overlap another thread's, whatever unit each thread folds.
template <class Op>
__device__ __forceinline__ Elem<Op>* one_slots(uint4* cells, int t)
{
    return reinterpret_cast<Elem<Op>*>(cells + t);
}
template <class Op>
__device__ __forceinline__ int one_slot_stride(int n)
{
    return n * int(sizeof(uint4) / sizeof(Elem<Op>));
}

// launchers, one per layout (dispatch on the plan's element type)
// Raise kernel fn's dynamic shared memory limit on the current device to at
// least `bytes`, never lowering it: the attribute belongs to the function and
// is shared by every plan, so a plan that needs less must not take it away
// from one that needs more.  *granted is the plan's cache of what it already
// has (launches that fit skip the call).
int grant_smem(const void* fn, size_t bytes, int* granted, const char* what);

int launch_stream(Plan* P, FusedArgs a, cudaStream_t s);
int launch_tile(Plan* P, FusedArgs a, cudaStream_t s);
int launch_split(Plan* P, FusedArgs a, cudaStream_t s);
int launch_bulk(Plan* P, FusedArgs a, cudaStream_t s);
int launch_tree(Plan* P, FusedArgs a, cudaStream_t s);
int tile_lg_wu(const Plan* P);

template <template <class> class L>
int dispatch(Plan* P, FusedArgs a, cudaStream_t s)
{
    switch (P->dtype) {
    case DPDR_INT32: return L<SumI32>::run(P, a, s);
    case DPDR_FLOAT32: return L<SumF32>::run(P, a, s);
    case DPDR_MAT2X2_F32: return L<MatF32>::run(P, a, s);
    default: return L<MatU32>::run(P, a, s);
    }
}

// The fused kernels are launched with programmatic stream serialisation: a
// kernel is set up while the one before it in the stream drains, and its
// threads wait here, before they touch any memory, until that one is complete
// and its writes are visible.  So calls are ordered as ever, and so is what
// follows in the stream; what goes is the gap between two kernels (back to
// back, p = 7, m = 1000 int32 in 4.1 and 2.7 us; p = 36, m = 2^16 2x2 matrices
// 16.4 and 14.5; p = 1152 int32, m = 1024 10.3 and 8.9, and m = 2^16, two
// kernels of the split layout, 113 and 107).
// No kernel asks for the next one to start early, so a CTA never
// waits here in a place that a running kernel needs.  Calls on host memory
// are launched the plain way: they gain nothing, and back to back their reads
// and writes share the link less evenly (p = 36, m = 2^16 2x2 matrices 242
// against 230 us).
__device__ __forceinline__ void wait_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

inline int launch_kernel(void (*kernel)(FusedArgs), dim3 grid, int threads, size_t smem, cudaStream_t s,
                         const FusedArgs& a)
{
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(unsigned(threads));
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = &attr;
    cfg.numAttrs = a.overlap ? 1 : 0;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, a);
    return e == cudaSuccess ? DPDR_OK : cuda_fail(e, "fused kernel launch");
}

}  // namespace fused
}  // namespace dpdr
