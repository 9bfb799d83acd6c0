// schedule_cells.cuh -- device pieces shared by the schedule kernels that
// gather the virtual ranks into subtree cells: flagged words between cells
// for short blocks (schedule_words.cu), counters for large ones
// (schedule_walk.cu).
//
// A cell is a connected piece of a post-order tree.  One warp runs a cell
// for one column slice of every block, and every lane owns the same columns
// of all the cell's ranks, so an exchange between two ranks of a cell is a
// value handed on inside the lane; only the exchanges along cut edges and
// between the dual roots cross warps.
#pragma once

#include "fused_common.cuh"
#include "schedule_common.cuh"

namespace dpdr {
namespace cells {

constexpr int kCtr = 32;                 // words from one counter to the next (an L2 line)
constexpr unsigned kAll = 0xffffffffu;
// Counters and flags start again from 0 at this base.  A call uses at most
// 2^30 + 64 values, so they never wrap.
constexpr uint32_t kRestart = 1u << 29;

typedef unsigned long long u64;

__device__ __forceinline__ void cp_async16(void* smem, const void* gmem)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                     static_cast<uint32_t>(__cvta_generic_to_shared(smem))),
                 "l"(gmem)
                 : "memory");
}
__device__ __forceinline__ void cp_async4(void* smem, const void* gmem)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(
                     static_cast<uint32_t>(__cvta_generic_to_shared(smem))),
                 "l"(gmem)
                 : "memory");
}
__device__ __forceinline__ void cp_async_wait_all()
{
    asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;" ::: "memory");
}

__device__ __forceinline__ void ld_words2(const u64* p, u64& a, u64& b)
{
    asm volatile("ld.relaxed.gpu.global.v2.b64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "l"(p) : "memory");
}
__device__ __forceinline__ u64 ld_word(const u64* p)
{
    u64 a;
    asm volatile("ld.relaxed.gpu.global.b64 %0, [%1];" : "=l"(a) : "l"(p) : "memory");
    return a;
}
__device__ __forceinline__ void st_words2(u64* p, u64 a, u64 b)
{
    asm volatile("st.relaxed.gpu.global.v2.b64 [%0], {%1, %2};" ::"l"(p), "l"(a), "l"(b) : "memory");
}
__device__ __forceinline__ void st_word(u64* p, u64 a)
{
    asm volatile("st.relaxed.gpu.global.b64 [%0], %1;" ::"l"(p), "l"(a) : "memory");
}
__device__ __forceinline__ u64 flagged(uint32_t v, uint32_t flag) { return (u64(flag) << 32) | v; }
__device__ __forceinline__ bool fresh(u64 w, uint32_t flag) { return uint32_t(w >> 32) == flag; }

// One unit of a row: 16 bytes, or one element where rows are only 4-byte
// aligned and for the last elements of a row.  A unit travels between warps
// as kBytes / 4 flagged words.
template <class Op, bool kVec>
struct Unit;

template <class Op>
struct Unit<Op, true> {
    using T = uint4;
    static constexpr int kElems = Op::kEpv;
    static constexpr int kBytes = 16;
    __device__ __forceinline__ static T op(const T& a, const T& b) { return Op::vec(a, b); }
    __device__ __forceinline__ static void copy(uint4* slot, const char* p) { cp_async16(slot, p); }
    __device__ __forceinline__ static T ld(const char* p) { return ld_l2(p); }
    __device__ __forceinline__ static void st_keep(char* p, const T& v) { st_l2(p, v); }
    __device__ __forceinline__ static void st(char* p, const T& v) { st_stream(p, v); }
    // the unit's words, whether all carry the flag
    __device__ __forceinline__ static bool recv(const u64* p, uint32_t flag, T& v)
    {
        u64 a, b, c, d;
        ld_words2(p, a, b);
        ld_words2(p + 2, c, d);
        v = make_uint4(uint32_t(a), uint32_t(b), uint32_t(c), uint32_t(d));
        return fresh(a, flag) && fresh(b, flag) && fresh(c, flag) && fresh(d, flag);
    }
    __device__ __forceinline__ static void send(u64* p, uint32_t flag, const T& v)
    {
        st_words2(p, flagged(v.x, flag), flagged(v.y, flag));
        st_words2(p + 2, flagged(v.z, flag), flagged(v.w, flag));
    }
};

template <class Op>
struct Unit<Op, false> {
    using T = Elem<Op>;
    static constexpr int kElems = 1;
    static constexpr int kBytes = Op::kEsize;
    __device__ __forceinline__ static T op(const T& a, const T& b) { return comb<Op>(a, b); }
    __device__ __forceinline__ static void copy(uint4* slot, const char* p)
    {
        uint32_t* dst = reinterpret_cast<uint32_t*>(slot);
#pragma unroll
        for (int w = 0; w < T::kWords; w++) cp_async4(dst + w, p + 4 * w);
    }
    __device__ __forceinline__ static T ld(const char* p) { return ld_one_l2<Op>(p); }
    __device__ __forceinline__ static void st_keep(char* p, const T& v) { st_one_l2<Op>(p, v); }
    __device__ __forceinline__ static void st(char* p, const T& v) { st_one_stream<Op>(p, v); }
    __device__ __forceinline__ static bool recv(const u64* p, uint32_t flag, T& v)
    {
        bool ok = true;
#pragma unroll
        for (int w = 0; w < T::kWords; w++) {
            const u64 word = ld_word(p + w);
            v.w[w] = uint32_t(word);
            ok = ok && fresh(word, flag);
        }
        return ok;
    }
    __device__ __forceinline__ static void send(u64* p, uint32_t flag, const T& v)
    {
#pragma unroll
        for (int w = 0; w < T::kWords; w++) st_word(p + w, flagged(v.w[w], flag));
    }
};

// Column slices of 32 units, numbered through all blocks (per_block to a
// block): in step t warp g of a cell runs slice t nslices + g, so the blocks
// pass in their order, and every slice through the same warp of each cell.
// The schedule's rounds are the warp's steps: an exchange that Algorithm 1
// puts d rounds after another comes d steps after it.
// With 16-byte units the bounds of the blocks are rounded up to whole units
// (a block is then up to 3 elements longer or shorter than the partition
// says); the row's last elements that fill no unit are one more slice of one
// block, run element by element (tail).
struct Columns {
    int64_t m, q, rem;   // elements, block partition
    int b, nslices, per_block, steps;
    int tail;            // 1: there is a tail slice (the last one)
};

// The lane's unit of a slice: byte offset in every row, whether it is there.
template <class I>
struct SpotOf {
    I off;
    bool on;
};

// Block and slice of a step, moved on from one step to the next; past the
// last block in the last step of some warps (an empty extent).
struct Pos {
    int j, g;
    __host__ __device__ __forceinline__ Pos(const Columns& c, int slice)
        : j(slice / c.per_block), g(slice % c.per_block) {}
    __host__ __device__ __forceinline__ void advance(const Columns& c)
    {
        for (g += c.nslices; g >= c.per_block; g -= c.per_block) j++;
    }
};

// A slice's units: the first, and how many (up to 32).  I: an integer that
// holds every element's number.
template <class I>
struct Extent {
    I u;
    int n;
};

template <class Op, bool kVec, class I>
__host__ __device__ __forceinline__ Extent<I> extent(const Columns& c, const Pos& at, bool tail)
{
    constexpr int E = Unit<Op, kVec>::kElems;
    const I m = I(c.m);
    I u = sched::block_start(I(c.q), I(c.rem), at.j), e = sched::block_start(I(c.q), I(c.rem), at.j + 1);
    if (tail) {
        u = m - m % Op::kEpv;
        e = m;
    } else {
        if (E > 1) {
            u = (u + E - 1) / E;
            e = e == m ? e / E : (e + E - 1) / E;
        }
        u += I(at.g) * 32;
    }
    if (u >= e || (!tail && at.j >= c.b)) return Extent<I>{u, 0};
    return Extent<I>{u, e - u < 32 ? int(e - u) : 32};
}
// The first slice of a warp from `at` on that holds units, which `at` moves on
// to: blocks differ by a unit, so a slice past the end of one block may have
// units in the next.  False when there is none.
template <class Op, bool kVec, class I>
__host__ __device__ __forceinline__ bool next_slice(const Columns& c, Pos& at, bool tail, Extent<I>& x)
{
    for (; at.j < c.b; at.advance(c)) {
        x = extent<Op, kVec, I>(c, at, tail);
        if (x.n) return true;
    }
    return false;
}

// Records an expired wait (the first one of the call wins) and aborts the
// call: every other wait sees the abort word equal to its epoch.
// ctl: [0] epoch of this call, [1] CTAs started, [2] aborted epoch, [3] base
// of the call's counters and flags, [4] CTAs finished (a call that clears).
static __device__ __noinline__ void wait_expired(uint32_t* err, uint32_t* ctl, uint32_t epoch,
                                                 int rank, int j, int step)
{
    if (atomicCAS(err, 0u, uint32_t(DPDR_ERR_TIMEOUT)) == 0u) {
        err[1] = uint32_t(rank);
        err[2] = uint32_t(j);
        err[3] = uint32_t(step);
    }
    __threadfence();
    atomicExch(ctl + 2, epoch);
}

// Whether a wait that began at t0 must end: 1 the call was aborted, 2 its
// time is up, else 0; the same on every lane.
__device__ __forceinline__ int give_up(const uint32_t* ctl, uint32_t epoch, uint64_t t0, int64_t wait_ns)
{
    int r = 0;
    if ((threadIdx.x & 31) == 0) {
        if (sched::ld_relaxed(ctl + 2) == epoch) r = 1;
        else if (sched::now_ns() - t0 > uint64_t(wait_ns)) r = 2;
    }
    return __shfl_sync(kAll, r, 0);
}

// Waits until the counter of every lane with `mine` reaches its target; rank
// and step name the lane's exchange in an error record.  `seen`: the value
// that the lane read last from this counter (counters only grow, so one that
// was already far enough is not read again).  `never`: a lane whose partner
// is silent.  False when a wait of the call expired.
__device__ __forceinline__ bool wait_counters(uint32_t* ctl, uint32_t* err, int64_t wait_ns,
                                              uint32_t epoch, const uint32_t* c, uint32_t target,
                                              uint32_t& seen, bool mine, bool never, int rank, int j,
                                              int step)
{
    const int lane = int(threadIdx.x) & 31;
    bool pend = never || (mine && int32_t(seen - target) < 0);
    if (pend && !never) {
        seen = sched::ld_acquire(c);
        pend = int32_t(seen - target) < 0;
    }
    unsigned who = __ballot_sync(kAll, pend);
    if (who) {
        const uint64_t t0 = sched::now_ns();
        unsigned polls = 0, sleep = 0;
        while (true) {
            if (pend && !never) {
                seen = sched::ld_acquire(c);
                pend = int32_t(seen - target) < 0;
            }
            who = __ballot_sync(kAll, pend);
            if (!who) break;
            if ((polls & 15) == 15) {
                const int stop = give_up(ctl, epoch, t0, wait_ns);
                if (stop == 2 && lane == __ffs(who) - 1) wait_expired(err, ctl, epoch, rank, j, step);
                if (stop) return false;
            }
            if (++polls > 32) {
                sleep = sleep ? (sleep < 256 ? sleep * 2 : 256) : 32;
                __nanosleep(sleep);
            }
        }
    }
    __syncwarp();
    return true;
}

// A call's numbers, and (thread 0) this CTA's place among those that have
// read them.
struct Call {
    uint32_t epoch, base, place;
};

// At a kernel's start: thread 0 asks for the numbers.
__device__ __forceinline__ Call ask_call(const uint32_t* ctl)
{
    Call c{0, 0, 0};
    if (threadIdx.x == 0) {
        c.epoch = *reinterpret_cast<volatile const uint32_t*>(ctl);
        c.base = *reinterpret_cast<volatile const uint32_t*>(ctl + 3);
    }
    return c;
}

// Called by every thread some loads later: thread 0 hands the numbers to the
// CTA and, having them, counts it in.
__device__ __forceinline__ void start_call(uint32_t* ctl, Call& c)
{
    __shared__ volatile uint32_t numbers[2];
    if (threadIdx.x == 0) {
        numbers[0] = c.epoch;
        numbers[1] = c.base;
        c.place = atomicAdd(ctl + 1, 1u);
    }
    __syncthreads();
    c.epoch = numbers[0];
    c.base = numbers[1];
}

// Called by every thread at a kernel's end: the CTA that was the last to read
// the call's numbers moves the plan to the next call's, without waiting for
// the others to finish (captured calls with a count of finished CTAs at the
// end and without: p = 288, m = 250 int32 10.9 and 10.7 us; p = 36, m = 80000
// 15.8 and 14.8; p = 7, m = 1000, b = 4 7.5 and 6.8).  Long before the numbers
// could wrap a call clears the counters and flags (words from `scratch` on),
// and there the last CTA to finish does it.
__device__ __forceinline__ void finish_call(uint32_t* ctl, const Call& c, uint32_t used, uint32_t* scratch,
                                            int64_t words)
{
    const uint32_t next = c.base + used;
    bool mine = threadIdx.x == 0 && c.place == gridDim.x - 1;
    if (next >= kRestart) {
        __shared__ int last;
        __syncthreads();
        if (threadIdx.x == 0) {
            __threadfence();
            last = atomicAdd(ctl + 4, 1u) == gridDim.x - 1;
        }
        __syncthreads();
        if (!last) return;
        for (int64_t i = threadIdx.x; i < words; i += blockDim.x) scratch[i] = 0;
        mine = threadIdx.x == 0;
        if (mine) ctl[4] = 0;
    }
    if (mine) {
        ctl[1] = 0;
        *reinterpret_cast<volatile uint32_t*>(ctl + 3) = next >= kRestart ? 0 : next;
        *reinterpret_cast<volatile uint32_t*>(ctl) = c.epoch + 1 == 0 ? 1 : c.epoch + 1;
    }
}

}  // namespace cells
}  // namespace dpdr
