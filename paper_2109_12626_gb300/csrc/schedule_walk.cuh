// schedule_walk.cuh -- the schedule-faithful kernels on large pipeline
// blocks, the virtual ranks gathered into subtree cells of at most
// kWalkRanks ranks (dpdr_allreduce_schedule and dpdr_allreduce_reduce_bcast
// where every schedule option is automatic; schedule_cells.cuh).
//
// The schedule is Algorithm 1's: in round j every rank takes its children's
// partial blocks j, forms Y[j] = t1 (.) (t0 (.) x_i) and hands it to its
// parent (the dual roots exchange theirs); a rank at depth d receives final
// block j - d.  A cell whose root is at depth D does this for all its ranks at
// once: in step t the partial block t goes up through them, and then the final
// block t - D goes down to all of them.  So a rank l levels below the cell's
// root has a final block up to l rounds before the schedule asks for it, and a
// child cell, which takes it from there l + 1 rounds later, seldom waits.
//
// What bounds it: a step of a warp (32 units of all its ranks, 8 KB in and
// 8 KB out for 16 ranks) is a chain of about 8 us -- the children's counters
// and partial blocks, the fold, a release fence, the parent's final block, the
// stores, another fence -- and device memory.  24 warps per SM, each with its
// next step's inputs on their way into shared memory (cp.async) while it
// waits, cover most of the chain; the warps of cells with child cells have the
// longest one.  With a warp group per rank (schedule.cu) every block crosses
// L2 once per tree edge and direction, each time behind such a chain; here one
// edge in fifteen does.  Measured (captured calls, inputs larger than L2,
// before and after; copying the same rows in the same pieces takes 102, 385,
// 340 and 322 us for the first, second, fourth and sixth): p = 1152 int32,
// m = 2^16 in 246 and 126 us, m = 2^18 673 and 476; p = 288, m = 212500 244
// and 113; p = 32 float32, m = 2^23, b = 16 570 and 365; p = 36 2x2 matrices,
// m = 2^20 352 and 215; reduce, then broadcast at p = 288, m = 875000 in
// 16000-element blocks 909 and 425.
// Of that: final blocks to all ranks of a cell at once, not level by level,
// p = 1152 151 to 136 us and p = 32 395 to 361; the children's values through
// free shared-memory slots (stage) 133 to 130 and, reduced then broadcast, 457
// to 424; one fence for both counters of a step 130 to 126 and, m = 2^18, 496
// to 476; the parent's final block read ahead of the fold, m = 2^18, 521 to 507.
// Not kept: 4 units per lane (fewer, longer steps; the registers for them
// spilled, and a spilled value comes back from L2 after every acquire); a
// warp for each direction (the two loops together no longer fitted the
// instruction cache: 1.5 to 2.5 times as long); inputs in registers instead
// of shared memory; bulk copies of the inputs, one lane per row (8 % slower at
// p = 32), and of the outputs (their buffers cost a quarter of the warps); the
// counter ahead of the rows that no other cell reads (a second pass over the
// rows, 4 % slower).
//
// Exchanges between cells: the cell root's partial block goes to its y row
// (a dual root's to an exchange slot) and a release store of the cell's up
// counter publishes it; a final block is read from the parent rank's y row
// once the parent cell's done counter says that it finished the step that put
// it there.  Counters never repeat (finish_call), so a call is one kernel and
// a captured graph replays.
//
// Order and reuse.  A cell waits in step t for its children's partial blocks
// t, which they publish before they wait for any final block of their own step
// t; for the dual root's partial t, published before the wait; and for a step
// before t of its parent's cell, whose partial blocks it published in earlier
// steps (a partial block is published together with the step's end only where
// the parent's block is there already): with all CTAs resident (cooperative
// launch) nothing deadlocks.  The final block overwrites the partial block in
// the cell root's y row only after the parent, which holds it, has read that,
// and an exchange slot of parity t & 1 is written again in step t + 2, after
// the dual's partial t + 1 has shown that it finished step t.  In place
// (y_i == x_i) every lane reads x_i of a block before it writes any y_i of it.
// Every wait is bounded in time; an expired wait records {rank, round, step},
// marks the call's epoch aborted and every other wait of the call gives up.
#pragma once

#include "schedule_cells.cuh"

namespace dpdr {
namespace walk {

using namespace cells;
using Spot = SpotOf<int64_t>;

constexpr int kWarps = 4;     // per CTA
constexpr int kCtas = 6;      // per SM: 80 registers, 24 warps
constexpr int kNodes = 2;     // nodes that take their children's values at once
constexpr int kRanks = kWalkRanks;
constexpr int kLevels = kWalkLevels;
constexpr int kExt = kRanks / 2;
constexpr int kPast = 32;     // above the deepest rank's depth (schedule_walk_prepare)

// Bytes of staged inputs per CTA for cells of at most `ranks` ranks.
constexpr size_t smem_for(int ranks) { return size_t(kWarps) * size_t(ranks) * 32 * sizeof(uint4); }

struct WalkArgs {
    const char* const* x;
    char* const* y;
    const CellDesc* cells;
    uint32_t* ctl;
    uint32_t* up;        // [cells][slices] lines: partial blocks published
    uint32_t* done;      // the same: steps finished
    int64_t ctr_words;   // of both
    uint32_t* err;
    char* ring;          // [2 sides][2][slices] exchange slots of 512 bytes
    Columns col;
    int64_t wait_ns;
    int ncells, root0, root1;  // cells of the roots (root0 -1: one tree)
    int ranks;           // of the largest cell
    int used;            // counter values the call uses
    int skip_rank;
};

struct WarpInfo {        // one per warp, in shared memory
    const char* x[kRanks];      // input rows, in post-order
    char* y[kRanks];            // output rows, by level (the cell's root first)
    const char* ext[2 * kExt];  // y rows of the child cells' roots
    const char* par;            // y row of the parent rank
    uint8_t tape[kRanks];       // CellDesc::tape
    int ext_k[kExt];
    int ext_cell[2 * kExt];
    int ext_node[kExt];         // the nodes' ranks
    int n, next, depth, root, par_cell;
    int lag;                    // levels from the parent cell's root
    int staged;                 // nodes whose children's values fit the slots
    unsigned reread;            // bit t: row y[t] is read again
    int cell, g;                // this warp's cell and column slice
    uint32_t epoch, base;       // of the call: abort mark, counter base
    int dual;                   // the cell holds a dual root
    int mute;                   // fault injection: the cell's root never publishes
    int stuck, stuck_step;      // fault injection: parent in this cell of the silent rank
                                // (-1: none), and which child that is
    // where the units of the last steps lie: first unit, how many
    int64_t past_u[kPast];
    int past_n[kPast];
};

// One warp's run of its cell for its column slices.
template <class Op, bool kVec, bool kRB>
struct Runner {
    using U = Unit<Op, kVec>;
    using T = typename U::T;
    const WalkArgs& a;
    WarpInfo* s;
    uint4* slot;         // this lane's cells: the unit of position k at k * 32
    int lane;
    bool tail;

    // Notes where step t's units lie (the same on every lane); the lane's unit
    // of a step noted before.
    __device__ __forceinline__ Spot note(const Pos& c, int t) const
    {
        const Extent<int64_t> x = extent<Op, kVec, int64_t>(a.col, c, tail);
        __syncwarp();
        if (lane == 0) {
            s->past_u[t & (kPast - 1)] = x.u;
            s->past_n[t & (kPast - 1)] = x.n;
        }
        __syncwarp();
        return Spot{(x.u + lane) * U::kBytes, lane < x.n};
    }
    __device__ __forceinline__ Spot noted(int t) const
    {
        return Spot{(s->past_u[t & (kPast - 1)] + lane) * U::kBytes, lane < s->past_n[t & (kPast - 1)]};
    }

    __device__ __forceinline__ uint32_t* ctr(uint32_t* t, int c) const
    {
        return t + (int64_t(c) * (a.col.nslices + a.col.tail) + s->g) * kCtr;
    }
    __device__ __forceinline__ bool wait(bool mine, const uint32_t* c, uint32_t target, uint32_t& seen,
                                         bool never, int rank, int j, int step) const
    {
        return wait_counters(a.ctl, a.err, a.wait_ns, s->epoch, c, target, seen, mine, never, rank, j, step);
    }
    // Whether the counter has reached its target: read once, no wait.
    __device__ __forceinline__ bool reached(const uint32_t* c, uint32_t target, uint32_t& seen) const
    {
        if (lane == 0 && int32_t(seen - target) < 0) seen = sched::ld_acquire(c);
        const bool ok = __shfl_sync(kAll, int(int32_t(seen - target) >= 0), 0) != 0;
        __syncwarp();
        return ok;
    }
    __device__ __forceinline__ void publish(uint32_t* t, uint32_t v) const
    {
        __syncwarp();
        if (lane == 0 && !s->mute) sched::st_release(ctr(t, s->cell), v);
    }
    __device__ __forceinline__ char* ring(int side, int t) const
    {
        return a.ring + ((int64_t(side) * 2 + (t & 1)) * (a.col.nslices + a.col.tail) + s->g) * 512 +
               lane * U::kBytes;
    }

    __device__ __forceinline__ T& at(int k) const { return *reinterpret_cast<T*>(slot + k * 32); }

    // Starts the copies of every rank's input into the lane's slots.
    __device__ __forceinline__ void fetch(const Spot& p) const
    {
        const int n = s->n;
#pragma unroll 2
        for (int k = 0; k < n; k++)
            if (p.on) U::copy(slot + k * 32, s->x[k] + p.off);
    }

    // The cell root's value of the units in the slots, the bottom nodes having
    // taken their children's values: the fold of the slots in post-order.
    // A child_1 inside the cell waits for its parent in its own slot.
    __device__ __forceinline__ T fold() const
    {
        T acc{};
        const int n = s->n;
#pragma unroll 1
        for (int k = 0; k < n; k++) {
            const unsigned t = s->tape[k];
            T v = at(k);
            if (t & 3u) {
                v = U::op(acc, v);
                if (t & 2u) v = U::op(at(int(t >> 3)), v);
            }
            acc = v;
            if (t & 4u) at(k) = v;
        }
        return acc;
    }

    // Steps child_0 and child_1 of step t (of block j), the inputs being on
    // their way into the slots: v becomes the cell's partial block.  Returns
    // false when a wait expired.
    __device__ __forceinline__ bool up(int t, int j, const Spot& p, uint32_t& seen, T& v) const
    {
        const int next = s->next;
        if (next || s->stuck >= 0) {
            const bool mine = lane < 2 * next, never = s->stuck >= 0 && lane == 31;
            if (!wait(mine, ctr(a.up, mine ? s->ext_cell[lane] : 0), s->base + uint32_t(t) + 1u, seen, never,
                      never ? s->stuck : mine ? s->ext_node[lane >> 1] : 0, j,
                      never ? s->stuck_step : lane & 1))
                return false;
        }
        // the first nodes' values by way of the slots that the cell's ranks
        // leave free, the others' through registers, kNodes at a time
        const int staged = kVec ? s->staged : 0, n = s->n;
#pragma unroll 2
        for (int h = 0; h < 2 * staged; h++)
            if (p.on) U::copy(slot + (n + h) * 32, s->ext[h] + p.off);
        bool landed = false;
#pragma unroll 1
        for (int q0 = staged; q0 < next; q0 += kNodes) {
            T e[2 * kNodes];
#pragma unroll
            for (int h = 0; h < 2 * kNodes; h++)
                if (q0 + h / 2 < next && p.on) e[h] = U::ld(s->ext[2 * q0 + h] + p.off);
            if (!landed) cp_async_wait_all();
            landed = true;
            // t1 (.) (t0 (.) x) in the node's slot
#pragma unroll
            for (int h = 0; h < kNodes; h++)
                if (q0 + h < next) {
                    const int k = s->ext_k[q0 + h];
                    at(k) = U::op(e[2 * h + 1], U::op(e[2 * h], at(k)));
                }
        }
        if (!landed) cp_async_wait_all();
#pragma unroll 1
        for (int q = 0; q < staged; q++) {
            const int k = s->ext_k[q];
            at(k) = U::op(at(n + 2 * q + 1), U::op(at(n + 2 * q), at(k)));
        }
        v = fold();
        return true;
    }

    // The partial block of step t handed up: to the cell root's row, or a dual
    // root's exchange slot, and published (now) or left to the step's end.
    // Before the next inputs are asked for: the release would wait for them
    // (p = 32, m = 2^23 float32, 415 and 405 us).
    __device__ __forceinline__ void hand_up(int t, const Spot& p, const T& v, bool now) const
    {
        if (p.on) U::st_keep(s->dual ? ring(s->cell == a.root0 ? 0 : 1, t) : s->y[0] + p.off, v);
        if (now) publish(a.up, s->base + uint32_t(t) + 1u);
    }

    // v: a final block's unit, into the rows y[t0 .. t1)
    __device__ __forceinline__ void put(const Spot& p, const T& v, int t0, int t1) const
    {
        if (!p.on) return;
#pragma unroll 2
        for (int t = t0; t < t1; t++) {
            char* const y = s->y[t] + p.off;
            if ((s->reread >> t) & 1u)
                U::st_keep(y, v);
            else
                U::st(y, v);
        }
    }

    // Reduce, then broadcast.  A block passes through a cell at once.
    __device__ __forceinline__ void reduce_bcast() const
    {
        const int steps = tail ? 1 : a.col.steps;
        const bool root = s->par_cell < 0;
        uint32_t up_seen = s->base, seen = s->base;  // read last from the children's, the parent's counter
        Pos c(a.col, tail ? 0 : s->g);
        Spot p = note(c, 0);
        fetch(p);
#pragma unroll 1
        for (int t = 0; t < steps; t++) {
            T v;
            if (!up(t, c.j, p, up_seen, v)) return;
            const Spot was = p;
            c.advance(a.col);
            hand_up(t, was, v, true);
            if (t + 1 < steps) {  // the next block's inputs
                p = note(c, t + 1);
                fetch(p);
            }
        }
        c = Pos(a.col, tail ? 0 : s->g);
#pragma unroll 1
        for (int t = 0; t < steps; t++, c.advance(a.col)) {
            p = note(c, t);
            if (!root && !wait(lane == 0, ctr(a.done, s->par_cell), s->base + uint32_t(t) + 1u,
                               seen, false, s->root, c.j, 3))
                return;
            T v{};
            if (p.on) v = U::ld((root ? s->y[0] : s->par) + p.off);  // a root holds the block
            put(p, v, root ? 1 : 0, s->n);
            if (s->next) publish(a.done, s->base + uint32_t(t) + 1u);
        }
    }

    // Algorithm 1, a step at a time.
    __device__ __forceinline__ void algorithm_1() const
    {
        const int steps = tail ? 1 : a.col.steps, D = s->depth;
        const bool root = s->par_cell < 0;
        // read last from the children's counters, the dual's or the parent's
        uint32_t up_seen = s->base, seen = s->base;
        Pos c(a.col, tail ? 0 : s->g);
        fetch(note(c, 0));
        const int last = steps - 1 + D;
#pragma unroll 1
        for (int t = 0; t <= last; t++) {
            const int f = t - D;  // the step whose block is final in this cell now
            // the parent's cell put it there in step t - lag: read ahead of the
            // fold where that is over
            const uint32_t final_at = s->base + uint32_t(t - s->lag) + 1u;
            T v{}, w{};
            bool held = false;
            if (f >= 0 && !root) {
                held = reached(ctr(a.done, s->par_cell), final_at, seen);
                if (held) {
                    const Spot p = noted(f);
                    if (p.on) w = U::ld(s->par + p.off);
                }
            }
            // one fence for both counters where nothing of this step waits
            const bool join = held && t < steps && s->next;
            if (t < steps) {
                const Spot p = noted(t);
                if (!up(t, c.j, p, up_seen, v)) return;
                c.advance(a.col);
                if (!root || s->dual) hand_up(t, p, v, !join);
                if (t + 1 < steps) fetch(note(c, t + 1));  // the next block's inputs
                if (s->dual) {
                    const bool lower = s->cell == a.root0;
                    if (!wait(lane == 0, ctr(a.up, lower ? a.root1 : a.root0), s->base + uint32_t(t) + 1u,
                              seen, false, s->root, c.j, 2))
                        return;
                    if (p.on) {
                        const T o = U::ld(ring(lower ? 1 : 0, t));
                        v = U::op(lower ? v : o, lower ? o : v);
                    }
                }
            }
            if (f < 0) continue;
            const Spot p = noted(f);
            if (!root) {
                if (!held) {
                    if (!wait(lane == 0, ctr(a.done, s->par_cell), final_at, seen, false, s->root, t, 3)) return;
                    if (p.on) w = U::ld(s->par + p.off);
                }
                v = w;
            }
            put(p, v, 0, s->n);
            if (join) {
                __syncwarp();
                if (lane == 0 && !s->mute) {
                    __threadfence();
                    sched::st_relaxed(ctr(a.up, s->cell), s->base + uint32_t(t) + 1u);
                    sched::st_relaxed(ctr(a.done, s->cell), s->base + uint32_t(t) + 1u);
                }
            } else if (s->next) {
                publish(a.done, s->base + uint32_t(t) + 1u);
            }
        }
    }
};

// Warp i of the grid runs cell i / slices, slice i % slices: neighbouring
// warps read neighbouring columns.
template <class Op, bool kVec, bool kRB>
__global__ void __launch_bounds__(kWarps * 32, kCtas) walk_kernel(const __grid_constant__ WalkArgs a)
{
    extern __shared__ __align__(16) uint4 walk_slots[];
    __shared__ WarpInfo info[kWarps];
    const int lane = int(threadIdx.x) & 31, w = int(threadIdx.x >> 5);
    const int64_t gw = int64_t(blockIdx.x) * kWarps + w;
    Call call = ask_call(a.ctl);
    const int lines = a.col.nslices + a.col.tail;  // the tail slice comes last
    const bool here = gw < int64_t(a.ncells) * lines;
    const int cell = int(gw / lines), g = int(gw % lines);
    WarpInfo* const s = &info[w];
    if (here) {
        const CellDesc* c = a.cells + cell;
        const int n = __ldg(&c->n), next = __ldg(&c->next);
        // past its ranks and nodes a descriptor holds zeros: no need to wait for n
        if (lane < kRanks) {
            s->x[lane] = sched::rank_in(a.x, __ldg(c->rank + lane));
            s->y[lane] = sched::rank_out(a.y, __ldg(c->rank + __ldg(c->lev_k + lane)));
            s->tape[lane] = uint8_t(__ldg(c->tape + lane));
        }
        if (lane < 2 * kExt) {
            s->ext[lane] = sched::rank_out(a.y, __ldg(c->ext_rank + lane));
            s->ext_cell[lane] = __ldg(c->ext_cell + lane);
        }
        if (lane < kExt) {
            s->ext_k[lane] = __ldg(c->ext_k + lane);
            s->ext_node[lane] = __ldg(c->rank + __ldg(c->ext_k + lane));
        }
        if (lane == 31) {
            const int par = __ldg(&c->par_rank);
            s->n = n;
            s->next = next;
            s->staged = min(next, (a.ranks - n) / 2);
            s->depth = __ldg(&c->depth);
            s->root = __ldg(&c->root);
            s->par_cell = __ldg(&c->par_cell);
            s->lag = s->par_cell < 0 ? 0 : s->depth - __ldg(&a.cells[s->par_cell].depth);
            s->reread = unsigned(__ldg(&c->reread));
            if (par >= 0) s->par = sched::rank_out(a.y, par);
            s->cell = cell;
            s->g = g;
            s->dual = a.root0 >= 0 && par < 0;
            s->mute = a.skip_rank >= 0 && s->root == a.skip_rank;
            s->stuck = -1;
            s->stuck_step = 0;
            if (a.skip_rank >= 0)
                for (int k = 0; k + 1 < n; k++)
                    if (__ldg(c->rank + k) == a.skip_rank) {
                        s->stuck = __ldg(c->node_par + k);
                        s->stuck_step = (__ldg(c->tape + k) & 4) ? 1 : 0;
                    }
        }
    }
    start_call(a.ctl, call);
    if (here) {
        if (lane == 0) {
            s->epoch = call.epoch;
            s->base = call.base;
        }
        __syncwarp();
        uint4* const slot = walk_slots + w * a.ranks * 32 + lane;
        if (kVec && Op::kEpv > 1 && g == a.col.nslices) {
            const Runner<Op, false, kRB> r{a, s, slot, lane, true};
            if (kRB) r.reduce_bcast();
            else r.algorithm_1();
        } else {
            const Runner<Op, kVec, kRB> r{a, s, slot, lane, false};
            if (kRB) r.reduce_bcast();
            else r.algorithm_1();
        }
        cp_async_wait_all();
    }
    finish_call(a.ctl, call, uint32_t(a.used), a.up, a.ctr_words);
}

template <bool kRB>
const void* kernel_for(int dtype, bool vec)
{
    switch (dtype) {
    case DPDR_INT32:
        return vec ? reinterpret_cast<const void*>(&walk_kernel<SumI32, true, kRB>)
                   : reinterpret_cast<const void*>(&walk_kernel<SumI32, false, kRB>);
    case DPDR_FLOAT32:
        return vec ? reinterpret_cast<const void*>(&walk_kernel<SumF32, true, kRB>)
                   : reinterpret_cast<const void*>(&walk_kernel<SumF32, false, kRB>);
    case DPDR_MAT2X2_F32:
        return vec ? reinterpret_cast<const void*>(&walk_kernel<MatF32, true, kRB>)
                   : reinterpret_cast<const void*>(&walk_kernel<MatF32, false, kRB>);
    default:
        return vec ? reinterpret_cast<const void*>(&walk_kernel<MatU32, true, kRB>)
                   : reinterpret_cast<const void*>(&walk_kernel<MatU32, false, kRB>);
    }
}

}  // namespace walk
}  // namespace dpdr
