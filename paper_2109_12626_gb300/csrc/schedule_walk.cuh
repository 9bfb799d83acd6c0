// schedule_walk.cuh -- the schedule-faithful kernels on large pipeline
// blocks, the virtual ranks gathered into subtree cells of at most
// kWalkRanks ranks (dpdr_allreduce_schedule and dpdr_allreduce_reduce_bcast
// where every schedule option is automatic; schedule_cells.cuh).
//
// The schedule is Algorithm 1's, round by round: in round j every rank takes
// its children's partial blocks j, forms Y[j] = t1 (.) (t0 (.) x_i) and hands
// it to its parent (the dual roots exchange theirs), then receives final
// block j - d_i, which its parent holds since round j - 1.
//
// What bounds it: a step of a warp (32 units of all its ranks, 8 KB in and
// 8 KB out for 16 ranks) is a chain of about 6 us -- the children's counters
// and partial blocks, the fold, a release fence, the parent's counter and
// final block, the stores, another fence -- and device memory.  24 warps per
// SM, each with its next step's inputs on their way into shared memory
// (cp.async) while it waits, cover the chain.  With a warp group per rank
// (schedule.cu) every block crosses L2 once per tree edge and direction, each
// time behind such a chain; here one edge in fifteen does.  Measured (captured
// calls, inputs larger than L2, before and after): p = 1152 int32, m = 2^16 in
// 246 and 148 us, m = 2^18 673 and 532; p = 288, m = 212500 244 and 129; p = 32
// float32, m = 2^23, b = 16 570 and 395, b = 64 850 and 395; p = 36 2x2
// matrices, m = 2^20 352 and 231; reduce, then broadcast at p = 288,
// m = 875000 in 16000-element blocks 909 and 466.
// Not kept: 4 units per lane (fewer, longer steps; the registers for them
// spilled, and a spilled value comes back from L2 after every acquire); a
// warp for each direction (the two loops together no longer fitted the
// instruction cache: 1.5 to 2.5 times as long); inputs in registers instead
// of shared memory, 32 warps of 64 registers (p = 1152 16 % faster, blocks
// that do not fill the GPU 20 % slower).
//
// Exchanges between cells: the cell root's partial block goes to its y row
// (a dual root's to an exchange slot) and a release store of the cell's up
// counter publishes it; a final block is read from the parent rank's y row
// once the parent cell's done counter says that it finished round j - 1.
// Counters never repeat (finish_call), so a call is one kernel and a
// captured graph replays.
//
// Order and reuse.  A cell waits in round j for its children's partial blocks
// j, which they publish before they wait for anything later than round
// j - 1, for the dual root's partial j, published before the wait, and for
// its parent's round j - 1: with all CTAs resident (cooperative launch)
// nothing deadlocks.  The final block j overwrites partial block j in the
// cell root's y row only after the parent has read it, and an exchange slot
// of parity j & 1 is written again in round j + 2, after the dual's partial
// j + 1 has shown that it finished round j.  In place (y_i == x_i) every lane
// reads x_i of a block before it writes any y_i of it.  Every wait is bounded
// in time; an expired wait records {rank, round, step}, marks the call's
// epoch aborted and every other wait of the call gives up.
#pragma once

#include "schedule_cells.cuh"

namespace dpdr {
namespace walk {

using namespace cells;

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
    uint32_t* done;      // the same: rounds finished
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
    int lev_off[kLevels + 1];
    int ext_k[kExt];
    int ext_cell[2 * kExt];
    int ext_node[kExt];         // the nodes' ranks
    int n, next, nlev, depth, root, par_cell;
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
        const Extent x = extent<Op, kVec>(a.col, c, tail);
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
    __device__ __forceinline__ bool wait(bool mine, const uint32_t* c, uint32_t target, bool never,
                                         int rank, int j, int step) const
    {
        return wait_counters(a.ctl, a.err, a.wait_ns, s->epoch, c, target, mine, never, rank, j, step);
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

    // Steps child_0 and child_1 of step t (round j of its wave), the inputs
    // being on their way into the slots: v becomes the cell's partial block.
    // Returns false when a wait expired.
    __device__ __forceinline__ bool up(int t, int j, const Spot& p, T& v) const
    {
        const int next = s->next;
        if (next || s->stuck >= 0) {
            const bool mine = lane < 2 * next, never = s->stuck >= 0 && lane == 31;
            if (!wait(mine, ctr(a.up, mine ? s->ext_cell[lane] : 0), s->base + uint32_t(t) + 1u, never,
                      never ? s->stuck : mine ? s->ext_node[lane >> 1] : 0, j,
                      never ? s->stuck_step : lane & 1))
                return false;
        }
        bool landed = false;
#pragma unroll 1
        for (int q0 = 0; q0 < next; q0 += kNodes) {
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
        v = fold();
        return true;
    }

    // The partial block of step t handed up: to the cell root's row, or a dual
    // root's exchange slot.  Before the next inputs are asked for: the release
    // would wait for them (p = 32, m = 2^23 float32, 415 and 405 us).
    __device__ __forceinline__ void hand_up(int t, const Spot& p, const T& v) const
    {
        if (p.on) U::st_keep(s->dual ? ring(s->cell == a.root0 ? 0 : 1, t) : s->y[0] + p.off, v);
        publish(a.up, s->base + uint32_t(t) + 1u);
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
        Pos c(a.col, tail ? 0 : s->g);
        Spot p = note(c, 0);
        fetch(p);
#pragma unroll 1
        for (int t = 0; t < steps; t++) {
            T v;
            if (!up(t, c.j, p, v)) return;
            const Spot was = p;
            c.advance(a.col);
            hand_up(t, was, v);
            if (t + 1 < steps) {  // the next block's inputs
                p = note(c, t + 1);
                fetch(p);
            }
        }
        c = Pos(a.col, tail ? 0 : s->g);
#pragma unroll 1
        for (int t = 0; t < steps; t++, c.advance(a.col)) {
            p = note(c, t);
            if (!root && !wait(lane == 0, ctr(a.done, s->par_cell), s->base + uint32_t(t) + 1u, false,
                               s->root, c.j, 3))
                return;
            T v{};
            if (p.on) v = U::ld((root ? s->y[0] : s->par) + p.off);  // a root holds the block
            put(p, v, root ? 1 : 0, s->n);
            if (s->next) publish(a.done, s->base + uint32_t(t) + 1u);
        }
    }

    // Algorithm 1.  A final block that reaches the cell's root in step t
    // reaches the ranks l levels below it in step t + l, from the cell root's
    // row, which holds it since: those loads are under way from the start of
    // the step.
    __device__ __forceinline__ void algorithm_1() const
    {
        const int steps = tail ? 1 : a.col.steps, D = s->depth, nlev = s->nlev;
        const bool root = s->par_cell < 0;
        Pos c(a.col, tail ? 0 : s->g);
        fetch(note(c, 0));
        const int last = steps - 1 + D + nlev - 1;
#pragma unroll 1
        for (int t = 0; t <= last; t++) {
            const int f = t - D;  // the step whose block is final at the cell's root now
            T h[kLevels - 1];
#pragma unroll
            for (int l = 1; l < kLevels; l++)
                if (l < nlev && f - l >= 0 && f - l < steps) {
                    const Spot q = noted(f - l);
                    if (q.on) h[l - 1] = U::ld(s->y[0] + q.off);
                }
            T v{};
            if (t < steps) {
                const Spot p = noted(t);
                if (!up(t, c.j, p, v)) return;
                c.advance(a.col);
                if (!root || s->dual) hand_up(t, p, v);
                if (t + 1 < steps) fetch(note(c, t + 1));  // the next block's inputs
                if (s->dual) {
                    const bool lower = s->cell == a.root0;
                    if (!wait(lane == 0, ctr(a.up, lower ? a.root1 : a.root0), s->base + uint32_t(t) + 1u,
                              false, s->root, c.j, 2))
                        return;
                    if (p.on) {
                        const T o = U::ld(ring(lower ? 1 : 0, t));
                        v = U::op(lower ? v : o, lower ? o : v);
                    }
                }
            }
            if (f < 0) continue;
#pragma unroll
            for (int l = 1; l < kLevels; l++)
                if (l < nlev && f - l >= 0 && f - l < steps)
                    put(noted(f - l), h[l - 1], s->lev_off[l], s->lev_off[l + 1]);
            if (f < steps) {
                const Spot p = noted(f);
                if (!root) {
                    if (!wait(lane == 0, ctr(a.done, s->par_cell), s->base + uint32_t(t), false, s->root, t, 3))
                        return;
                    if (p.on) v = U::ld(s->par + p.off);
                }
                put(p, v, 0, 1);
            }
            if (s->next) publish(a.done, s->base + uint32_t(t) + 1u);
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
    const uint32_t epoch = *reinterpret_cast<volatile const uint32_t*>(a.ctl);
    const uint32_t base = *reinterpret_cast<volatile const uint32_t*>(a.ctl + 3);
    const int lines = a.col.nslices + a.col.tail;  // the tail slice comes last
    if (gw < int64_t(a.ncells) * lines) {
        WarpInfo* const s = &info[w];
        const int cell = int(gw / lines), g = int(gw % lines);
        const CellDesc* c = a.cells + cell;
        const int n = __ldg(&c->n), next = __ldg(&c->next);
        if (lane < n) {
            s->x[lane] = sched::rank_in(a.x, __ldg(c->rank + lane));
            s->y[lane] = sched::rank_out(a.y, __ldg(c->rank + __ldg(c->lev_k + lane)));
            s->tape[lane] = uint8_t(__ldg(c->tape + lane));
        }
        if (lane < 2 * next) {
            s->ext[lane] = sched::rank_out(a.y, __ldg(c->ext_rank + lane));
            s->ext_cell[lane] = __ldg(c->ext_cell + lane);
        }
        if (lane < next) {
            s->ext_k[lane] = __ldg(c->ext_k + lane);
            s->ext_node[lane] = __ldg(c->rank + __ldg(c->ext_k + lane));
        }
        if (lane <= kLevels) s->lev_off[lane] = __ldg(c->lev_off + lane);
        if (lane == 31) {
            const int par = __ldg(&c->par_rank);
            s->n = n;
            s->next = next;
            s->nlev = __ldg(&c->nlev);
            s->depth = __ldg(&c->depth);
            s->root = __ldg(&c->root);
            s->par_cell = __ldg(&c->par_cell);
            s->reread = unsigned(__ldg(&c->reread));
            if (par >= 0) s->par = sched::rank_out(a.y, par);
            s->cell = cell;
            s->g = g;
            s->epoch = epoch;
            s->base = base;
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
    finish_call(a.ctl, epoch, base, uint32_t(a.used), a.up, a.ctr_words);
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
