// schedule_words.cu -- the schedule-faithful kernel on short blocks with the
// virtual ranks gathered into subtree cells of at most 8 ranks and flagged
// words between them (dpdr_allreduce_schedule where every schedule option is
// automatic and the inputs are small; schedule_cells.cuh).
//
// The schedule is Algorithm 1's: in round j every rank takes its children's
// partial blocks j, forms Y[j] = t1 (.) (t0 (.) x_i), hands it to its parent
// (the dual roots exchange theirs) and receives final block j - d_i, which its
// parent received in round j - 1.  What passes in a round is not always a
// block of the partition, though: a warp's rounds are its column slices, up
// to two blocks' worth of them side by side (Columns), with the blocks in
// their order; a long block takes several rounds.
//
// What bounds it: the chain of exchanges from the leaves to the roots and
// back.  One trip through L2 takes 0.3 us on one die and 0.5 us across, and
// with one warp group per rank (schedule_ll.cu) there is one per tree level
// each way, about 1 us each with the polling loop; a cell takes three levels
// to one.  p = 288, m = 250 int32 in 10.5 us against 20.0 (captured calls,
// warm), p = 1152, m = 1 in 11.9 against 20.5, m = 4096 in 21.2 against 71,
// p = 36, m = 80000 in 14.2 against 47.
//
// Exchanges between cells go through slots of flagged words: every 32-bit
// word travels with the step's flag in one 64-bit store and the receiver
// polls the words themselves.  Flags never repeat (finish_call), so nothing
// is cleared between calls and a captured graph replays.  A sender never
// waits for a slot.  A warp's rounds are the slices that hold units, those
// without are passed over, alike in every cell: so in every round each cell
// hears from the others, which is what shows that a slot has been read.
//   dual  2 slots: the dual's partial j + 1 shows that it has read partial j.
//   up    depth + 1 slots: final block k shows that the parent has read
//         partial k, and final block j - 1 - d arrived in round j - 1.
//   down  depth + 1 slots of the receiving cell: final block f leaves the
//         root only with the cell's partial block f in it, which the cell,
//         at depth d, sent in round f, having taken final block f - 1 - d in
//         the round before.  While partial blocks come, a parent l levels
//         above knows of the last l + 1 rounds only and 5 slots would do; in
//         the rounds after the last partial block nothing tells it more than
//         that, however many final blocks it sends.
// A cell waits in round j for its children's partial blocks j, which they
// send before they wait for anything later than round j - 1, for the dual
// root's partial j, sent before the wait, and for final block j - d, which its
// parent sent in round j - 1 or before: with all CTAs resident (cooperative
// launch) nothing deadlocks.  In place (y_i == x_i) every lane reads x_i of a
// block before it writes any y_i of it.  Every wait is bounded in time.
//
// The loops over ranks stay rolled: unrolled, the code no longer fitted the
// instruction cache and the same calls took 1.5 to 2 times as long.  128
// registers: at 96 the polling loop spills (p = 36, m = 80000: 20 us).
#include "schedule_cells.cuh"

namespace dpdr {
namespace {

using namespace cells;
// Numbers of elements and bytes of a row: inputs on flagged words are at most
// 24 MiB (schedule_transport).  With 64 bits finding the next slice was long
// enough to hold up a step (p = 19, m = 39982, b = 175 int32 180 and 172 us,
// p = 288, m = 768, b = 12 24.9 and 23.0).
using Index = uint32_t;
using Spot = SpotOf<Index>;

constexpr int kRanks = kWordsRanks;
constexpr int kLevels = kWordsLevels;
constexpr int kExt = kRanks / 2;
constexpr int kWarps = 4;     // per CTA
constexpr int kNodes = 2;     // nodes that take their children's values at once
constexpr int kSlot = 32 * 4;  // words of a slot: 32 units of 16 bytes

struct WordsArgs {
    const char* const* x;
    char* const* y;
    const CellDesc* cells;
    uint32_t* ctl;
    uint32_t* err;
    u64* dual;           // [2 sides][slices][kDualSlots] slots: the roots' partial blocks
    u64* down;           // [cells with children][slices][slots]: final blocks
    u64* up;             // [cells][slices][slots]: partial blocks
    int64_t words;       // 32-bit words of all slots, from dual on
    Columns col;
    int64_t wait_ns;
    int slots;           // word_slots
    int ncells, root0;   // root0: cell of the lower root (-1: one tree)
    int used;            // flag values the call uses
    int skip_rank;
};

struct WarpInfo {        // one per warp, in shared memory
    const char* x[kRanks];      // input rows, in post-order
    char* y[kRanks];            // output rows, by level (the cell's root first)
    // slots of this warp's slice: the child cells' and its own partial blocks,
    // its parent's and its own final blocks, the dual's and its own
    const u64* up_in[2 * kExt];
    u64* up_out;
    const u64* down_in;
    u64* down_out;
    const u64* dual_in;
    u64* dual_out;
    u64 tape;                   // one byte per rank in post-order (CellDesc::tape)
    int n, next, nlev, depth, root, par_cell;
    int lev_off[kLevels + 1];
    int ext_k[kExt];
    int cell, g;                // this warp's cell and column slice
    uint32_t epoch, base;       // of the call: abort mark, flag base
    int dual;                   // the cell holds a dual root
    int mute;                   // fault injection: the cell's root never sends
    int stuck, stuck_step;      // fault injection: parent in this cell of the silent rank
                                // (-1: none), and which child that is
};

// One warp's run of its cell for its column slices.
template <class Op, bool kVec>
struct Runner {
    using U = Unit<Op, kVec>;
    using T = typename U::T;
    const WordsArgs& a;
    const WarpInfo* s;
    uint4* slot;         // this lane's cells: the unit of position k at k * 32
    int lane;
    bool tail;

    // Receives the lane's unit of n <= N slots that carry `flag`, all polled
    // together; one that is complete on every lane is not read again.
    template <int N>
    __device__ __forceinline__ bool recv(const u64* const* from, int64_t at, int n, uint32_t flag,
                                         const Spot& p, T* v, int j, int step) const
    {
        unsigned pend = (1u << n) - 1u;
        const int64_t w = at + lane * (U::kBytes / 4);
        uint64_t t0 = 0;
        for (unsigned polls = 0;; polls++) {
            unsigned left = 0;
            if (p.on) {
#pragma unroll
                for (int h = 0; h < N; h++)
                    if ((pend >> h) & 1u)
                        if (!U::recv(from[h] + w, flag, v[h])) left |= 1u << h;
            }
            pend = __reduce_or_sync(kAll, left);
            if (!pend) return true;
            if (polls == 0) t0 = sched::now_ns();
            else if ((polls & 15) == 0) {
                const int stop = give_up(a.ctl, s->epoch, t0, a.wait_ns);
                if (stop == 2 && lane == 0)
                    wait_expired(a.err, a.ctl, s->epoch, s->root, j,
                                 step < 0 ? (__ffs(pend) - 1) & 1 : step);
                if (stop) return false;
                if (polls >= 64) __nanosleep(64);
            }
        }
    }
    __device__ __forceinline__ void send(u64* to, uint32_t flag, const Spot& p, const T& v) const
    {
        if (p.on && !s->mute) U::send(to + lane * (U::kBytes / 4), flag, v);
    }

    __device__ __forceinline__ T& at(int k) const { return *reinterpret_cast<T*>(slot + k * 32); }

    // Starts the copies of every rank's input into the lane's slots.
    __device__ __forceinline__ void fetch(const Spot& p) const
    {
        const int n = s->n;
#pragma unroll 1
        for (int k = 0; k < n; k++)
            if (p.on) U::copy(slot + k * 32, s->x[k] + p.off);
    }

    // The cell root's value of the units in the slots, the bottom nodes having
    // taken their children's values: the fold of the slots in post-order.
    // A child_1 inside the cell waits for its parent in its own slot.
    __device__ __forceinline__ T fold() const
    {
        T acc{};
        u64 tape = s->tape;
        const int n = s->n;
#pragma unroll 1
        for (int k = 0; k < n; k++, tape >>= 8) {
            const unsigned t = unsigned(tape);
            T v = at(k);
            if (t & 3u) {
                v = U::op(acc, v);
                if (t & 2u) v = U::op(at(int((t >> 3) & 31u)), v);
            }
            acc = v;
            if (t & 4u) at(k) = v;
        }
        return acc;
    }

    // Steps child_0 and child_1 of step t (round j of its wave), the inputs
    // being on their way into the slots: v becomes the cell's partial block.
    // Returns false when a wait expired.
    __device__ __forceinline__ bool fold_step(int t, int j, const Spot& p, T& v) const
    {
        const int next = s->next;
        const uint32_t flag = s->base + uint32_t(t) + 1u;
        if (s->stuck >= 0) {  // the silent rank of the fault injection: wait in vain
            uint32_t seen = 0;
            if (!wait_counters(a.ctl, a.err, a.wait_ns, s->epoch, a.ctl, 0, seen, false, lane == 0,
                               s->stuck, j, s->stuck_step))
                return false;
        }
        bool landed = false;
#pragma unroll 1
        for (int q0 = 0; q0 < next; q0 += kNodes) {
            T e[2 * kNodes];
            if (!recv<2 * kNodes>(s->up_in + 2 * q0, int64_t(t & (a.slots - 1)) * kSlot,
                                  2 * min(kNodes, next - q0), flag, p, e, j, -1))
                return false;
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

    // v: a final block's unit, into the rows y[t0 .. t1)
    __device__ __forceinline__ void put(const Spot& p, const T& v, int t0, int t1) const
    {
#pragma unroll 1
        for (int t = t0; t < t1; t++)
            if (p.on) U::st(s->y[t] + p.off, v);
    }

    // The lane's unit of the warp's next slice, from `at` on; false past the last.
    __device__ __forceinline__ bool ahead(Pos& at, Spot& p) const
    {
        Extent<Index> x{0, 0};
        const bool there = next_slice<Op, kVec>(a.col, at, tail, x);
        p = Spot{(x.u + lane) * U::kBytes, lane < x.n};
        return there;
    }

    // A final block that reaches the cell's root in step t reaches the ranks
    // l levels below it in step t + l: the last ones wait in registers.
    __device__ __forceinline__ void run() const
    {
        static_assert(kLevels == 4, "the history of final blocks is three deep");
        const int D = s->depth, nlev = s->nlev;
        const bool root = s->par_cell < 0;
        int steps = tail ? 1 : a.col.steps;  // or fewer, once the last slice is seen
        Pos c(a.col, tail ? 0 : s->g), d(a.col, tail ? 0 : s->g);
        Spot next;
        if (!ahead(c, next)) return;
        fetch(next);
        T v1{}, v2{}, v3{};
        Spot p1{0, false}, p2{0, false}, p3{0, false};
#pragma unroll 1
        for (int t = 0; t < steps + D + nlev - 1; t++) {
            T v{}, in[1];
            Spot now = next;
            if (t < steps) {
                const uint32_t flag = s->base + uint32_t(t) + 1u;
                if (!fold_step(t, c.j, now, v)) return;
                if (!root) {
                    send(s->up_out + (t & (a.slots - 1)) * kSlot, flag, now, v);
                } else if (s->dual) {
                    send(s->dual_out + (t & (kDualSlots - 1)) * kSlot, flag, now, v);
                    if (!recv<1>(&s->dual_in, (t & (kDualSlots - 1)) * kSlot, 1, flag, now, in, c.j, 2))
                        return;
                    v = s->cell == a.root0 ? U::op(v, in[0]) : U::op(in[0], v);
                }
                c.advance(a.col);
                if (t + 1 < steps) {  // the next block's inputs
                    if (ahead(c, next)) fetch(next);
                    else steps = t + 1;
                }
            }
            const int f = t - D;  // the step whose block is final here now
            if (f < 0) continue;
            if (f < steps) {
                const uint32_t flag = s->base + uint32_t(f) + 1u;
                if (!root) {
                    ahead(d, now);
                    if (!recv<1>(&s->down_in, (f & (a.slots - 1)) * kSlot, 1, flag, now, in, d.j + D, 3))
                        return;
                    v = in[0];
                    d.advance(a.col);
                }
                if (s->next) send(s->down_out + (f & (a.slots - 1)) * kSlot, flag, now, v);
            } else {
                now.on = false;
            }
            put(now, v, 0, 1);
            if (nlev > 1) put(p1, v1, s->lev_off[1], s->lev_off[2]);
            if (nlev > 2) put(p2, v2, s->lev_off[2], s->lev_off[3]);
            if (nlev > 3) put(p3, v3, s->lev_off[3], s->lev_off[4]);
            p3 = p2, v3 = v2, p2 = p1, v2 = v1, p1 = now, v1 = v;
        }
    }
};

// Warp i of the grid runs cell i / slices, slice i % slices.
template <class Op, bool kVec>
__global__ void __launch_bounds__(kWarps * 32, 4) words_kernel(const __grid_constant__ WordsArgs a)
{
    __shared__ __align__(16) uint4 slots[kWarps * kRanks * 32];
    __shared__ WarpInfo info[kWarps];
    const int lane = int(threadIdx.x) & 31, w = int(threadIdx.x) >> 5;
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
            reinterpret_cast<uint8_t*>(&s->tape)[lane] = uint8_t(__ldg(c->tape + lane));
        }
        if (lane < 2 * kExt)
            s->up_in[lane] = a.up + (int64_t(__ldg(c->ext_cell + lane)) * lines + g) * a.slots * kSlot;
        if (lane < kExt) s->ext_k[lane] = __ldg(c->ext_k + lane);
        if (lane <= kLevels) s->lev_off[lane] = __ldg(c->lev_off + lane);
        if (lane == 31) {
            const int side = cell == a.root0 ? 0 : 1;
            s->n = n;
            s->next = next;
            s->nlev = __ldg(&c->nlev);
            s->depth = __ldg(&c->depth);
            s->root = __ldg(&c->root);
            s->par_cell = __ldg(&c->par_cell);
            s->cell = cell;
            s->g = g;
            s->dual = a.root0 >= 0 && s->par_cell < 0;
            s->up_out = a.up + (int64_t(cell) * lines + g) * a.slots * kSlot;
            s->down_in = a.down + (int64_t(__ldg(&c->par_down)) * lines + g) * a.slots * kSlot;
            s->down_out = a.down + (int64_t(__ldg(&c->down)) * lines + g) * a.slots * kSlot;
            s->dual_out = a.dual + (int64_t(side) * lines + g) * kDualSlots * kSlot;
            s->dual_in = a.dual + (int64_t(1 - side) * lines + g) * kDualSlots * kSlot;
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
        uint4* const slot = slots + w * kRanks * 32 + lane;
        if (kVec && Op::kEpv > 1 && g == a.col.nslices)
            Runner<Op, false>{a, s, slot, lane, true}.run();
        else
            Runner<Op, kVec>{a, s, slot, lane, false}.run();
        cp_async_wait_all();
    }
    finish_call(a.ctl, call, uint32_t(a.used), reinterpret_cast<uint32_t*>(a.dual), a.words);
}

template <class Op>
const void* words_ptr(bool vec)
{
    return vec ? reinterpret_cast<const void*>(&words_kernel<Op, true>)
               : reinterpret_cast<const void*>(&words_kernel<Op, false>);
}
const void* words_kernel_for(int dtype, bool vec)
{
    switch (dtype) {
    case DPDR_INT32: return words_ptr<SumI32>(vec);
    case DPDR_FLOAT32: return words_ptr<SumF32>(vec);
    case DPDR_MAT2X2_F32: return words_ptr<MatF32>(vec);
    default: return words_ptr<MatU32>(vec);
    }
}

// 64-bit words of the slots of a call on S.n slices and the tail.
size_t slot_words(const Plan* P, const CellSlices& S)
{
    return size_t(S.n + 1) * kSlot *
           (2 * kDualSlots + size_t(P->words.down + P->words.n) * word_slots(P, S.steps));
}

}  // namespace

int schedule_words_prepare(Plan* P)
{
    CellPlan& C = P->words;
    C.ready = false;
    int occ[2] = {0, 0};
    for (int vec = 0; vec < 2; vec++) {
        const cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(
            &occ[vec], words_kernel_for(P->dtype, vec != 0), kWarps * 32, 0);
        if (e != cudaSuccess) return cuda_fail(e, "schedule words: occupancy");
    }
    C.warps = std::min(occ[0], occ[1]) * P->num_sms * kWarps;
    std::vector<CellDesc> desc;
    if (!make_cells(P, kRanks, kLevels, C.warps / 2, &C, &desc))
        return DPDR_OK;  // a slice and the tail do not fit
    C.off_scratch = 256 + (sizeof(CellDesc) * desc.size() + 255) / 256 * 256;
    C.scratch = std::max(slot_words(P, cell_slices(P, C, false)), slot_words(P, cell_slices(P, C, true))) *
                sizeof(u64);
    const int rc = cell_scratch(P, &C, desc.data(), sizeof(CellDesc) * desc.size());
    C.ready = rc == DPDR_OK;
    return rc;
}

int schedule_words_launch(Plan* P, cudaStream_t s)
{
    const CellPlan& C = P->words;
    const bool vec = cell_vector(P);
    WordsArgs a;
    a.x = P->d_x;
    a.y = P->d_y;
    a.cells = reinterpret_cast<const CellDesc*>(C.d + 256);
    a.ctl = reinterpret_cast<uint32_t*>(C.d);
    a.err = P->d_err;
    const CellSlices S = cell_slices(P, C, vec);
    a.col = Columns{P->m, P->m / P->b, P->m % P->b, P->b, S.n, S.per_block, S.steps, cell_tail(P, vec)};
    const int lines = S.n + a.col.tail;
    a.dual = reinterpret_cast<u64*>(C.d + C.off_scratch);
    a.slots = word_slots(P, S.steps);
    a.down = a.dual + size_t(lines) * 2 * kDualSlots * kSlot;
    a.up = a.down + size_t(C.down) * lines * a.slots * kSlot;
    a.words = int64_t(C.scratch / 4);
    a.wait_ns = P->wait_ns;
    a.ncells = C.n;
    a.root0 = C.root0;
    a.used = S.steps + 1;
    a.skip_rank = P->skip_rank;
    return cell_launch(words_kernel_for(P->dtype, vec), &a, int64_t(C.n) * lines, kWarps, 0, s);
}

}  // namespace dpdr
