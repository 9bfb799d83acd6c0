// cells_protocol.cu -- replays the exchanges of the schedule kernel on short
// blocks (words_kernel) on the host, over the cells, column slices and slot
// counts that the library computes (test infrastructure only).
//
// The kernel's cells send without waiting, so a slot of flagged words may be
// written again only when every reader of what it holds is known to have read
// it: the read must come before the write in every order in which the cells'
// warps can run.  Each cell's operations are put down in their program order,
// the cells run as far as their waits allow, and every cell keeps, per cell,
// the number of that cell's operations known to lie before its own next one
// (a send passes the sender's on).  A write is safe exactly when that number
// covers the readers' reads; holding back any warp at any point cannot break
// what this order proves.
#include <map>
#include <tuple>
#include <vector>

#include "schedule_cells.cuh"

using namespace dpdr;

namespace {

// One cell's operations for one column slice, in the order of Runner::run.
enum Channel { kUp, kDown, kDual };
struct Op {
    bool send;
    int channel, owner;  // owner: the sending cell
    int seq;             // the step whose block travels
};

// The rounds of line g, and whether its slice of the round holds units: the
// kernel's have one each; with `empty` those without are rounds, too.
template <class T, bool kVec>
std::vector<char> line_rounds(const cells::Columns& c, int g, bool empty)
{
    if (g == c.nslices) return {1};  // the tail
    std::vector<char> live;
    cells::Extent<uint32_t> x;
    if (empty)
        for (cells::Pos at(c, g); at.j < c.b; at.advance(c))
            live.push_back(cells::extent<T, kVec, uint32_t>(c, at, false).n > 0);
    else
        for (cells::Pos at(c, g); cells::next_slice<T, kVec>(c, at, false, x); at.advance(c))
            live.push_back(1);
    return live;
}

std::vector<Op> program(const std::vector<CellDesc>& cells, const CellPlan& C, int me,
                        const std::vector<char>& live)
{
    const CellDesc& c = cells[me];
    const int steps = int(live.size()), D = c.depth;
    const bool root = c.par_cell < 0, dual = root && C.root0 >= 0;
    std::vector<Op> ops;
    for (int t = 0; steps && t < steps + D + c.nlev - 1; t++) {
        if (t < steps && live[t]) {
            for (int h = 0; h < 2 * c.next; h++) ops.push_back({false, kUp, c.ext_cell[h], t});
            if (!root) ops.push_back({true, kUp, me, t});
            if (dual) {
                ops.push_back({true, kDual, me, t});
                ops.push_back({false, kDual, me == C.root0 ? C.root1 : C.root0, t});
            }
        }
        const int f = t - D;
        if (f >= 0 && f < steps && live[f]) {
            if (!root) ops.push_back({false, kDown, c.par_cell, f});
            if (c.next) ops.push_back({true, kDown, me, f});
        }
    }
    return ops;
}

// 0, or 1 a slot written before it was read, 2 cells that wait for ever;
// where: {channel, sending cell, its root's depth, step}.
int replay(const std::vector<CellDesc>& cells, const CellPlan& C, const std::vector<char>& live,
           const int slots[3], int* where)
{
    const int n = int(cells.size());
    std::vector<std::vector<Op>> ops(n);
    std::vector<std::vector<int>> readers(n);  // of the cell's final blocks
    for (int i = 0; i < n; i++) {
        ops[i] = program(cells, C, i, live);
        if (cells[i].par_cell >= 0) readers[cells[i].par_cell].push_back(i);
    }
    std::vector<int> pc(n, 0);
    std::vector<std::vector<int>> known(n, std::vector<int>(n, 0));
    std::map<std::tuple<int, int, int>, std::vector<int>> sent;  // what the sender knew
    std::map<std::tuple<int, int, int, int>, int> read;          // reader's operations up to its read
    std::map<std::tuple<int, int, int>, int> holds;              // step in a slot
    for (bool moved = true; moved;) {
        moved = false;
        for (int i = 0; i < n; i++)
            for (; pc[i] < int(ops[i].size()); pc[i]++, moved = true) {
                const Op& o = ops[i][pc[i]];
                const auto key = std::make_tuple(o.channel, o.owner, o.seq);
                known[i][i] = pc[i] + 1;
                if (!o.send) {
                    const auto s = sent.find(key);
                    if (s == sent.end()) break;
                    for (int k = 0; k < n; k++)
                        if (k != i && s->second[k] > known[i][k]) known[i][k] = s->second[k];
                    read[std::make_tuple(o.channel, o.owner, o.seq, i)] = pc[i] + 1;
                    continue;
                }
                const auto slot = std::make_tuple(o.channel, i, o.seq % slots[o.channel]);
                const auto old = holds.find(slot);
                if (old != holds.end()) {
                    const std::vector<int> one{o.channel == kUp ? cells[i].par_cell
                                               : i == C.root0   ? C.root1 : C.root0};
                    for (int r : o.channel == kDown ? readers[i] : one) {
                        const auto at = read.find(std::make_tuple(o.channel, i, old->second, r));
                        if (at == read.end() || at->second > known[i][r]) {
                            const int w[4] = {o.channel, i, cells[i].depth, o.seq};
                            for (int k = 0; k < 4; k++) where[k] = w[k];
                            return 1;
                        }
                    }
                }
                holds[slot] = o.seq;
                sent[key] = known[i];
            }
    }
    for (int i = 0; i < n; i++)
        if (pc[i] < int(ops[i].size())) {
            const Op& o = ops[i][pc[i]];
            const int w[4] = {o.channel, o.owner, cells[i].depth, o.seq};
            for (int k = 0; k < 4; k++) where[k] = w[k];
            return 2;
        }
    return 0;
}

}  // namespace

// Every line of a call on `warps` resident warps: 0, what replay returns, 3
// more steps than the call counts on, 4 the cells do not fit; out: {steps of
// the longest line, cells, depth of the deepest cell} and where it failed.
// down_slots (0: the kernel's) and empty change the kernel's rules.
extern "C" int words_protocol(int p, int64_t m, int esize, int single, int b, int aligned, int warps,
                              int down_slots, int empty, int* out)
{
    Plan P;
    P.p = p;
    P.m = m;
    P.b = b;
    P.esize = size_t(esize);
    P.topo = single ? DPDR_TOPO_SINGLE : DPDR_TOPO_DUAL;
    P.last_vector_path = aligned;
    P.parent.assign(p, -1);
    P.child0 = P.child1 = P.dual = P.parent;
    P.depth.assign(p, 0);
    build_tree(p, P.topo, P.parent.data(), P.child0.data(), P.child1.data(), P.dual.data(),
               P.depth.data());
    P.max_depth = *std::max_element(P.depth.begin(), P.depth.end());
    P.r0 = single ? -1 : p / 2 - 1;
    P.r1 = p - 1;
    CellPlan C;
    std::vector<CellDesc> cells;
    C.warps = warps;
    const bool fit = make_cells(&P, kWordsRanks, kWordsLevels, warps / 2, &C, &cells);
    out[1] = C.n;
    if (!fit) return 4;
    const bool vec = cell_vector(&P);
    const CellSlices S = cell_slices(&P, C, vec);
    const cells::Columns c{m, m / b, m % b, b, S.n, S.per_block, S.steps, cell_tail(&P, vec)};
    const int slots[3] = {word_slots(&P, S.steps), down_slots ? down_slots : word_slots(&P, S.steps),
                          kDualSlots};
    out[0] = 0;
    out[2] = 0;
    for (const CellDesc& d : cells) out[2] = std::max(out[2], d.depth);
    std::map<std::vector<char>, bool> seen;
    for (int g = 0; g < S.n + c.tail; g++) {
        const std::vector<char> live =
            esize == 4 ? (vec ? line_rounds<SumI32, true>(c, g, empty)
                              : line_rounds<SumI32, false>(c, g, empty))
                       : (vec ? line_rounds<MatU32, true>(c, g, empty)
                              : line_rounds<MatU32, false>(c, g, empty));
        if (int(live.size()) > S.steps) return 3;  // more than the call's flags
        out[0] = std::max(out[0], int(live.size()));
        if (seen[live]) continue;
        seen[live] = true;
        if (const int bad = replay(cells, C, live, slots, out + 3)) return bad;
    }
    return 0;
}

// The base of the next call's counters and flags of a plan on cells (walk:
// those of the counters kernels): returned, and set where `set` is not
// negative.  -1 after a CUDA error.
extern "C" long long cells_base(void* plan, int walk, long long set)
{
    const Plan* P = static_cast<const Plan*>(plan);
    uint32_t* const at = reinterpret_cast<uint32_t*>(walk ? P->walk.d : P->words.d) + 3;
    uint32_t base = uint32_t(set);
    if (cudaDeviceSynchronize() != cudaSuccess) return -1;
    if (set >= 0 && cudaMemcpy(at, &base, sizeof base, cudaMemcpyHostToDevice) != cudaSuccess) return -1;
    if (cudaMemcpy(&base, at, sizeof base, cudaMemcpyDeviceToHost) != cudaSuccess) return -1;
    return base;
}
