// cells.cpp -- host side of the schedule kernels on subtree cells: how the
// trees are cut into cells, the cells' device descriptors, their column
// slices, scratch and launches (schedule_cells.cuh, schedule_words.cu,
// schedule_walk.cu).
#include <algorithm>
#include <utility>

#include "dpdr_internal.h"

namespace dpdr {
namespace {

// One way to cut a subtree: its open piece (the part that holds the subtree's
// root) joins what lies above, the cells below it are closed.
struct Cut {
    int tiers, cells;   // cells on the longest path below the piece; cells below
    bool join;          // the node's children are in its piece, as pieces s0, s1
    int s0, s1;
    bool operator<(const Cut& o) const { return tiers != o.tiers ? tiers < o.tiers : cells < o.cells; }
};
constexpr int kNoCut = 1 << 28;

// A cut of the plan's trees.  Cells are numbered by their root ranks, so
// that child cells come before their parents' cells.
struct Cells {
    std::vector<int> cell, pos;     // of each rank: its cell, its place in the cell's post-order
    std::vector<char> top;          // whether it is the cell's root
    std::vector<int> first, ranks;  // cell k: ranks[first[k]] .. ranks[first[k + 1] - 1]
};

// The cells of the plan's trees, and how many (returned); when they are more
// than max_cells, that alone.  A node's children are both in its cell or
// both roots of other cells, and a cell holds at most max_ranks ranks on
// max_levels levels.  Of all such cuts: the fewest cells between a leaf and
// the root (each costs an exchange through L2 each way), then the fewest
// cells.  Subtrees of a complete tree that have the same size have the same
// shape, so the best cut is found once per size; pieces are numbered
// (ranks - 1) * max_levels + (levels - 1).
int cut_cells(const Plan* P, int max_ranks, int max_levels, int max_cells, Cells* out)
{
    const int p = P->p, pieces = max_ranks * max_levels;
    std::vector<int> size(p), shape_of(p + 1, -1), best;  // a size's shape, a shape's best piece
    std::vector<std::vector<Cut>> cuts;                   // by shape
    for (int i = 0; i < p; i++) {  // post-order: children first
        const int c0 = P->child0[i], c1 = P->child1[i];
        size[i] = 1 + (c0 >= 0 ? size[c0] : 0) + (c1 >= 0 ? size[c1] : 0);
        if (shape_of[size[i]] >= 0) continue;
        std::vector<Cut> c(pieces, Cut{kNoCut, 0, false, 0, 0});
        if (c0 < 0) {
            c[0] = Cut{0, 0, false, 0, 0};
        } else {
            const int sa = shape_of[size[c0]], sd = c1 >= 0 ? shape_of[size[c1]] : sa;
            const std::vector<Cut>&a = cuts[sa], &d = cuts[sd];
            if (c1 >= 0) {
                const Cut x = a[best[sa]], y = d[best[sd]];
                c[0] = Cut{1 + std::max(x.tiers, y.tiers), 2 + x.cells + y.cells, false, 0, 0};
            }
            for (int s0 = 0; s0 < pieces; s0++) {
                if (a[s0].tiers >= kNoCut) continue;
                for (int s1 = 0; s1 < (c1 >= 0 ? pieces : 1); s1++) {
                    const Cut x = a[s0], y = c1 >= 0 ? d[s1] : Cut{0, 0, false, 0, 0};
                    if (y.tiers >= kNoCut) continue;
                    const int n = 1 + s0 / max_levels + 1 + (c1 >= 0 ? s1 / max_levels + 1 : 0);
                    const int l = 1 + std::max(s0 % max_levels + 1, c1 >= 0 ? s1 % max_levels + 1 : 0);
                    if (n > max_ranks || l > max_levels) continue;
                    Cut& b = c[(n - 1) * max_levels + l - 1];
                    const Cut j{std::max(x.tiers, y.tiers), x.cells + y.cells, true, s0, s1};
                    if (j < b) b = j;
                }
            }
        }
        shape_of[size[i]] = int(cuts.size());
        best.push_back(int(std::min_element(c.begin(), c.end()) - c.begin()));
        cuts.push_back(std::move(c));
    }
    auto cells_below = [&](int i) { return cuts[shape_of[size[i]]][best[shape_of[size[i]]]].cells; };
    const int n = 1 + cells_below(P->r1) + (P->r0 >= 0 ? 1 + cells_below(P->r0) : 0);
    if (n > max_cells) return n;

    std::vector<int> piece(p, 0);
    out->top.assign(p, 0);
    for (int i = p - 1; i >= 0; i--) {  // parents first: the pieces chosen
        const int shape = shape_of[size[i]];
        if (P->parent[i] < 0) out->top[i] = 1;
        if (out->top[i]) piece[i] = best[shape];
        const int c0 = P->child0[i], c1 = P->child1[i];
        if (c0 < 0) continue;
        const Cut& k = cuts[shape][piece[i]];
        out->top[c0] = !k.join;
        piece[c0] = k.s0;
        if (c1 >= 0) {
            out->top[c1] = !k.join;
            piece[c1] = k.s1;
        }
    }
    out->cell.resize(p);
    out->first.assign(n + 1, 0);
    for (int i = p - 1, k = n; i >= 0; i--) {
        out->cell[i] = out->top[i] ? --k : out->cell[P->parent[i]];
        out->first[out->cell[i] + 1]++;
    }
    for (int k = 0; k < n; k++) out->first[k + 1] += out->first[k];
    std::vector<int> held(n, 0);
    out->pos.resize(p);
    out->ranks.resize(p);
    for (int i = 0; i < p; i++) {  // the cell's root is its last rank
        const int k = out->cell[i];
        out->pos[i] = held[k]++;
        out->ranks[out->first[k] + out->pos[i]] = i;
    }
    return n;
}

bool is_second(const Plan* P, int i) { return P->parent[i] >= 0 && P->child1[P->parent[i]] == i; }

}  // namespace

// The cells' descriptors; false when there are more than max_cells of them.
bool make_cells(const Plan* P, int max_ranks, int max_levels, int max_cells, CellPlan* C,
                std::vector<CellDesc>* out)
{
    Cells cells;
    C->n = cut_cells(P, max_ranks, max_levels, max_cells, &cells);
    out->clear();
    if (C->n > max_cells) return false;
    out->resize(C->n);  // zeros
    C->root0 = P->r0 >= 0 ? cells.cell[P->r0] : -1;
    C->root1 = cells.cell[P->r1];
    C->down = C->ranks = 0;
    for (int k = 0; k < C->n; k++) {
        const int* const ranks = cells.ranks.data() + cells.first[k];
        CellDesc& c = (*out)[k];
        c.n = cells.first[k + 1] - cells.first[k];
        C->ranks = std::max(C->ranks, c.n);
        c.root = ranks[c.n - 1];
        c.depth = P->depth[c.root];
        c.par_rank = P->parent[c.root];
        c.par_cell = c.par_rank < 0 ? -1 : cells.cell[c.par_rank];
        unsigned again = 0;  // positions whose final blocks child cells read
        for (int t = 0; t < c.n; t++) {
            const int i = ranks[t], c0 = P->child0[i], c1 = P->child1[i];
            const bool in = c0 >= 0 && !cells.top[c0];
            const int pos1 = in && c1 >= 0 ? cells.pos[c1] : 0;
            c.nlev = std::max(c.nlev, P->depth[i] - c.depth + 1);
            c.lev_off[P->depth[i] - c.depth + 1]++;
            c.rank[t] = i;
            c.node_par[t] = i == c.root ? -1 : P->parent[i];
            c.tape[t] = (in ? (c1 >= 0 ? 2 : 1) : 0) | (i != c.root && is_second(P, i) ? 4 : 0) |
                        (pos1 << 3);
            if (c0 >= 0 && !in) {  // two children: a single one always joins
                c.ext_k[c.next] = t;
                c.ext_cell[2 * c.next] = cells.cell[c0];
                c.ext_cell[2 * c.next + 1] = cells.cell[c1];
                c.ext_rank[2 * c.next] = c0;
                c.ext_rank[2 * c.next + 1] = c1;
                c.next++;
                again |= 1u << t;
            }
        }
        for (int l = 0; l < kCellLevels; l++) c.lev_off[l + 1] += c.lev_off[l];
        int at[kCellLevels];
        std::copy(c.lev_off, c.lev_off + kCellLevels, at);
        for (int q = 0; q < c.n; q++) {
            const int t = at[P->depth[ranks[q]] - c.depth]++;
            c.lev_k[t] = q;
            c.reread |= int((again >> q) & 1u) << t;
        }
        c.down = c.next ? C->down++ : 0;
    }
    for (CellDesc& c : *out) c.par_down = c.par_cell < 0 ? 0 : (*out)[c.par_cell].down;
    return true;
}

// Slices of 32 units, those of all blocks one after another, dealt out to the
// warps there are for them (but for a slice of the row's last elements), so
// that a step keeps all of them busy whatever a block's length: p = 1152,
// m = 2^16 int32 (57 slices to a block, 44 warps to a cell) in 148 us, 169
// with whole blocks dealt out; p = 32, m = 2^23 float32, b = 64 394 and 439.
// A step holds at most two blocks' worth of slices, so that short blocks
// still go up and down the trees as a pipeline of steps.
constexpr int64_t kBlocksPerStep = 2;

CellSlices cell_slices(const Plan* P, const CellPlan& C, bool vec)
{
    const int64_t epu = vec ? 16 / int64_t(P->esize) : 1;
    const int64_t maxblk = (P->m + P->b - 1) / P->b;
    // bounds are rounded up to units, so a block may hold one more
    const int64_t units = std::max<int64_t>(1, (maxblk + epu - 1) / epu + (epu > 1 && P->b > 1 ? 1 : 0));
    const int64_t slices = (units + 31) / 32, all = slices * P->b;
    const int64_t cap = std::min<int64_t>(C.warps / C.n - cell_tail(P, vec), kBlocksPerStep * slices);
    const int64_t steps = (all + cap - 1) / cap;
    return CellSlices{int((all + steps - 1) / steps), int(slices), int(steps)};
}

// Whether a call on aligned buffers moves 16-byte units: not when blocks are
// so short that rounding their bounds to units would change them by much.
bool cell_vector(const Plan* P)
{
    return P->last_vector_path && (P->esize == 16 || P->m / P->b >= 64);
}

int cell_tail(const Plan* P, bool vec) { return vec && P->m % (16 / int64_t(P->esize)) ? 1 : 0; }

// Slots of flagged words per cell and slice, of its partial blocks and of its
// final blocks, in a call of so many steps: a power of two above the deepest
// rank's depth + 1 (schedule_words.cu, reuse of slots), or of at least one
// slot per step.
int word_slots(const Plan* P, int steps)
{
    int n = 1;
    while (n < P->max_depth + 2 && n < steps) n *= 2;
    return n;
}

// The cells' device memory: control words (epoch 1 first), descriptors at 256,
// scratch (zeroed) at off_scratch.
int cell_scratch(Plan* P, CellPlan* C, const void* desc, size_t desc_bytes)
{
    const size_t bytes = C->off_scratch + C->scratch;
    cudaError_t e;
    if (bytes > C->bytes) {
        if (C->d) cudaFree(C->d);
        C->d = nullptr;
        C->bytes = 0;
        e = cudaMalloc(&C->d, bytes);
        if (e != cudaSuccess) {
            C->d = nullptr;
            return cuda_fail(e, "schedule cells: cudaMalloc");
        }
        C->bytes = bytes;
    }
    e = cudaMemset(C->d, 0, 256);
    if (e == cudaSuccess) e = cudaMemset(C->d, 1, 1);  // the epoch's low byte
    if (e == cudaSuccess) e = cudaMemset(C->d + C->off_scratch, 0, C->scratch);
    if (e == cudaSuccess) e = cudaMemcpy(C->d + 256, desc, desc_bytes, cudaMemcpyHostToDevice);
    return e == cudaSuccess ? DPDR_OK : cuda_fail(e, "schedule cells: upload");
}

int cell_launch(const void* kernel, void* args, int64_t warps, int per_cta, size_t smem, cudaStream_t s)
{
    void* argv[] = {args};
    const cudaError_t e = cudaLaunchCooperativeKernel(
        kernel, dim3(unsigned((warps + per_cta - 1) / per_cta)), dim3(unsigned(32 * per_cta)), argv, smem, s);
    if (e == cudaErrorCooperativeLaunchTooLarge) {
        cudaGetLastError();
        return fail(DPDR_ERR_NOT_COOPERATIVE, "schedule kernel: CTAs cannot be co-resident");
    }
    return e == cudaSuccess ? DPDR_OK : cuda_fail(e, "schedule kernel launch");
}

// The cells take over where nothing asks for another layout.
static bool all_automatic(const Plan* P)
{
    return !P->sched_transport && !P->sched_layout && !P->sched_copy && !P->sched_slices &&
           !P->sched_rpc && !P->sched_threads;
}

int schedule_cells_prepare(Plan* P)
{
    P->words.ready = P->walk.ready = false;
    if (P->m == 0 || !all_automatic(P)) return DPDR_OK;
    const bool words = schedule_transport(P) == 2;
    int rc = words ? schedule_words_prepare(P) : DPDR_OK;
    if (rc == DPDR_OK && (!words || P->topo == DPDR_TOPO_SINGLE)) rc = schedule_walk_prepare(P);
    return rc;
}

// The cells that dpdr_allreduce_schedule (algo 0) or
// dpdr_allreduce_reduce_bcast (1) runs on, null when it does not.
const CellPlan* schedule_cells(const Plan* P, int algo)
{
    const CellPlan* C = algo == 0 && schedule_transport(P) == 2 ? &P->words : &P->walk;
    return C->ready && all_automatic(P) ? C : nullptr;
}

}  // namespace dpdr
