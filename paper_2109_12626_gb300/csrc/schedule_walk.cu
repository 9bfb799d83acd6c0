// schedule_walk.cu -- Algorithm 1 on large blocks: instantiations, scratch
// and launches of the walk kernels (schedule_walk.cuh); the reduction, then
// broadcast, is instantiated in schedule_walk_rb.cu.
#include "schedule_walk.cuh"

namespace dpdr {

const void* walk_reduce_bcast_kernel(int dtype, bool vec);  // schedule_walk_rb.cu

namespace {

const void* kernel(int dtype, bool vec, int algo)
{
    return algo ? walk_reduce_bcast_kernel(dtype, vec) : walk::kernel_for<false>(dtype, vec);
}

constexpr int kMaxWarpsPerSm = 64;

}  // namespace

int schedule_walk_prepare(Plan* P)
{
    CellPlan& C = P->walk;
    C.ready = false;
    // Cells of at most 16 ranks, and of up to 20 where that takes a whole tree
    // (p = 36: two cells of 18 ranks; 2x2 matrices, m = 2^20, took 1.3 times
    // as long with six cells; with larger trees 20 ranks make the longest walk
    // longer: p = 1152, m = 2^16 int32 15 % slower).
    const int tree = P->r0 >= 0 ? P->p - P->p / 2 : P->p;
    std::vector<CellDesc> desc;
    if (P->max_depth + 1 >= walk::kPast) return DPDR_OK;
    if (!make_cells(P, tree <= walk::kRanks ? walk::kRanks : 16, walk::kLevels,
                    kMaxWarpsPerSm * P->num_sms / 2, &C, &desc))
        return DPDR_OK;
    int occ = 1 << 20;
    for (int algo = 0; algo < (P->topo == DPDR_TOPO_SINGLE ? 2 : 1); algo++)
        for (bool vec : {false, true}) {
            int o = 0, granted = 48 * 1024;
            const void* const k = kernel(P->dtype, vec, algo);
            const size_t smem = walk::smem_for(C.ranks);
            if (int rc = fused::grant_smem(k, smem, &granted, "schedule walk attribute")) return rc;
            const cudaError_t e =
                cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o, k, walk::kWarps * 32, smem);
            if (e != cudaSuccess) return cuda_fail(e, "schedule walk: occupancy");
            occ = std::min(occ, o);
        }
    C.warps = occ * P->num_sms * walk::kWarps;
    if (2 * C.n > C.warps) return DPDR_OK;  // a slice and the tail do not fit
    const int lines = 1 + std::max(cell_slices(P, C, false).n, cell_slices(P, C, true).n);
    const size_t counters = sizeof(uint32_t) * walk::kCtr * 2 * size_t(C.n) * lines;
    C.off_scratch = 256 + (sizeof(CellDesc) * desc.size() + 255) / 256 * 256;
    C.scratch = counters + size_t(lines) * 4 * 512;
    const int rc = cell_scratch(P, &C, desc.data(), sizeof(CellDesc) * desc.size());
    C.ready = rc == DPDR_OK;
    return rc;
}

int schedule_walk_launch(Plan* P, cudaStream_t s, int algo)
{
    const CellPlan& C = P->walk;
    const bool vec = cell_vector(P);
    walk::WalkArgs a;
    a.x = P->d_x;
    a.y = P->d_y;
    a.cells = reinterpret_cast<const CellDesc*>(C.d + 256);
    a.ctl = reinterpret_cast<uint32_t*>(C.d);
    a.err = P->d_err;
    const CellSlices S = cell_slices(P, C, vec);
    a.col = cells::Columns{P->m, P->m / P->b, P->m % P->b, P->b, S.n, S.per_block, S.steps, cell_tail(P, vec)};
    const int64_t warps = int64_t(C.n) * (S.n + a.col.tail);
    // counters of all geometries share one array, so that clearing it once
    // clears what another geometry left; the exchange slots lie behind it
    const int64_t lines = int64_t(C.scratch / (walk::kCtr * 8 * size_t(C.n) + 4 * 512));
    a.ctr_words = lines * C.n * 2 * walk::kCtr;
    a.up = reinterpret_cast<uint32_t*>(C.d + C.off_scratch);
    a.done = a.up + lines * C.n * walk::kCtr;
    a.ring = reinterpret_cast<char*>(a.up + a.ctr_words);
    a.wait_ns = P->wait_ns;
    a.ncells = C.n;
    a.root0 = C.root0;
    a.root1 = C.root1;
    a.ranks = C.ranks;
    a.used = S.steps + P->max_depth + 2;
    a.skip_rank = P->skip_rank;
    return cell_launch(kernel(P->dtype, vec, algo), &a, warps, walk::kWarps,
                       walk::smem_for(C.ranks), s);
}

}  // namespace dpdr
