// Neighbour pipeline (paper Section 2.3 and Section 4):
//   cell hash -> counting sort by cell (histogram, exclusive scan, scatter)
//   -> in-cell order by (type, id) + reorder of the particle arrays
//   -> cell start/end table (the scan itself) -> split neighbour list.
//
// Deterministic: the histogram counts are order-free, the in-cell rank is a
// comparison count on the unique key (type, id), so the sorted arrays are
// bit-identical from run to run whatever order the atomics took.
#include <algorithm>

#include "pipeline.cuh"

namespace sphg {

namespace {

// kernels of the pipeline bodies (pipeline.cuh); a skin list gates them with
// status->rebuild (no rebuild this step: every kernel exits at once)
__global__ void __launch_bounds__(kPipeBlock) k_hash(const float4* __restrict__ pos, const uint32_t* __restrict__ cell,
                                                     const uint32_t* __restrict__ pinfo,
                                                     const SceneDev* __restrict__ scenes,
                                                     const DevStatus* __restrict__ st, uint32_t* __restrict__ key,
                                                     uint32_t* __restrict__ slot, uint32_t* __restrict__ count,
                                                     uint32_t sentinel, const uint32_t* __restrict__ gate) {
    if (gate && *gate == 0u) return;
    hash_body(pos, cell, pinfo, scenes, st, key, slot, count, sentinel);
}

__global__ void __launch_bounds__(kScanThreads) k_scan_reduce(const uint32_t* __restrict__ count, uint32_t nb,
                                                              uint32_t* __restrict__ bsum,
                                                              const uint32_t* __restrict__ gate) {
    if (gate && *gate == 0u) return;
    scan_reduce_tile(count, nb, bsum, blockIdx.x);
}

// block 1, where launched: the step's time-step update (nothing of the pipeline reads it)
__global__ void __launch_bounds__(1024) k_scan_bsums(uint32_t* __restrict__ bsum, uint32_t nblocks, const DtArgs dt,
                                                     const uint32_t* __restrict__ gate) {
    if (blockIdx.x == 1) {
        dt_body(dt);
        return;
    }
    if (gate && *gate == 0u) return;
    scan_bsums_body(bsum, nblocks);
}

__global__ void __launch_bounds__(1024, 1) k_scan_one(uint32_t* __restrict__ count, uint32_t nb,
                                                   uint32_t* __restrict__ start, DevStatus* __restrict__ st,
                                                   const DtArgs dt, const uint32_t* __restrict__ gate) {
    if (blockIdx.x == 1) {
        dt_body(dt);
        return;
    }
    if (gate && *gate == 0u) return;
    scan_one_body(count, nb, start, st);
}

__global__ void __launch_bounds__(kScanThreads) k_scan_down(uint32_t* __restrict__ count, uint32_t nb,
                                                            const uint32_t* __restrict__ bsum,
                                                            uint32_t* __restrict__ start,
                                                            DevStatus* __restrict__ st,
                                                            const uint32_t* __restrict__ gate) {
    if (gate && *gate == 0u) return;
    scan_down_tile(count, nb, bsum, start, st, blockIdx.x);
}

__global__ void __launch_bounds__(kPipeBlock) k_scatter(const uint32_t* __restrict__ key,
                                                        const uint32_t* __restrict__ slot,
                                                        const uint32_t* __restrict__ start,
                                                        const DevStatus* __restrict__ st,
                                                        uint32_t* __restrict__ unsorted, uint32_t nkeys,
                                                        const uint32_t* __restrict__ gate) {
    if (gate && *gate == 0u) return;
    scatter_body(key, slot, start, st, unsorted, nkeys);
}

template <int kCells, bool kCopy>
__global__ void __launch_bounds__(kPipeBlock) k_reorder(
    const float4* __restrict__ pos, const float4* __restrict__ vel, const float* __restrict__ phat,
    const uint32_t* __restrict__ pinfo, const uint32_t* __restrict__ pid, const uint32_t* __restrict__ start,
    const uint32_t* __restrict__ unsorted, const SceneDev* __restrict__ scenes, uint32_t n_cells,
    DevStatus* __restrict__ st, uint32_t* __restrict__ cell_nfluid, float4* __restrict__ pos_o,
    float4* __restrict__ vel_o, float* __restrict__ phat_o, uint32_t* __restrict__ cell_o,
    uint32_t* __restrict__ pinfo_o, uint32_t* __restrict__ pid_o, float* __restrict__ quads, const SortedCopy copy,
    const uint32_t* __restrict__ gate) {
    if (gate && *gate == 0u) return;
    reorder_body<kCells, kCopy>(pos, vel, phat, pinfo, pid, start, unsorted, scenes, n_cells, st, cell_nfluid, pos_o, vel_o,
                                phat_o, cell_o, pinfo_o, pid_o, quads, copy);
}

// 1024 resident threads per SM (64 registers, a 24-byte spill); 1280 threads at 48 registers were
// slower (1.65M dam break 466 -> 511 us)
template <int kBlockT>
__global__ void __launch_bounds__(kBlockT, 1024 / kBlockT) k_build_tpp(
    const float4* __restrict__ pos, const float* __restrict__ quads, const uint32_t* __restrict__ cell, const uint32_t* __restrict__ pinfo,
    const uint32_t* __restrict__ start, const uint32_t* __restrict__ cell_nfluid, const SceneDev* __restrict__ scenes,
    DevStatus* __restrict__ st, uint32_t* __restrict__ nlist, uint32_t* __restrict__ ncount, float R2,
    uint32_t max_neibs, uint32_t stride, const uint32_t* __restrict__ gate) {
    if (gate && *gate == 0u) return;
    build_tpp_body(pos, quads, cell, pinfo, start, cell_nfluid, scenes, st, nlist, ncount, R2, max_neibs, stride);
}

// the same list by nine warps per 32 particles (build_rows_body)
template <int kMinBlocks>
__global__ void __launch_bounds__(kRowBlock, kMinBlocks) k_build_rows(
    const float4* __restrict__ pos, const float* __restrict__ quads, const uint32_t* __restrict__ cell,
    const uint32_t* __restrict__ pinfo, const uint32_t* __restrict__ start, const uint32_t* __restrict__ cell_nfluid,
    const SceneDev* __restrict__ scenes, DevStatus* __restrict__ st, uint32_t* __restrict__ nlist,
    uint32_t* __restrict__ ncount, float R2, uint32_t max_neibs, uint32_t stride, const uint32_t* __restrict__ gate) {
    if (gate && *gate == 0u) return;
    build_rows_body(pos, quads, cell, pinfo, start, cell_nfluid, scenes, st, nlist, ncount, R2, max_neibs, stride);
}

inline unsigned grid_for(uint64_t n, int block) {
    const uint64_t g = (n + block - 1) / block;
    return g ? (unsigned)g : 1u;
}

}  // namespace

uint32_t scan_blocks(uint32_t n_buckets) { return (n_buckets + kScanTile - 1) / kScanTile; }

void launch_hash(const Buffers& b, int cur, const Geometry& g, cudaStream_t st) {
    k_hash<<<grid_for(g.cap, kPipeBlock), kPipeBlock, 0, st>>>(b.pos[cur], b.cell[cur], b.pinfo[cur], b.scenes, b.status,
                                                        b.key, b.slot, b.count, g.n_cells, b.gate);
}

// One block scans few buckets (217 buckets 8.6 -> 3.9 us, with the time-step kernel's 2 us saved
// besides; 4,117 buckets 11.1 -> 6.4 us); more take three kernels.
void launch_scan(const Buffers& b, const Geometry& g, const DtArgs* dt, cudaStream_t st) {
    const uint32_t nb = g.n_cells + 1;
    const DtArgs none{};
    if (nb <= kScanOneMax) {
        k_scan_one<<<dt ? 2 : 1, 1024, 0, st>>>(b.count, nb, b.start, b.status, dt ? *dt : none, b.gate);
        return;
    }
    const uint32_t blocks = scan_blocks(nb);
    k_scan_reduce<<<blocks, kScanThreads, 0, st>>>(b.count, nb, b.bsum, b.gate);
    k_scan_bsums<<<dt ? 2 : 1, 1024, 0, st>>>(b.bsum, blocks, dt ? *dt : none, b.gate);
    k_scan_down<<<blocks, kScanThreads, 0, st>>>(b.count, nb, b.bsum, b.start, b.status, b.gate);
}

void launch_scatter(const Buffers& b, const Geometry& g, cudaStream_t st) {
    k_scatter<<<grid_for(g.cap, kPipeBlock), kPipeBlock, 0, st>>>(b.key, b.slot, b.start, b.status, b.unsorted,
                                                           g.n_cells + 1, b.gate);
}

template <int kCells, bool kCopy>
void launch_reorder_c(const Buffers& b, int cur, const Geometry& g, const SortedCopy& copy, cudaStream_t st) {
    const int nxt = cur ^ 1;
    const uint32_t warps = (g.n_cells + kCells - 1) / kCells;
    k_reorder<kCells, kCopy><<<grid_for(warps, kPipeBlock / 32), kPipeBlock, 0, st>>>(
        b.pos[cur], b.vel[cur], b.phat[cur], b.pinfo[cur], b.pid[cur], b.start, b.unsorted, b.scenes, g.n_cells, b.status,
        b.cell_nfluid, b.pos[nxt], b.vel[nxt], b.phat[nxt], b.cell[nxt], b.pinfo[nxt], b.pid[nxt], b.quads, copy, b.gate);
}

void launch_reorder(const Buffers& b, int cur, const Geometry& g, cudaStream_t st, const SortedCopy* copy) {
    const bool one = g.n_cells <= kReorderOneMax;
    if (copy) {
        if (one) launch_reorder_c<1, true>(b, cur, g, *copy, st);
        else launch_reorder_c<kReorderCells, true>(b, cur, g, *copy, st);
    } else if (one) {
        launch_reorder_c<1, false>(b, cur, g, SortedCopy(), st);
    } else {
        launch_reorder_c<kReorderCells, false>(b, cur, g, SortedCopy(), st);
    }
}

template <int B>
void launch_build_tpp(const Buffers& b, int cur, const Geometry& g, const Phys& ph, cudaStream_t st) {
    k_build_tpp<B><<<grid_for(g.cap, B), B, 0, st>>>(b.pos[cur], b.quads, b.cell[cur], b.pinfo[cur], b.start, b.cell_nfluid,
                                                     b.scenes, b.status, b.nlist, b.ncount, ph.R2_list, ph.max_neibs,
                                                     ph.stride, b.gate);
}

template <int MB>
void launch_build_rows(const Buffers& b, int cur, const Geometry& g, const Phys& ph, cudaStream_t st) {
    const size_t smem = ph.max_neibs <= kStageNeibs ? sizeof(uint32_t) * rows_smem_words(ph.max_neibs) : 0;
    // resident blocks at most: a block then takes several tiles in turn
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms <= 0)
        sms = 1;
    const unsigned grid = std::min(grid_for(g.cap, 32), (unsigned)sms * MB);
    k_build_rows<MB><<<grid, kRowBlock, smem, st>>>(b.pos[cur], b.quads, b.cell[cur], b.pinfo[cur], b.start, b.cell_nfluid,
                                                   b.scenes, b.status, b.nlist, b.ncount, ph.R2_list, ph.max_neibs,
                                                   ph.stride, b.gate);
}

const char* build_variant_name(int v) {
    static const char* names[kBuildVariants] = {"thread/particle x128", "thread/particle x256", "warp/row x2 blocks/SM",
                                                "warp/row x3 blocks/SM", "warp/row x4 blocks/SM"};
    return v >= 0 && v < kBuildVariants ? names[v] : "?";
}

// skin list: the reorder wrote the sorted arrays to the other buffer; copy
// them back (the step graph keeps one buffer) and record the offsets at the
// build for the displacement check.
__global__ void k_copyback(const float4* __restrict__ pos, const float4* __restrict__ vel,
                           const float* __restrict__ phat, const uint32_t* __restrict__ cell,
                           const uint32_t* __restrict__ pinfo, const uint32_t* __restrict__ pid,
                           const DevStatus* __restrict__ st, float4* __restrict__ pos_o, float4* __restrict__ vel_o,
                           float* __restrict__ phat_o, uint32_t* __restrict__ cell_o, uint32_t* __restrict__ pinfo_o,
                           uint32_t* __restrict__ pid_o, float4* __restrict__ pos_ref,
                           const uint32_t* __restrict__ gate) {
    if (gate && *gate == 0u) return;
    const uint32_t n = st->n_active;
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const float4 p = pos[i];
        pos_o[i] = p;
        pos_ref[i] = p;
        vel_o[i] = vel[i];
        phat_o[i] = phat[i];
        cell_o[i] = cell[i];
        pinfo_o[i] = pinfo[i];
        pid_o[i] = pid[i];
    }
}

__global__ void k_force_rebuild(DevStatus* st) {
    st->rebuild = 1u;
    st->since = 0u;  // steps taken with the list built now
    st->maxdisp2_bits = 0u;
    st->builds += 1u;
}

void launch_copyback(const Buffers& b, int cur, const Geometry& g, cudaStream_t st) {
    const int alt = cur ^ 1;
    k_copyback<<<grid_for(g.cap, kPipeBlock), kPipeBlock, 0, st>>>(b.pos[alt], b.vel[alt], b.phat[alt], b.cell[alt],
                                                            b.pinfo[alt], b.pid[alt], b.status, b.pos[cur],
                                                            b.vel[cur], b.phat[cur], b.cell[cur], b.pinfo[cur],
                                                            b.pid[cur], b.pos_ref, b.gate);
}

void launch_force_rebuild(const Buffers& b, cudaStream_t st) { k_force_rebuild<<<1, 1, 0, st>>>(b.status); }

void launch_build(const Buffers& b, int cur, const Geometry& g, const Phys& ph, cudaStream_t st) {
    switch (ph.build_variant) {
        case 0: launch_build_tpp<128>(b, cur, g, ph, st); break;
        case 1: launch_build_tpp<256>(b, cur, g, ph, st); break;
        case 2: launch_build_rows<2>(b, cur, g, ph, st); break;
        case 3: launch_build_rows<3>(b, cur, g, ph, st); break;
        default: launch_build_rows<4>(b, cur, g, ph, st); break;
    }
}

}  // namespace sphg
