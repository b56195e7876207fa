// Bodies of the neighbour-pipeline kernels (paper Section 2.3 and Section 4):
// cell hash, counting sort (histogram, scan, scatter), in-cell order and
// reorder, thread-per-particle list build.  Each body is a device function of
// the threads of one launch; neighbors.cu wraps each in its own kernel, and the
// persistent step kernel (forces.cu) runs them one after the other with grid-wide
// barriers between them.  Grid-stride loops: any grid size computes the same.
#pragma once
#include "packed.cuh"
#include "sph_internal.cuh"

namespace sphg {

namespace {

constexpr int kPipeBlock = 256;   // threads per block of the pipeline kernels
constexpr int kScanThreads = 256;
constexpr int kScanItems = 8;                       // per thread
constexpr int kScanTile = kScanThreads * kScanItems;  // buckets per block

// ---------------------------------------------------------------------
// dt.  The CFL time step of a scene from the largest |a|^2 of the last reduction (reading C7)
__device__ __forceinline__ double cfl_dt_of(const SceneDev& sc, const SceneDyn& d, double h, double cfl,
                                            double dt_fixed) {
    if (dt_fixed > 0.0) return dt_fixed;
    double dt = sc.dt_cap;
    const double a2 = (double)__uint_as_float(d.amax2_bits);
    if (a2 > 0.0) dt = fmin(dt, cfl * sqrt(h / sqrt(a2)));
    return dt;
}

// One block, a thread per scene: dt for the coming step (reading C7), simulated
// time, reset of the |a|^2 accumulator.
__device__ __forceinline__ void dt_body(const DtArgs& a) {
    const SceneDev* __restrict__ scenes = a.scenes;
    SceneDyn* __restrict__ dyn = a.dyn;
    DevStatus* __restrict__ st = a.st;
    const double dt_host = st->dt_next;  // the host's time step for this step (sph_set_dt), or <= 0
    __syncthreads();
    for (uint32_t s = threadIdx.x; s < a.n_scenes; s += blockDim.x) {
        const double dt = dt_host > 0.0 ? dt_host : cfl_dt_of(scenes[s], dyn[s], a.h, a.cfl, a.dt_fixed);
        dyn[s].dt = (float)dt;
        dyn[s].dt_d = dt;
        if (a.advance) dyn[s].time += dt;
        dyn[s].amax2_bits = 0u;
    }
    if (threadIdx.x == 0 && dt_host > 0.0) st->dt_next = 0.0;
    if (threadIdx.x == 0 && a.advance) {
        st->steps += 1ull;
        if (a.rebuild_every > 1) {
            // skin list: rebuild when a particle has moved skin/4 (the predicted state of
            // the step then stays within skin/2: a CFL step moves less than 0.3 h) or after
            // a.rebuild_every steps
            const bool rb = st->since >= a.rebuild_every || __uint_as_float(st->maxdisp2_bits) > a.trig2;
            st->rebuild = rb ? 1u : 0u;
            st->since = rb ? 1u : st->since + 1u;
            if (rb) st->maxdisp2_bits = 0u;
            st->builds += rb ? 1u : 0u;
        } else {
            st->builds += a.builds_inc;
        }
    }
}

// ---------------------------------------------------------------------
// a1: cell hash.  New cell = old cell + floor(offset/cell + 1/2) per axis
// (cell-relative positions never leave FP32 range); periodic axes wrap;
// on other axes a particle outside the grid goes to the sentinel bucket
// (removed during the sort, paper "The GPU in GPUSPH").
// ---------------------------------------------------------------------
__device__ __forceinline__ void hash_body(const float4* __restrict__ pos, const uint32_t* __restrict__ cell,
                                          const uint32_t* __restrict__ pinfo, const SceneDev* __restrict__ scenes,
                                          const DevStatus* __restrict__ st, uint32_t* __restrict__ key,
                                          uint32_t* __restrict__ slot, uint32_t* __restrict__ count, uint32_t sentinel) {
    const uint32_t n = st->n_active;
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const SceneDev& sc = scenes[pinfo[i]];
        const float4 p = pos[i];
        const uint32_t c = cell[i];
        const int sx = cell_shift(p.x, sc.cell_f[0], sc.inv_cell_f[0]);
        const int sy = cell_shift(p.y, sc.cell_f[1], sc.inv_cell_f[1]);
        const int sz = cell_shift(p.z, sc.cell_f[2], sc.inv_cell_f[2]);
        uint32_t k = c;
        if ((sx | sy | sz) != 0) {
            int cx, cy, cz;
            decode_local(c - sc.cell_offset, sc, cx, cy, cz);
            int nc[3] = {cx + sx, cy + sy, cz + sz};
            bool out = false;
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                const int n_a = sc.ncell[a];
                if ((sc.periodic >> a) & 1u) {
                    nc[a] %= n_a;
                    if (nc[a] < 0) nc[a] += n_a;
                } else if (nc[a] < 0 || nc[a] >= n_a) {
                    out = true;
                }
            }
            k = out ? sentinel
                    : sc.cell_offset + (uint32_t)nc[0] +
                          (uint32_t)sc.ncell[0] * ((uint32_t)nc[1] + (uint32_t)sc.ncell[1] * (uint32_t)nc[2]);
        }
        key[i] = k;
        // one atomic per distinct cell of the warp (consecutive particles mostly share
        // one): the leader reserves the slots of its peers, each takes base + its rank.
        // The order within a cell is the reorder's to fix, so any slot order will do.
        const unsigned act = __activemask();
        const unsigned peers = __match_any_sync(act, k);
        const int lane = threadIdx.x & 31;
        const int leader = __ffs(peers) - 1;
        uint32_t base = 0;
        if (lane == leader) base = atomicAdd(&count[k], (uint32_t)__popc(peers));
        base = __shfl_sync(peers, base, leader);
        slot[i] = base + (uint32_t)__popc(peers & ((1u << lane) - 1u));
    }
}

// ---------------------------------------------------------------------
// a2/a4: exclusive scan of the bucket counts -> cell start table.
// Three passes: block sums, scan of block sums, down-sweep.  The down-sweep
// zeroes the counts for the next hash and publishes the in-domain count.
// ---------------------------------------------------------------------
__device__ __forceinline__ uint32_t warp_incl_scan(uint32_t v) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += t;
    }
    return v;
}

// block-wide exclusive scan of one value per thread; returns the block total in *total
__device__ __forceinline__ uint32_t block_excl_scan(uint32_t v, uint32_t* total) {
    __shared__ uint32_t wsum[32];
    __shared__ uint32_t wtotal;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const uint32_t inc = warp_incl_scan(v);
    if (lane == 31) wsum[w] = inc;
    __syncthreads();
    if (w == 0) {
        const int nw = blockDim.x >> 5;
        const uint32_t s = lane < nw ? wsum[lane] : 0u;
        const uint32_t si = warp_incl_scan(s);
        if (lane < nw) wsum[lane] = si - s;
        if (lane == nw - 1) wtotal = si;
    }
    __syncthreads();
    const uint32_t res = wsum[w] + inc - v;
    *total = wtotal;
    __syncthreads();
    return res;
}

// A thread's kScanItems consecutive counts, zero past the last bucket: in 16-byte loads (the tables and
// the thread's first bucket are aligned), but for the thread that holds the table's end.  A load and two
// stores of 4 bytes per bucket, 32 bytes apart over a warp, took three kernels 20.3 us on the 1.65M dam
// break (536,257 buckets; now 16.6) and 85 us on 20.1M (now 36), the one-block scan of 4,117 buckets
// 10.4 us (now 7.5).
__device__ __forceinline__ void scan_load(const uint32_t* __restrict__ count, uint32_t nb, uint32_t base, uint32_t* v) {
    static_assert(kScanItems == 8, "two 16-byte words");
    if (base < nb && nb - base >= (uint32_t)kScanItems) {
        const uint4 a = *reinterpret_cast<const uint4*>(count + base), b = *reinterpret_cast<const uint4*>(count + base + 4);
        v[0] = a.x, v[1] = a.y, v[2] = a.z, v[3] = a.w;
        v[4] = b.x, v[5] = b.y, v[6] = b.z, v[7] = b.w;
    } else {
#pragma unroll
        for (int k = 0; k < kScanItems; ++k) v[k] = base < nb && (uint32_t)k < nb - base ? count[base + k] : 0u;
    }
}

// the starts of those buckets, from the first one's; their counts zeroed; the thread that holds the
// last bucket, the sentinel of removed particles, publishes the particle counts
__device__ __forceinline__ void scan_store(uint32_t* __restrict__ count, uint32_t nb, uint32_t* __restrict__ start,
                                           DevStatus* __restrict__ st, uint32_t base, uint32_t run, const uint32_t* v) {
    if (base >= nb) return;
    const uint32_t left = nb - base;
    uint32_t o[kScanItems];
#pragma unroll
    for (int k = 0; k < kScanItems; ++k) {
        o[k] = run;
        run += v[k];
    }
    if (left >= (uint32_t)kScanItems) {
        *reinterpret_cast<uint4*>(start + base) = make_uint4(o[0], o[1], o[2], o[3]);
        *reinterpret_cast<uint4*>(start + base + 4) = make_uint4(o[4], o[5], o[6], o[7]);
        *reinterpret_cast<uint4*>(count + base) = make_uint4(0u, 0u, 0u, 0u);
        *reinterpret_cast<uint4*>(count + base + 4) = make_uint4(0u, 0u, 0u, 0u);
    }
#pragma unroll
    for (int k = 0; k < kScanItems; ++k) {
        if (left < (uint32_t)kScanItems && (uint32_t)k < left) {
            start[base + k] = o[k];
            count[base + k] = 0u;
        }
        if ((uint32_t)k + 1u == left) {
            start[nb] = o[k] + v[k];
            st->n_sorted = o[k];
            st->n_removed += v[k];
        }
    }
}

__device__ __forceinline__ void scan_reduce_tile(const uint32_t* __restrict__ count, uint32_t nb,
                                                 uint32_t* __restrict__ bsum, uint32_t tile) {
    const uint32_t base = tile * kScanTile + threadIdx.x * kScanItems;
    uint32_t v[kScanItems];
    scan_load(count, nb, base, v);
    uint32_t s = 0;
#pragma unroll
    for (int k = 0; k < kScanItems; ++k) s += v[k];
    uint32_t total;
    block_excl_scan(s, &total);
    if (threadIdx.x == 0) bsum[tile] = total;
}

__device__ __forceinline__ void scan_bsums_body(uint32_t* __restrict__ bsum, uint32_t nblocks) {

    uint32_t carry = 0;
    for (uint32_t base = 0; base < nblocks; base += blockDim.x) {
        const uint32_t i = base + threadIdx.x;
        const uint32_t v = i < nblocks ? bsum[i] : 0u;
        uint32_t total;
        const uint32_t ex = block_excl_scan(v, &total);
        if (i < nblocks) bsum[i] = carry + ex;
        carry += total;
    }
}

__device__ __forceinline__ void scan_down_tile(uint32_t* __restrict__ count, uint32_t nb,
                                               const uint32_t* __restrict__ bsum, uint32_t* __restrict__ start,
                                               DevStatus* __restrict__ st, uint32_t tile) {
    const uint32_t base = tile * kScanTile + threadIdx.x * kScanItems;
    uint32_t v[kScanItems];
    scan_load(count, nb, base, v);
    uint32_t s = 0;
#pragma unroll
    for (int k = 0; k < kScanItems; ++k) s += v[k];
    uint32_t total;
    const uint32_t run = block_excl_scan(s, &total) + bsum[tile];
    scan_store(count, nb, start, st, base, run, v);
}

// the whole scan by one block of 1024 threads, for few buckets
constexpr uint32_t kScanOneMax = 24576;

__device__ __forceinline__ void scan_one_body(uint32_t* __restrict__ count, uint32_t nb, uint32_t* __restrict__ start,
                                              DevStatus* __restrict__ st) {
    uint32_t carry = 0;
    for (uint32_t base0 = 0; base0 < nb; base0 += blockDim.x * kScanItems) {
        const uint32_t base = base0 + threadIdx.x * kScanItems;
        uint32_t v[kScanItems];
        scan_load(count, nb, base, v);
        uint32_t s = 0;
#pragma unroll
        for (int k = 0; k < kScanItems; ++k) s += v[k];
        uint32_t total;
        const uint32_t run = block_excl_scan(s, &total) + carry;
        carry += total;
        scan_store(count, nb, start, st, base, run, v);
    }
}

// ---------------------------------------------------------------------
// a2: scatter particle indices to their bucket slots (order within a
// bucket is the atomics' order; the reorder fixes it).
// ---------------------------------------------------------------------
__device__ __forceinline__ void scatter_body(const uint32_t* __restrict__ key, const uint32_t* __restrict__ slot,
                                             const uint32_t* __restrict__ start, const DevStatus* __restrict__ st,
                                             uint32_t* __restrict__ unsorted, uint32_t nkeys) {
    const uint32_t n = st->n_active;
    (void)nkeys;
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        SPH_GUARD(key[i] < nkeys && start[key[i]] + slot[i] < start[key[i] + 1], st, continue)
        unsorted[start[key[i]] + slot[i]] = i;
    }
}

// ---------------------------------------------------------------------
// a3: one warp per cell (a warp takes kReorderCells consecutive cells in turn).
// Rank each particle of the cell by its unique key (type, id) -> final slot; gather its data from the old arrays, re-base
// the offset to the new cell (exact: Sterbenz), write the new arrays.
// ---------------------------------------------------------------------
// (type, id) in 32 bits (ids < kMaxParticles = 2^26): one shuffle per comparison of the rank
static_assert(kMaxParticles <= (1u << 31), "the id fits below the type bit");
__device__ __forceinline__ uint32_t sort_key(float mass, uint32_t id) {
    return (__float_as_uint(mass) & 0x80000000u) | id;  // sign bit = boundary
}

// cells per warp: 4 measured fastest on large grids (1.65M dam break, most cells empty: 78 -> 61 us;
// 2.1M box, no empty cell: unchanged at 56 us; 8 and 16 cells per warp leave too few warps; a cell's
// gathers issued together, before its rank is counted: 66 -> 57 us); 1 on
// grids of up to kReorderOneMax cells, whose warps are too few to hide a cell's chain of loads (216
// cells 8.6 -> 2.5 us, 4,116 cells 8.6 -> 4.5 us)
constexpr int kReorderCells = 4;
static_assert(kReorderCells >= 1 && kReorderCells <= 32, "one lane per cell");
constexpr uint32_t kReorderOneMax = 32768;

// kCopy: the sorted state is also written to `copy` (a step of the backward pass' tape)
template <int kCells, bool kCopy = false>
__device__ __forceinline__ void reorder_body(
    const float4* __restrict__ pos, const float4* __restrict__ vel, const float* __restrict__ phat,
    const uint32_t* __restrict__ pinfo,
    const uint32_t* __restrict__ pid, const uint32_t* __restrict__ start, const uint32_t* __restrict__ unsorted,
    const SceneDev* __restrict__ scenes, uint32_t n_cells, DevStatus* __restrict__ st, uint32_t* __restrict__ cell_nfluid,
    float4* __restrict__ pos_o,
    float4* __restrict__ vel_o, float* __restrict__ phat_o, uint32_t* __restrict__ cell_o,
    uint32_t* __restrict__ pinfo_o, uint32_t* __restrict__ pid_o, float* __restrict__ quads,
    const SortedCopy& copy = SortedCopy()) {
    const int lane = threadIdx.x & 31;
    const uint32_t warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const uint32_t nwarps = (gridDim.x * blockDim.x) >> 5;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        st->n_active = st->n_sorted;
        st->max_neibs_seen = 0u;
    }
    // kCells consecutive cells per warp: their ranges in one load, empty cells
    // (most of a tank's cells) skipped without a round trip each
    for (uint32_t c0 = warp * kCells; c0 < n_cells; c0 += nwarps * kCells) {
        const uint32_t cl = c0 + (uint32_t)lane;
        const bool own = lane < kCells && cl < n_cells;
        const uint32_t b_l = own ? start[cl] : 0u, e_l = own ? start[cl + 1] : 0u;
        if (own && e_l == b_l) cell_nfluid[cl] = 0u;
        unsigned todo = __ballot_sync(0xffffffffu, e_l > b_l);
        while (todo) {
            const int kc = __ffs(todo) - 1;
            todo &= todo - 1u;
            const uint32_t c = c0 + (uint32_t)kc;
            const uint32_t beg = __shfl_sync(0xffffffffu, b_l, kc), end = __shfl_sync(0xffffffffu, e_l, kc);
            const uint32_t n = end - beg;
            uint32_t nfluid = 0;
            for (uint32_t base = 0; base < n; base += 32) {
                const uint32_t l = base + lane;
                uint32_t mine = ~0u;  // above every key
                // everything gathered at once: the loads return while the rank is counted
                float4 p = make_float4(0.f, 0.f, 0.f, 0.f), v = p;
                float h = 0.f;
                uint32_t s = 0, id = 0;
                if (l < n) {
                    const uint32_t idx = unsorted[beg + l];
                    p = pos[idx];
                    id = pid[idx];
                    s = pinfo[idx];
                    v = vel[idx];
                    h = phat[idx];
                    mine = sort_key(p.w, id);
                }
                nfluid += __popc(__ballot_sync(0xffffffffu, l < n && (mine >> 31) == 0u));
                uint32_t rank = 0;
                if (n <= 32) {
                    for (uint32_t k = 0; k < n; ++k) {
                        const uint32_t o = __shfl_sync(0xffffffffu, mine, (int)k);
                        rank += o < mine;
                    }
                } else {
                    for (uint32_t k = 0; k < n; ++k) {
                        const uint32_t j = unsorted[beg + k];
                        const uint32_t o = sort_key(pos[j].w, pid[j]);
                        rank += o < mine;
                    }
                }
                if (l < n) {
                    const SceneDev& sc = scenes[s];
                    cell_shift(p.x, sc.cell_f[0], sc.inv_cell_f[0], &p.x);
                    cell_shift(p.y, sc.cell_f[1], sc.inv_cell_f[1], &p.y);
                    cell_shift(p.z, sc.cell_f[2], sc.inv_cell_f[2], &p.z);
                    const uint32_t d = beg + rank;
                    SPH_GUARD(d < end, st, continue)
                    pos_o[d] = p;
                    float* qd = quads + quad_word(d);
                    qd[0] = p.x;
                    qd[4] = p.y;
                    qd[8] = p.z;
                    vel_o[d] = v;
                    phat_o[d] = h;
                    cell_o[d] = c;
                    pinfo_o[d] = s;
                    pid_o[d] = id;
                    if constexpr (kCopy) {
                        copy.pos[d] = p;
                        copy.vel[d] = v;
                        copy.phat[d] = h;
                        copy.pinfo[d] = s;
                        copy.pid[d] = id;
                    }
                }
            }
            if (lane == 0) cell_nfluid[c] = nfluid;
        }
    }
}

// ---------------------------------------------------------------------
// a5: split neighbour list (paper Section 4), one thread per particle (the paper's baseline
// build, Section 7).  Lanes of a warp are consecutive particles of ~2 cells
// and read the same candidates (L1 broadcast).  Candidates are fluid-first
// in each cell (cell_nfluid), so a boundary particle walks only the fluid
// part of each neighbour cell and types need no per-candidate test.
//
// Bound by instruction issue (64% busy) and the L1 pipe (58%).  Measured, with the offsets
// read as float4 records and tested one by one in FP32 before: 547 -> 463 us on the 1.65M dam
// break (435M -> 368M warp instructions), 757 -> 571 us on 64 tanks of 2.0M particles, 530 -> 438 us
// on a 1.0M box.  The group loop unrolled twice, three or four times: 476, 488, 490 us.  The
// appends take a quarter (354 us with the lists left unwritten).
// ---------------------------------------------------------------------

// m with all but its k highest set bits cleared
__device__ __forceinline__ uint32_t highest_set_bits(uint32_t m, uint32_t k) {
    uint32_t out = 0u;
    for (uint32_t c = 0; c < k && m; ++c) {
        const uint32_t b = 0x80000000u >> __clz((int)m);
        out |= b;
        m ^= b;
    }
    return out;
}

// the entries e0 + (u << kCodeBits) of the set bits of mask, u counted from the top bit, appended
// to w in that order: the first completes a chunk left open, then two per chunk store
__device__ __forceinline__ void append_mask(ListWriter& w, uint32_t mask, uint32_t e0) {
    if (mask && (w.n & 1u)) {
        const uint32_t u = (uint32_t)__clz((int)mask);
        mask ^= 0x80000000u >> u;
        w.put(e0 + (u << kCodeBits));
    }
    while (mask) {
        const uint32_t u0 = (uint32_t)__clz((int)mask);
        mask ^= 0x80000000u >> u0;
        const uint32_t a = e0 + (u0 << kCodeBits);
        if (!mask) {
            w.open(a);
            break;
        }
        const uint32_t u1 = (uint32_t)__clz((int)mask);
        mask ^= 0x80000000u >> u1;
        w.put2(a, e0 + (u1 << kCodeBits));
    }
}

// r^2 + init of two candidates at (dx, dy, dz)
__device__ __forceinline__ f2 r2_plus(f2 dx, f2 dy, f2 dz, f2 init) {
    return f2_fma(dx, dx, f2_fma(dy, dy, f2_fma(dz, dz, init)));
}

// 0 < r2 < R2 as one unsigned compare on the bits, in the top bit
__device__ __forceinline__ uint32_t centre_hit(float r2, uint32_t r2lim) {
    return __float_as_uint(r2) - 1u < r2lim ? 0x80000000u : 0u;
}

// The list of particle i; returns its entry count, *nfound = pairs found
// (more than max_neibs: overflow, the list keeps the first ones).
// Candidates are tested four at a time: one 16-byte load per axis from the offsets' own arrays
// (aligned: a group may begin before the cell's first particle and end after its last, masked
// off), packed FP32 subtractions and FMAs on two candidates each, and the sign bit of r^2 - R^2
// shifted into a hit mask by one funnel shift: 4.75 instructions a candidate.  In the particle's
// own cell r^2 itself is tested, 0 < r^2 < R^2 (the particle, coincident ones).  The hits of a
// window of up to 32 candidates are appended by a loop over the mask's set bits, so a lane's
// append work follows its own hits.  Past max_neibs entries the list keeps the first ones in
// candidate order (the mask is cut to the room left).
__device__ __forceinline__ uint32_t build_particle(uint32_t i, const float4* __restrict__ pos, const float* __restrict__ quads,
                                                   const uint32_t* __restrict__ cell, const uint32_t* __restrict__ pinfo,
                                                   const uint32_t* __restrict__ start,
                                                   const uint32_t* __restrict__ cell_nfluid,
                                                   const SceneDev* __restrict__ scenes, uint32_t* __restrict__ nlist,
                                                   uint32_t* __restrict__ ncount, float R2, uint32_t max_neibs,
                                                   uint32_t stride, uint32_t* nfound_out, DevStatus* st, uint32_t n) {
    const SceneDev& sc = scenes[pinfo[i]];
    const float4 pi = pos[i];
    const bool fluid_i = pi.w > 0.f;
    int cx, cy, cz;
    decode_local(cell[i] - sc.cell_offset, sc, cx, cy, cz);
    const uint32_t r2lim = __float_as_uint(R2) - 1u;
    const f2 mR2 = f2_dup(-R2);
    uint32_t nfound = 0;
    ListWriter wf = list_fluid_writer(nlist, i, stride);
    ListWriter wb = list_bnd_writer(nlist, i, stride, max_neibs);
    for (int dz = -1; dz <= 1; ++dz) {
        int z = cz + dz;
        if (z < 0 || z >= sc.ncell[2]) {
            if (!((sc.periodic >> 2) & 1u)) continue;
            z = z < 0 ? z + sc.ncell[2] : z - sc.ncell[2];
        }
        for (int dy = -1; dy <= 1; ++dy) {
            int y = cy + dy;
            if (y < 0 || y >= sc.ncell[1]) {
                if (!((sc.periodic >> 1) & 1u)) continue;
                y = y < 0 ? y + sc.ncell[1] : y - sc.ncell[1];
            }
            const uint32_t row = sc.cell_offset + (uint32_t)sc.ncell[0] * ((uint32_t)y + (uint32_t)sc.ncell[1] * (uint32_t)z);
            const f2 ny = f2_dup((float)dy * sc.cell_f[1] - pi.y), nz = f2_dup((float)dz * sc.cell_f[2] - pi.z);
            // the row's three cell ranges, loaded together (one round trip per row)
            uint32_t rb[3], ref[3], re[3];
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                int x = cx + k - 1;
                bool ok = true;
                if (x < 0 || x >= sc.ncell[0]) {
                    if (sc.periodic & 1u) x = x < 0 ? x + sc.ncell[0] : x - sc.ncell[0];
                    else ok = false;
                }
                rb[k] = ref[k] = re[k] = 0u;
                if (ok) {
                    const uint32_t cc = row + (uint32_t)x;
                    rb[k] = start[cc];
                    ref[k] = rb[k] + cell_nfluid[cc];  // end of the fluid part
                    re[k] = fluid_i ? start[cc + 1] : ref[k];
                    SPH_GUARD(rb[k] <= ref[k] && ref[k] <= start[cc + 1] && start[cc + 1] <= n, st,
                              rb[k] = ref[k] = re[k] = 0u)
                }
            }
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const int dx = k - 1;
                const f2 nx = f2_dup((float)dx * sc.cell_f[0] - pi.x);
                const uint32_t code = (uint32_t)(dx + 1) | ((uint32_t)(dy + 1) << 2) | ((uint32_t)(dz + 1) << 4);
                const bool centre = dx == 0 && dy == 0 && dz == 0;
                const uint32_t b = rb[k], e = re[k];
                for (uint32_t w0 = b & ~3u; w0 < e; w0 += 32u) {
                    const uint32_t wend = min(e, w0 + 32u);
                    uint32_t mask = 0u;
                    uint32_t g = w0;
                    const ulonglong2* q4 = reinterpret_cast<const ulonglong2*>(quads + quad_word(w0));
                    if (!centre) {
#pragma unroll 1
                        for (; g < wend; g += 4u, q4 += 3) {
                            const ulonglong2 X = q4[0], Y = q4[1], Z = q4[2];
                            const f2 q0 = r2_plus(f2_add(X.x, nx), f2_add(Y.x, ny), f2_add(Z.x, nz), mR2);
                            const f2 q1 = r2_plus(f2_add(X.y, nx), f2_add(Y.y, ny), f2_add(Z.y, nz), mR2);
                            mask = __funnelshift_l((uint32_t)q0, mask, 1);
                            mask = __funnelshift_l((uint32_t)(q0 >> 32), mask, 1);
                            mask = __funnelshift_l((uint32_t)q1, mask, 1);
                            mask = __funnelshift_l((uint32_t)(q1 >> 32), mask, 1);
                        }
                    } else {
                        for (; g < wend; g += 4u, q4 += 3) {
                            const ulonglong2 X = q4[0], Y = q4[1], Z = q4[2];
                            const f2 a0 = r2_plus(f2_add(X.x, nx), f2_add(Y.x, ny), f2_add(Z.x, nz), 0ull);
                            const f2 a1 = r2_plus(f2_add(X.y, nx), f2_add(Y.y, ny), f2_add(Z.y, nz), 0ull);
                            mask = __funnelshift_l(centre_hit(f2_lo(a0), r2lim), mask, 1);
                            mask = __funnelshift_l(centre_hit(f2_hi(a0), r2lim), mask, 1);
                            mask = __funnelshift_l(centre_hit(f2_lo(a1), r2lim), mask, 1);
                            mask = __funnelshift_l(centre_hit(f2_hi(a1), r2lim), mask, 1);
                        }
                    }
                    // the window's first candidate to the top bit, those outside the cell off
                    const uint32_t first = w0 < b ? b - w0 : 0u, last = wend - w0;  // last in 1..32
                    mask = (mask << (32u - (g - w0))) & (0xffffffffu >> first) & (0xffffffffu << (32u - last));
                    if (!mask) continue;
                    const uint32_t found = (uint32_t)__popc(mask);
                    nfound += found;
                    const uint32_t room = max_neibs - (wf.n + wb.n);
                    if (found > room) mask = highest_set_bits(mask, room);
                    const uint32_t e0 = (w0 << kCodeBits) | code;
                    if (ref[k] < wend) {  // fluid candidates come first in the cell
                        const uint32_t nfl = ref[k] > w0 ? ref[k] - w0 : 0u;  // below 32
                        append_mask(wb, mask & (0xffffffffu >> nfl), e0);
                        mask &= ~(0xffffffffu >> nfl);
                    }
                    append_mask(wf, mask, e0);
                }
            }
        }
    }
    wf.flush();
    wb.flush();
    ncount[i] = wf.n | (wb.n << 16);
    *nfound_out = nfound;
    return wf.n + wb.n;
}

// warp-level list statistics: overflow flag, largest count, entries written
__device__ __forceinline__ void build_stats(DevStatus* st, uint32_t nfound, uint32_t nent, uint32_t max_neibs,
                                            unsigned mask) {
    if (nfound > max_neibs) atomicOr(&st->error_bits, SPH_EBIT_NEIB_OVERFLOW);
    const uint32_t m = __reduce_max_sync(mask, nfound);
    const uint32_t wsum = __reduce_add_sync(mask, nent);
    if ((threadIdx.x & 31) == (uint32_t)(__ffs(mask) - 1)) {
        atomicMax(&st->max_neibs_seen, m);
        atomicAdd(&st->list_entries, (unsigned long long)wsum);
    }
}

__device__ __forceinline__ void build_tpp_body(
    const float4* __restrict__ pos, const float* __restrict__ quads, const uint32_t* __restrict__ cell,
    const uint32_t* __restrict__ pinfo, const uint32_t* __restrict__ start, const uint32_t* __restrict__ cell_nfluid,
    const SceneDev* __restrict__ scenes, DevStatus* __restrict__ st, uint32_t* __restrict__ nlist,
    uint32_t* __restrict__ ncount, float R2, uint32_t max_neibs, uint32_t stride) {
    const uint32_t n = st->n_active;
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        uint32_t nfound;
        const uint32_t nent = build_particle(i, pos, quads, cell, pinfo, start, cell_nfluid, scenes, nlist, ncount, R2,
                                             max_neibs, stride, &nfound, st, n);
        build_stats(st, nfound, nent, max_neibs, __activemask());
    }
}

// The same list by a block of nine warps for 32 particles: lane l of every warp is particle l of the
// tile, warp r tests the candidates of neighbour row r (three cells), with the broadcast loads of
// the one thread's build.  The rows' hit counts give each row's hits their place; the lists are put
// together in shared memory and written chunk by chunk, the tile's particles side by side.  The one
// thread's list, entry for entry.  For states too small to fill the GPU with a thread per particle,
// whose nine rows are one long chain of instructions: one thread against the nine warps, us: 38 / 9
// at 4,096 particles, 48 / 19 at 19,683, 51 / 42 at 71,680; 466 / 725 at 1.65M (380 warp
// instructions a particle against 224).  Before, a warp per particle with a lane per cell: 11, 36, 102 us
// (1,019 instructions, every lane at an address of its own); nine lanes per particle: 11, 33, 91 us.
// A tile beside a cell of over 64 candidate slots, and lists of over kStageNeibs entries, take the one
// thread's build, after the block's other tiles: marked in ncount, one tile per warp.  (By the first warp, at
// once: 556 us for 79,507 particles at h = 1.9 dp, every tile of them; now 222, a thread per particle 144.
// The marks keep the main loop's registers: with the put-off tiles in registers the three-block shape spilled,
// 2 to 3% of a step.)
constexpr int kRowWarps = 9;
constexpr int kRowBlock = 32 * kRowWarps;
constexpr uint32_t kPutOff = ~0u;  // a list count that no list has
// shared words: the tile's lists (an odd stride apart: lanes of a warp write different banks), the
// hits of every row and particle
__host__ __device__ constexpr uint32_t rows_list_words(uint32_t max_neibs) { return max_neibs | 1u; }
__host__ __device__ constexpr uint32_t rows_smem_words(uint32_t max_neibs) {
    return 32u * (rows_list_words(max_neibs) + 2u * kRowWarps);
}

// hit mask (first candidate in the top bit) of the candidates [b, e) at or after h0, 32 at most;
// h0 a multiple of four
__device__ __forceinline__ uint32_t cell_mask(const float* __restrict__ quads, uint32_t h0, uint32_t b, uint32_t e, f2 nx,
                                              f2 ny, f2 nz, f2 mR2, bool centre, uint32_t r2lim) {
    if (h0 >= e) return 0u;
    const uint32_t hend = min(e, h0 + 32u);
    const ulonglong2* q4 = reinterpret_cast<const ulonglong2*>(quads + quad_word(h0));
    uint32_t g = h0, mask = 0u;
    if (!centre) {
#pragma unroll 1
        for (; g < hend; g += 4u, q4 += 3) {
            const ulonglong2 X = q4[0], Y = q4[1], Z = q4[2];
            const f2 q0 = r2_plus(f2_add(X.x, nx), f2_add(Y.x, ny), f2_add(Z.x, nz), mR2);
            const f2 q1 = r2_plus(f2_add(X.y, nx), f2_add(Y.y, ny), f2_add(Z.y, nz), mR2);
            mask = __funnelshift_l((uint32_t)q0, mask, 1);
            mask = __funnelshift_l((uint32_t)(q0 >> 32), mask, 1);
            mask = __funnelshift_l((uint32_t)q1, mask, 1);
            mask = __funnelshift_l((uint32_t)(q1 >> 32), mask, 1);
        }
    } else {
#pragma unroll 1
        for (; g < hend; g += 4u, q4 += 3) {
            const ulonglong2 X = q4[0], Y = q4[1], Z = q4[2];
            const f2 a0 = r2_plus(f2_add(X.x, nx), f2_add(Y.x, ny), f2_add(Z.x, nz), 0ull);
            const f2 a1 = r2_plus(f2_add(X.y, nx), f2_add(Y.y, ny), f2_add(Z.y, nz), 0ull);
            mask = __funnelshift_l(centre_hit(f2_lo(a0), r2lim), mask, 1);
            mask = __funnelshift_l(centre_hit(f2_hi(a0), r2lim), mask, 1);
            mask = __funnelshift_l(centre_hit(f2_lo(a1), r2lim), mask, 1);
            mask = __funnelshift_l(centre_hit(f2_hi(a1), r2lim), mask, 1);
        }
    }
    const uint32_t first = h0 < b ? b - h0 : 0u, last = hend - h0;
    return (mask << (32u - (g - h0))) & (0xffffffffu >> first) & (0xffffffffu << (32u - last));
}

// the fallback, out of line (its registers would spill the common path's)
__device__ __noinline__ uint32_t build_particle_alone(uint32_t i, const float4* __restrict__ pos,
                                                      const float* __restrict__ quads, const uint32_t* __restrict__ cell,
                                                      const uint32_t* __restrict__ pinfo, const uint32_t* __restrict__ start,
                                                      const uint32_t* __restrict__ cell_nfluid,
                                                      const SceneDev* __restrict__ scenes, uint32_t* __restrict__ nlist,
                                                      uint32_t* __restrict__ ncount, float R2, uint32_t max_neibs,
                                                      uint32_t stride, uint32_t* nfound, DevStatus* st, uint32_t n) {
    return build_particle(i, pos, quads, cell, pinfo, start, cell_nfluid, scenes, nlist, ncount, R2, max_neibs, stride,
                          nfound, st, n);
}

__device__ __forceinline__ void build_rows_body(
    const float4* __restrict__ pos, const float* __restrict__ quads, const uint32_t* __restrict__ cell,
    const uint32_t* __restrict__ pinfo, const uint32_t* __restrict__ start, const uint32_t* __restrict__ cell_nfluid,
    const SceneDev* __restrict__ scenes, DevStatus* __restrict__ st, uint32_t* __restrict__ nlist,
    uint32_t* __restrict__ ncount, float R2, uint32_t max_neibs, uint32_t stride) {
    extern __shared__ uint32_t rows_smem[];
    const int lane = (int)(threadIdx.x & 31u), r = (int)(threadIdx.x >> 5);
    const bool can_stage = max_neibs <= kStageNeibs;
    uint32_t* const list = rows_smem + lane * rows_list_words(max_neibs);  // fluid entries from the front, boundary from the back
    uint32_t* const hit_s = rows_smem + 32u * rows_list_words(max_neibs);  // [row][particle]: fluid | boundary << 16
    uint32_t* const kept_s = hit_s + 32 * kRowWarps;                       // the same after a cut at max_neibs
    const uint32_t n = st->n_active;
    const uint32_t r2lim = __float_as_uint(R2) - 1u;
    const f2 mR2 = f2_dup(-R2);
    uint32_t most = 0, sum = 0;  // of this lane's particles
    __shared__ uint32_t put_off;
    if (threadIdx.x == 0) put_off = 0u;
    for (uint32_t i0 = blockIdx.x * 32u; i0 < n; i0 += gridDim.x * 32u) {
        const uint32_t i = i0 + (uint32_t)lane;
        const bool have = i < n;
        uint32_t b[3] = {0u, 0u, 0u}, f[3] = {0u, 0u, 0u}, e[3] = {0u, 0u, 0u};
        float4 pi = make_float4(0.f, 0.f, 0.f, 0.f);
        f2 ny = 0ull, nz = 0ull;
        float cell_x = 0.f;
        if (have) {
            const SceneDev& sc = scenes[pinfo[i]];
            pi = pos[i];
            int cx, cy, cz;
            decode_local(cell[i] - sc.cell_offset, sc, cx, cy, cz);
            const int dy = r % 3 - 1, dz = r / 3 - 1;
            int y = cy + dy, z = cz + dz;
            bool row_ok = true;
            if (y < 0 || y >= sc.ncell[1]) {
                if ((sc.periodic >> 1) & 1u) y = y < 0 ? y + sc.ncell[1] : y - sc.ncell[1];
                else row_ok = false;
            }
            if (z < 0 || z >= sc.ncell[2]) {
                if ((sc.periodic >> 2) & 1u) z = z < 0 ? z + sc.ncell[2] : z - sc.ncell[2];
                else row_ok = false;
            }
            const uint32_t row = sc.cell_offset + (uint32_t)sc.ncell[0] * ((uint32_t)y + (uint32_t)sc.ncell[1] * (uint32_t)z);
            cell_x = sc.cell_f[0];
            ny = f2_dup((float)dy * sc.cell_f[1] - pi.y);
            nz = f2_dup((float)dz * sc.cell_f[2] - pi.z);
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                int x = cx + k - 1;
                bool ok = row_ok;
                if (x < 0 || x >= sc.ncell[0]) {
                    if (sc.periodic & 1u) x = x < 0 ? x + sc.ncell[0] : x - sc.ncell[0];
                    else ok = false;
                }
                if (ok) {
                    const uint32_t cc = row + (uint32_t)x;
                    b[k] = start[cc];
                    f[k] = b[k] + cell_nfluid[cc];  // end of the fluid part
                    e[k] = pi.w > 0.f ? start[cc + 1] : f[k];
                    SPH_GUARD(b[k] <= f[k] && f[k] <= start[cc + 1] && start[cc + 1] <= n, st, b[k] = f[k] = e[k] = 0u)
                }
            }
        }
        const bool crowded = e[0] > (b[0] & ~3u) + 64u || e[1] > (b[1] & ~3u) + 64u || e[2] > (b[2] & ~3u) + 64u;
        if (__syncthreads_or(crowded || !can_stage)) {  // put off
            if (r == 0 && have) ncount[i] = kPutOff;
            if (threadIdx.x == 0) put_off = 1u;
            continue;
        }
        // hits of the row's three cells, up to 64 candidate slots each; fluid candidates first in a cell
        uint32_t m[6], fluid[6], hits = 0u;
#pragma unroll
        for (int q = 0; q < 6; ++q) {
            const int k = q / 2;
            const uint32_t h0 = (b[k] & ~3u) + 32u * (uint32_t)(q & 1);
            m[q] = 0u;
            if ((q & 1) == 0 || h0 < e[k])
                m[q] = cell_mask(quads, h0, b[k], e[k], f2_dup((float)(k - 1) * cell_x - pi.x), ny, nz, mR2, k == 1 && r == 4,
                                 r2lim);
            const uint32_t nfl = f[k] > h0 ? min(f[k] - h0, 32u) : 0u;
            fluid[q] = nfl ? 0xffffffffu << (32u - nfl) : 0u;
            hits += (uint32_t)__popc(m[q] & fluid[q]) | (uint32_t)__popc(m[q] & ~fluid[q]) << 16;
        }
        hit_s[32 * r + lane] = hits;
        __syncthreads();
        uint32_t at = 0u, all = 0u;  // hits of the rows before, of all rows
#pragma unroll
        for (int q = 0; q < kRowWarps; ++q) {
            const uint32_t h = hit_s[32 * q + lane];
            at += q < r ? h : 0u;
            all += h;
        }
        const uint32_t nfound = (all & 0xffffu) + (all >> 16);
        if (__syncthreads_or(nfound > max_neibs)) {  // keep the first ones in candidate order
            const uint32_t before = (at & 0xffffu) + (at >> 16);
            uint32_t keep = before < max_neibs ? max_neibs - before : 0u;
            hits = 0u;
#pragma unroll
            for (int q = 0; q < 6; ++q) {
                const uint32_t c = min(keep, (uint32_t)__popc(m[q]));
                m[q] = highest_set_bits(m[q], c);
                keep -= c;
                hits += (uint32_t)__popc(m[q] & fluid[q]) | (uint32_t)__popc(m[q] & ~fluid[q]) << 16;
            }
            kept_s[32 * r + lane] = hits;
            __syncthreads();
            at = all = 0u;
            for (int q = 0; q < kRowWarps; ++q) {
                const uint32_t h = kept_s[32 * q + lane];
                at += q < r ? h : 0u;
                all += h;
            }
        }
        uint32_t kf = at & 0xffffu, kb = max_neibs - 1u - (at >> 16);
        const uint32_t code = ((uint32_t)(r % 3) << 2) | ((uint32_t)(r / 3) << 4);
#pragma unroll
        for (int q = 0; q < 6; ++q) {
            const int k = q / 2;
            const uint32_t e0 = (((b[k] & ~3u) + 32u * (uint32_t)(q & 1)) << kCodeBits) | code | (uint32_t)k;
            for (uint32_t s = m[q] & fluid[q]; s; ++kf) {
                const uint32_t u = (uint32_t)__clz((int)s);
                s ^= 0x80000000u >> u;
                list[kf] = e0 + (u << kCodeBits);
            }
            for (uint32_t s = m[q] & ~fluid[q]; s; --kb) {
                const uint32_t u = (uint32_t)__clz((int)s);
                s ^= 0x80000000u >> u;
                list[kb] = e0 + (u << kCodeBits);
            }
        }
        __syncthreads();
        // chunks r, r + 9, ... of both parts, one particle per lane
        const uint32_t nf = all & 0xffffu, nb = all >> 16;
        uint2* const rows = reinterpret_cast<uint2*>(nlist) + i;
        for (uint32_t c = (uint32_t)r; 2u * c < nf; c += kRowWarps)
            rows[(size_t)c * stride] = make_uint2(list[2u * c], 2u * c + 1u < nf ? list[2u * c + 1u] : kMarker);
        for (uint32_t c = (uint32_t)r; 2u * c < nb; c += kRowWarps)
            rows[(size_t)(list_chunks(max_neibs) - 1u - c) * stride] =
                make_uint2(list[max_neibs - 1u - 2u * c], 2u * c + 1u < nb ? list[max_neibs - 2u - 2u * c] : kMarker);
        if (r == 0 && have) {
            ncount[i] = all;
            most = max(most, nfound);
            sum += nf + nb;
        }
        __syncthreads();  // the shared lists are free again
    }
    __syncthreads();
    if (put_off) {  // the block's tiles one by one over its warps
        for (uint32_t i = (blockIdx.x + (uint32_t)r * gridDim.x) * 32u + (uint32_t)lane; i < n;
             i += kRowWarps * gridDim.x * 32u) {
            if (ncount[i] != kPutOff) continue;
            uint32_t nfound;
            sum += build_particle_alone(i, pos, quads, cell, pinfo, start, cell_nfluid, scenes, nlist, ncount, R2,
                                        max_neibs, stride, &nfound, st, n);
            most = max(most, nfound);
        }
    }
    most = __reduce_max_sync(0xffffffffu, most);
    sum = __reduce_add_sync(0xffffffffu, sum);
    if (lane == 0 && most) {
        if (most > max_neibs) atomicOr(&st->error_bits, SPH_EBIT_NEIB_OVERFLOW);
        atomicMax(&st->max_neibs_seen, most);
        atomicAdd(&st->list_entries, (unsigned long long)sum);
    }
}

}  // namespace

}  // namespace sphg
