// Particle interactions and time integration (paper Section 2.1; readings
// of the passages the paper leaves to its references are stated inline).
//
//   drho_i/dt = sum_j m_j (u_i - u_j).x_ij F_ij                        (C1)
//   du_i/dt   = -sum_j m_j (P_i/rho_i^2 + P_j/rho_j^2 + Pi_ij) x_ij F_ij  (C2)
//               + sum_j 4 nu m_j/(rho_i + rho_j) F_ij (u_i - u_j) + g     (C3)
//   Pi_ij = -alpha h c0 mu_ij / rhobar_ij for u_ij.x_ij < 0,
//   mu_ij = u_ij.x_ij/(r^2 + 0.01 h^2), rhobar = (rho_i + rho_j)/2          (C4)
//   F = (1/r) dW/dr = aF (q - 2)^3 for q = r/h < 2 (Wendland C2, Section 4)
//   Dynamic boundary particles: zero velocity, continuity only      (C5)
//
// One thread per particle, sorted order.  The neighbour list is read
// neighbour-major (a warp reads 256 contiguous bytes per two-entry chunk),
// fluid chunks from the front and boundary chunks from the back (split list,
// Section 4), each with its own loop.  Per neighbour the kernel gathers pos4 + vel4
// (32 bytes, served by L1/L2: neighbours of consecutive particles are the
// same cell-sorted particles) and P_j/rho_j^2, which the passes over a list
// built at this step recompute from delta_j instead (see fluid_pair).
// The predictor (dt/2) and corrector (dt) updates of reading C6 are fused
// into the epilogues of the two force passes; the corrector pass reduces
// max |a|^2 per scene (warp reduction + one atomic) for the CFL dt (C7).
#include <cooperative_groups.h>

#include "forces_common.cuh"
#include "packed.cuh"
#include "pipeline.cuh"

namespace cg = cooperative_groups;

namespace sphg {

namespace {

// One neighbour of a fluid particle.  BND: the neighbour is a boundary
// particle (mass stored negated, velocity zero).  The kernel constant aF is
// factored out of every term (all terms are linear in F) and applied once.
// P_j/rho_j^2 comes from delta_j (the function that stores the per-particle
// value, so bit-identical to it) in place of a third gather.
// The pair's terms go to `out` as they are formed: the running sums (Acc), or their values
// (Terms), for a group of lanes that adds its lanes' terms in list order.
__device__ __forceinline__ void add_rate(Acc& a, float mF, float udx) { a.drho = fmaf(mF, udx, a.drho); }
__device__ __forceinline__ void add_force(Acc& a, float coef, float rx, float ry, float rz) {
    a.ax = fmaf(-coef, rx, a.ax);
    a.ay = fmaf(-coef, ry, a.ay);
    a.az = fmaf(-coef, rz, a.az);
}
__device__ __forceinline__ void add_laminar(Acc& a, float lam, float ux, float uy, float uz) {
    a.ax = fmaf(lam, ux, a.ax);
    a.ay = fmaf(lam, uy, a.ay);
    a.az = fmaf(lam, uz, a.az);
}
struct Terms {
    float mF, udx, coef, rx, ry, rz;
    float lam, ux, uy, uz;  // laminar only
    float dd, mF_rho;       // density diffusion only
};
__device__ __forceinline__ void add_rate(Terms& t, float mF, float udx) {
    t.mF = mF;
    t.udx = udx;
}
__device__ __forceinline__ void add_force(Terms& t, float coef, float rx, float ry, float rz) {
    t.coef = coef;
    t.rx = rx;
    t.ry = ry;
    t.rz = rz;
}
__device__ __forceinline__ void add_laminar(Terms& t, float lam, float ux, float uy, float uz) {
    t.lam = lam;
    t.ux = ux;
    t.uy = uy;
    t.uz = uz;
}

// density diffusion (reading D1): drho += dd mF/(rho_j/rho0)
__device__ __forceinline__ void add_diffusion(Acc& a, float dd, float mF_rho) { a.drho = fmaf(dd, mF_rho, a.drho); }
__device__ __forceinline__ void add_diffusion(Terms& t, float dd, float mF_rho) {
    t.dd = dd;
    t.mF_rho = mF_rho;
}

// The model of a pass, template parameter VISC: the viscosity (SPH_VISC_ARTIFICIAL or _LAMINAR), with
// this bit for Molteni & Colagrossi density diffusion.  (The general kernels took 151 / 154 us a pass
// on the 572,120-particle dam break with diffusion, these 122 / 126.)
constexpr int kDiffusion = 8;
__host__ __device__ constexpr bool is_artificial(int v) { return (v & ~kDiffusion) == SPH_VISC_ARTIFICIAL; }
__host__ __device__ constexpr bool is_laminar(int v) { return (v & ~kDiffusion) == SPH_VISC_LAMINAR; }
__host__ __device__ constexpr bool has_diffusion(int v) { return (v & kDiffusion) != 0; }

// FILTER: a pair beyond the cutoff is left out.
template <int VISC, bool BND, bool FILTER, class Out>
__device__ __forceinline__ void fluid_pair(uint32_t e, const float4& pj, const float4& vj, const Central& ci,
                                           const float4& vi, float phat_i, float phat_coef, float pi_coef, float dd_coef,
                                           const Phys& ph, Out& out) {
    const float phat_j = eos_phat(vj.w, ph, phat_coef);
    const float rx = pick(e, ci.xm, ci.x0, ci.xp) - pj.x;
    const float ry = pick(e >> 2, ci.ym, ci.y0, ci.yp) - pj.y;
    const float rz = pick(e >> 4, ci.zm, ci.z0, ci.zp) - pj.z;
    const float r2 = fmaxf(fmaf(rx, rx, fmaf(ry, ry, rz * rz)), 1e-30f);
    if (FILTER && !(r2 < ph.R2)) return;
    const float r = r2 * rsqrt_fast(r2);
    const float t = fminf(fmaf(r, ph.inv_h, -2.0f), 0.0f);
    const float mj = BND ? -pj.w : pj.w;
    const float mF = mj * (t * t * t);  // m_j F / aF
    const float ux = BND ? vi.x : vi.x - vj.x;
    const float uy = BND ? vi.y : vi.y - vj.y;
    const float uz = BND ? vi.z : vi.z - vj.z;
    const float udx = fmaf(ux, rx, fmaf(uy, ry, uz * rz));
    add_rate(out, mF, udx);
    if (has_diffusion(VISC) && !BND) add_diffusion(out, dd_coef * (vi.w - vj.w), mF * rcp_fast(1.0f + vj.w));
    float bracket = phat_i + phat_j;
    if (is_artificial(VISC)) {
        // approaching pairs only (u.x < 0), without a branch: receding pairs add -pi*0
        const float den = (r2 + ph.eps_h2) * fmaf(0.5f, vi.w + vj.w, 1.0f);
        bracket = fmaf(-pi_coef, fminf(udx, 0.f) * rcp_fast(den), bracket);
    }
    add_force(out, mF * bracket, rx, ry, rz);
    if (is_laminar(VISC))
        add_laminar(out, ph.nu4 * ph.inv_rho0 * (mF * rcp_fast(2.0f + vi.w + vj.w)), ux, uy, uz);
}

// one fluid neighbour of a boundary particle: continuity, u_i = 0
template <bool FILTER, class Out>
__device__ __forceinline__ void boundary_pair(uint32_t e, const Central& ci, const float4* __restrict__ pos,
                                              const float4* __restrict__ vel, const Phys& ph, Out& out) {
    const uint32_t j = e >> kCodeBits;
    const float4 pj = pos[j];
    const float4 vj = vel[j];
    const float rx = pick(e, ci.xm, ci.x0, ci.xp) - pj.x;
    const float ry = pick(e >> 2, ci.ym, ci.y0, ci.yp) - pj.y;
    const float rz = pick(e >> 4, ci.zm, ci.z0, ci.zp) - pj.z;
    const float r2 = fmaxf(fmaf(rx, rx, fmaf(ry, ry, rz * rz)), 1e-30f);
    if (FILTER && !(r2 < ph.R2)) return;
    const float r = r2 * rsqrt_fast(r2);
    const float t = fminf(fmaf(r, ph.inv_h, -2.0f), 0.0f);
    add_rate(out, pj.w * (t * t * t), -fmaf(vj.x, rx, fmaf(vj.y, ry, vj.z * rz)));
}

// A part of a particle's list by LANES consecutive lanes of a warp: each lane evaluates
// every LANES-th entry's terms, then all lanes add the group's terms in list order, so the sums are
// those of one thread, to the bit (the terms travel by shuffles: 6 a pair and lane).  For states too
// small to fill the GPU with a thread per particle, where one thread's list is a long chain of
// instructions: a pass over 4,096 particles 17 -> 7 us (8 lanes).  terms(entry, tm) gives an entry's terms.
template <int VISC, int LANES, class F>
__device__ __forceinline__ void lanes_sum(const uint2* __restrict__ lp, ptrdiff_t step, uint32_t cnt, uint32_t n,
                                          DevStatus* st, Acc& acc, F&& terms) {
    const uint32_t sub = threadIdx.x % LANES;
    const unsigned gmask = ((1u << (LANES & 31)) - 1u) << ((threadIdx.x & 31u) & ~(uint32_t)(LANES - 1));
    auto entry = [&](uint32_t k) -> uint32_t {
        return __ldg(reinterpret_cast<const uint32_t*>(lp + (ptrdiff_t)(k >> 1) * step) + (k & 1u));
    };
    uint32_t next = sub < cnt ? entry(sub) : 0u;
    for (uint32_t k0 = 0; k0 < cnt; k0 += LANES) {
        const uint32_t k = k0 + sub, e = next;
        if (k + LANES < cnt) next = entry(k + LANES);  // one round ahead
        Terms tm{};  // past the end (and what an entry's model lacks): zeros
        bool ok = k < cnt;
        SPH_GUARD(!ok || (e >> kCodeBits) < n, st, ok = false)
        if (ok) terms(e, tm);
#pragma unroll
        for (int l = 0; l < LANES; ++l) {
            Terms o;
            o.mF = __shfl_sync(gmask, tm.mF, l, LANES);
            o.udx = __shfl_sync(gmask, tm.udx, l, LANES);
            o.coef = __shfl_sync(gmask, tm.coef, l, LANES);
            o.rx = __shfl_sync(gmask, tm.rx, l, LANES);
            o.ry = __shfl_sync(gmask, tm.ry, l, LANES);
            o.rz = __shfl_sync(gmask, tm.rz, l, LANES);
            if (is_laminar(VISC)) {
                o.lam = __shfl_sync(gmask, tm.lam, l, LANES);
                o.ux = __shfl_sync(gmask, tm.ux, l, LANES);
                o.uy = __shfl_sync(gmask, tm.uy, l, LANES);
                o.uz = __shfl_sync(gmask, tm.uz, l, LANES);
            }
            add_rate(acc, o.mF, o.udx);
            if (has_diffusion(VISC)) {
                o.dd = __shfl_sync(gmask, tm.dd, l, LANES);
                o.mF_rho = __shfl_sync(gmask, tm.mF_rho, l, LANES);
                add_diffusion(acc, o.dd, o.mF_rho);
            }
            add_force(acc, o.coef, o.rx, o.ry, o.rz);
            if (is_laminar(VISC)) add_laminar(acc, o.lam, o.ux, o.uy, o.uz);
        }
    }
}

// (the forces-only pass over a list of every step keeps the |a|^2 reduction for dt0 live beside the sums: it
// gets a looser register cap than the step's passes)
// One particle of a force pass (one iteration of the pass's particle loop): its pair sums
// over its list and the epilogue of the pass (store, predictor or corrector update).
__device__ __forceinline__ uint32_t ld_count_fresh(const uint32_t* p) {
    uint32_t v;
    asm volatile("ld.global.cg.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// List chunk loads: through the read-only path, or (FRESH: the list was written earlier in
// the same kernel, by this thread) through L2 only, coherent with those stores.
template <bool FRESH>
__device__ __forceinline__ uint2 ld_chunk(const uint2* p) {
    if (!FRESH) return __ldg(p);
    uint2 v;
    asm volatile("ld.global.cg.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "l"(p) : "memory");
    return v;
}

// SKIN: nlist/ncount are the step's exact list in its four-entry chunks, but in the forces-only pass, which
// leaves out the skin list's pairs beyond the cutoff itself; the corrector also checks and reduces the
// displacement since the list's build.
// WIDE: list chunks of two entries evaluated together as long as the fluid part has so many left, their
// gathers issued before the first is used.  A state that does not fill the GPU is bound by
// that latency, and has the registers to spare (see launch_forces_v).
template <int VISC, int MODE, bool SKIN, bool FRESH = false, int LANES = 1, int WIDE = 0>
__device__ __forceinline__ void particle_pass(
    uint32_t i, uint32_t n, const float4* __restrict__ pos, const float4* __restrict__ vel,
    const float* __restrict__ phat, float4* io_pos, float4* io_vel, float* io_phat, float4* __restrict__ force_out,
    const uint32_t* __restrict__ pinfo, const uint32_t* __restrict__ nlist, const uint32_t* __restrict__ ncount,
    const SceneDev* __restrict__ scenes, SceneDyn* __restrict__ dyn, DevStatus* __restrict__ st, const Phys& ph,
    int acc_dt, const float4* __restrict__ pos_ref, const uint32_t* __restrict__ pid, uint32_t cnt_fresh = 0) {
    static_assert(LANES == 1 || !(FRESH || SKIN), "a group of lanes takes an every-step list");
    constexpr bool FILTER = SKIN && MODE == kForcesOnly, EXACT = SKIN && !FILTER;
    const uint32_t s = pinfo[i];
    const SceneDev& sc = scenes[s];
    const float4 pi = pos[i];
    const float4 vi = vel[i];
    const uint32_t cnt = FRESH ? cnt_fresh : ncount[i];
    uint32_t nf = cnt & 0xffffu, nb = cnt >> 16;
    SPH_GUARD(nf + nb <= ph.max_neibs, st, nf = nb = 0)
    const bool fluid_i = pi.w > 0.f;
    const float cx = sc.cell_f[0], cy = sc.cell_f[1], cz = sc.cell_f[2];
    Acc acc{0.f, 0.f, 0.f, 0.f};
    const size_t S = ph.stride;
#define SPH_PAIR_OF(BND, e, pj, vj, out) \
    fluid_pair<VISC, BND, FILTER>(e, pj, vj, ci, vi, phat_i, sc.phat_coef, pic, sc.dd_coef, ph, out)
// both gathers issued together
#define SPH_PAIR(BND, e, out)                                                              \
    do {                                                                                   \
        const float4 pj_ = pos[(e) >> kCodeBits], vj_ = vel[(e) >> kCodeBits];             \
        SPH_PAIR_OF(BND, e, pj_, vj_, out);                                                \
    } while (0)
// the filter's branch would keep the second pair's gathers behind the first pair
#define SPH_PAIR2(BND, e0, e1, out)                                                        \
    do {                                                                                   \
        if (FILTER) {                                                                      \
            const float4 pa_ = pos[(e0) >> kCodeBits], va_ = vel[(e0) >> kCodeBits];       \
            const float4 pb_ = pos[(e1) >> kCodeBits], vb_ = vel[(e1) >> kCodeBits];       \
            SPH_PAIR_OF(BND, e0, pa_, va_, out);                                           \
            SPH_PAIR_OF(BND, e1, pb_, vb_, out);                                           \
        } else {                                                                           \
            SPH_PAIR(BND, e0, out);                                                        \
            SPH_PAIR(BND, e1, out);                                                        \
        }                                                                                  \
    } while (0)
    if (LANES > 1) {
        const float phat_i = phat[i];
        const float pic = sc.pi_coef;
        const Central ci = central_of(pi, cx, cy, cz);
        const uint2* fl = reinterpret_cast<const uint2*>(nlist) + i;
        const uint2* bl = fl + (size_t)(list_chunks(ph.max_neibs) - 1u) * S;
        if (fluid_i) {
            lanes_sum<VISC, LANES>(fl, (ptrdiff_t)S, nf, n, st, acc, [&](uint32_t e, Terms& tm) { SPH_PAIR(false, e, tm); });
            lanes_sum<VISC, LANES>(bl, -(ptrdiff_t)S, nb, n, st, acc, [&](uint32_t e, Terms& tm) { SPH_PAIR(true, e, tm); });
            acc.ax = fmaf(ph.aF, acc.ax, ph.g[0]);
            acc.ay = fmaf(ph.aF, acc.ay, ph.g[1]);
            acc.az = fmaf(ph.aF, acc.az, ph.g[2]);
        } else {
            lanes_sum<VISC, LANES>(fl, (ptrdiff_t)S, nf, n, st, acc, [&](uint32_t e, Terms& tm) {
                boundary_pair<false>(e, ci, pos, vel, ph, tm); });
        }
        acc.drho *= ph.aF;
        if (threadIdx.x % LANES != 0) return;  // the first lane finishes the particle
    } else if (fluid_i && EXACT) {
        const float phat_i = phat[i];
        const float pic = sc.pi_coef;
        const Central ci = central_of(pi, cx, cy, cz);
        // full chunks: four pairs with no test between them (their gathers issue together);
        // then the last chunk of each part (1 to 3 entries, the rest kMarker)
#define SPH_OK_E(e) (((e) >> kCodeBits) < n)
        const uint4* cp = reinterpret_cast<const uint4*>(nlist) + i;
        uint32_t k = 0;
        uint4 qn = make_uint4(0u, 0u, 0u, 0u);
        if (nf >= 4) qn = __ldg(cp);
        for (; k + 4 <= nf; k += 4, cp += S) {
            const uint4 q = qn;
            if (k + 8 <= nf) qn = __ldg(cp + S);  // the next full chunk, one iteration ahead
            SPH_GUARD(SPH_OK_E(q.x) && SPH_OK_E(q.y) && SPH_OK_E(q.z) && SPH_OK_E(q.w), st, break)
            SPH_PAIR(false, q.x, acc);
            SPH_PAIR(false, q.y, acc);
            SPH_PAIR(false, q.z, acc);
            SPH_PAIR(false, q.w, acc);
        }
        do {
            if (k >= nf) break;
            const uint4 q = __ldg(cp);
            SPH_GUARD(SPH_OK_E(q.x) && (k + 1 >= nf || SPH_OK_E(q.y)) && (k + 2 >= nf || SPH_OK_E(q.z)), st, break)
            SPH_PAIR(false, q.x, acc);
            if (k + 1 < nf) SPH_PAIR(false, q.y, acc);
            if (k + 2 < nf) SPH_PAIR(false, q.z, acc);
        } while (0);
        cp = reinterpret_cast<const uint4*>(nlist) + (size_t)exact_bnd_chunk(ph.max_neibs) * S + i;
        for (k = 0; k + 4 <= nb; k += 4, cp += S) {
            const uint4 q = __ldg(cp);
            SPH_GUARD(SPH_OK_E(q.x) && SPH_OK_E(q.y) && SPH_OK_E(q.z) && SPH_OK_E(q.w), st, break)
            SPH_PAIR(true, q.x, acc);
            SPH_PAIR(true, q.y, acc);
            SPH_PAIR(true, q.z, acc);
            SPH_PAIR(true, q.w, acc);
        }
        do {
            if (k >= nb) break;
            const uint4 q = __ldg(cp);
            SPH_GUARD(SPH_OK_E(q.x) && (k + 1 >= nb || SPH_OK_E(q.y)) && (k + 2 >= nb || SPH_OK_E(q.z)), st, break)
            SPH_PAIR(true, q.x, acc);
            if (k + 1 < nb) SPH_PAIR(true, q.y, acc);
            if (k + 2 < nb) SPH_PAIR(true, q.z, acc);
        } while (0);
#undef SPH_OK_E
        acc.ax = fmaf(ph.aF, acc.ax, ph.g[0]);
        acc.ay = fmaf(ph.aF, acc.ay, ph.g[1]);
        acc.az = fmaf(ph.aF, acc.az, ph.g[2]);
        acc.drho *= ph.aF;
    } else if (fluid_i) {
        const float phat_i = phat[i];
        const float pic = sc.pi_coef;
        const Central ci = central_of(pi, cx, cy, cz);
        // list chunks come from DRAM: two chunks (four entries) per iteration, loaded one
        // iteration ahead so that their latency is not on the path to the gathers
        const uint2* lp = reinterpret_cast<const uint2*>(nlist) + i;
        uint32_t k = 0;
        if constexpr (WIDE > 0) {
            constexpr uint32_t kRound = 2 * WIDE;
            uint2 next[WIDE];
            if (nf >= kRound)
#pragma unroll
                for (int c = 0; c < WIDE; ++c) next[c] = ld_chunk<FRESH>(lp + c * S);
            for (; k + kRound <= nf; k += kRound, lp += WIDE * S) {
                uint2 a[WIDE];
                uint32_t top = 0u;
#pragma unroll
                for (int c = 0; c < WIDE; ++c) {
                    a[c] = next[c];
                    top = max(top, max(a[c].x, a[c].y));
                }
                if (k + 2 * kRound <= nf)
#pragma unroll
                    for (int c = 0; c < WIDE; ++c) next[c] = ld_chunk<FRESH>(lp + (WIDE + c) * S);
                SPH_GUARD((top >> kCodeBits) < n, st, break)
#pragma unroll
                for (int c = 0; c < WIDE; ++c) {
                    SPH_PAIR(false, a[c].x, acc);
                    SPH_PAIR(false, a[c].y, acc);
                }
            }
        }
        uint2 an = make_uint2(0u, 0u), bn = make_uint2(0u, 0u);
        if (k + 4 <= nf) {
            an = ld_chunk<FRESH>(lp);
            bn = ld_chunk<FRESH>(lp + S);
        }
        for (; k + 4 <= nf; k += 4, lp += 2 * S) {
            const uint2 a = an, b = bn;
            if (k + 8 <= nf) {  // the next iteration's chunks (within the fluid part)
                an = ld_chunk<FRESH>(lp + 2 * S);
                bn = ld_chunk<FRESH>(lp + 3 * S);
            }
            SPH_GUARD((max(max(a.x, a.y), max(b.x, b.y)) >> kCodeBits) < n, st, break)
            SPH_PAIR2(false, a.x, a.y, acc);
            SPH_PAIR2(false, b.x, b.y, acc);
        }
        for (; k < nf; k += 2, lp += S) {
            const uint2 a = ld_chunk<FRESH>(lp);
            const bool two = k + 1 < nf;
            SPH_GUARD((a.x >> kCodeBits) < n && (!two || (a.y >> kCodeBits) < n), st, break)
            SPH_PAIR(false, a.x, acc);
            if (two) SPH_PAIR(false, a.y, acc);
        }
        lp = reinterpret_cast<const uint2*>(nlist) + (size_t)(list_chunks(ph.max_neibs) - 1u) * S + i;
        for (k = 0; k < nb; k += 2, lp -= S) {
            const uint2 a = ld_chunk<FRESH>(lp);
            const bool two = k + 1 < nb;
            SPH_GUARD((a.x >> kCodeBits) < n && (!two || (a.y >> kCodeBits) < n), st, break)
            SPH_PAIR(true, a.x, acc);
            if (two) SPH_PAIR(true, a.y, acc);
        }
        acc.ax = fmaf(ph.aF, acc.ax, ph.g[0]);
        acc.ay = fmaf(ph.aF, acc.ay, ph.g[1]);
        acc.az = fmaf(ph.aF, acc.az, ph.g[2]);
        acc.drho *= ph.aF;
    } else {
        // boundary particle: continuity over its fluid neighbours, u_i = 0
        const Central ci = central_of(pi, cx, cy, cz);
        const uint2* lp = reinterpret_cast<const uint2*>(nlist) + i;
        const uint4* cp = reinterpret_cast<const uint4*>(nlist) + i;  // EXACT
        uint4 q = make_uint4(0u, 0u, 0u, 0u);
        uint2 q2 = make_uint2(0u, 0u);
#pragma unroll 2
        for (uint32_t k = 0; k < nf; ++k) {
            uint32_t e;
            if (EXACT) {
                if ((k & 3u) == 0u) {
                    q = __ldg(cp);
                    cp += S;
                }
                e = (k & 3u) == 0u ? q.x : ((k & 3u) == 1u ? q.y : ((k & 3u) == 2u ? q.z : q.w));
            } else {
                if ((k & 1u) == 0u) {
                    q2 = ld_chunk<FRESH>(lp);
                    lp += S;
                }
                e = (k & 1u) ? q2.y : q2.x;
            }
            SPH_GUARD((e >> kCodeBits) < n, st, continue)
            boundary_pair<FILTER>(e, ci, pos, vel, ph, acc);
        }
        acc.drho *= ph.aF;
    }
#undef SPH_PAIR2
#undef SPH_PAIR
#undef SPH_PAIR_OF

    // epilogue written out here rather than through finish_particle() of
    // forces_common.cuh (same operations): measured 7 % faster in these kernels
    if (MODE == kForcesOnly) {
        force_out[i] = make_float4(acc.ax, acc.ay, acc.az, acc.drho);
    } else {
        const float dt = dyn[s].dt;
        if (MODE == kPredict) {
            const float hd = 0.5f * dt;
            float4 po = pi, vo = vi;
            vo.w = fmaf(hd * ph.inv_rho0, acc.drho, vi.w);
            if (fluid_i) {
                vo.x = fmaf(hd, acc.ax, vi.x);
                vo.y = fmaf(hd, acc.ay, vi.y);
                vo.z = fmaf(hd, acc.az, vi.z);
                po.x = fmaf(hd, vi.x, pi.x);
                po.y = fmaf(hd, vi.y, pi.y);
                po.z = fmaf(hd, vi.z, pi.z);
            }
            io_pos[i] = po;
            io_vel[i] = vo;
            io_phat[i] = eos_phat(vo.w, ph, sc.phat_coef);
        } else {  // kCorrect: state n in io_*, overwritten by n+1
            float4 po = io_pos[i], vo = io_vel[i];
            const float un_x = vo.x, un_y = vo.y, un_z = vo.z;
            vo.w = fmaf(dt * ph.inv_rho0, acc.drho, vo.w);
            if (fluid_i) {
                vo.x = fmaf(dt, acc.ax, un_x);
                vo.y = fmaf(dt, acc.ay, un_y);
                vo.z = fmaf(dt, acc.az, un_z);
                const float hd = 0.5f * dt;
                po.x = fmaf(hd, un_x + vo.x, po.x);
                po.y = fmaf(hd, un_y + vo.y, po.y);
                po.z = fmaf(hd, un_z + vo.z, po.z);
            }
            io_pos[i] = po;
            io_vel[i] = vo;
            io_phat[i] = eos_phat(vo.w, ph, sc.phat_coef);
            const float chk = po.x + po.y + po.z + vo.x + vo.y + vo.z + vo.w;
            if (!isfinite(chk)) atomicOr(&st->error_bits, SPH_EBIT_NONFINITE);
            if (SKIN) {
                // the list (built with a skin) covers the cutoff while no particle has
                // moved more than skin/2 since the build; the largest displacement
                // decides the next rebuild (k_dt)
                const float4 r0 = pos_ref[i];
                const float dx = po.x - r0.x, dy = po.y - r0.y, dz = po.z - r0.z;
                const float d2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
                if (d2 > ph.skin_lim2) atomicOr(&st->error_bits, SPH_EBIT_SKIN);
                const unsigned mk = __activemask();
                const uint32_t m = __reduce_max_sync(mk, __float_as_uint(d2));
                if ((threadIdx.x & 31) == (uint32_t)(__ffs(mk) - 1)) atomicMax(&st->maxdisp2_bits, m);
            }
        }
    }
    if (MODE == kCorrect || acc_dt) {
        const float a2 = fluid_i && cfl_counts(ph, pid, i)
                             ? fmaf(acc.ax, acc.ax, fmaf(acc.ay, acc.ay, acc.az * acc.az)) : 0.f;
        const uint32_t bits = __float_as_uint(a2);
        const unsigned mask = __activemask();
        const unsigned same = __match_any_sync(mask, s);
        if (same == mask) {
            const uint32_t m = __reduce_max_sync(mask, bits);
            if ((threadIdx.x & 31) == (uint32_t)(__ffs(mask) - 1) && m) atomicMax(&dyn[s].amax2_bits, m);
        } else if (bits) {
            atomicMax(&dyn[s].amax2_bits, bits);
        }
    }
}

template <int VISC, int MODE, bool SKIN, int LANES = 1, int WIDE = 0>
__device__ __forceinline__ void forces_body(
    const float4* __restrict__ pos, const float4* __restrict__ vel, const float* __restrict__ phat,
    float4* io_pos, float4* io_vel, float* io_phat, float4* __restrict__ force_out,
    const uint32_t* __restrict__ pinfo, const uint32_t* __restrict__ nlist, const uint32_t* __restrict__ ncount,
    const SceneDev* __restrict__ scenes, SceneDyn* __restrict__ dyn, DevStatus* __restrict__ st, const Phys& ph,
    int acc_dt, const float4* __restrict__ pos_ref, const uint32_t* __restrict__ pid) {
    const uint32_t n = st->n_active;
    for (uint32_t i = (blockIdx.x * blockDim.x + threadIdx.x) / LANES; i < n; i += gridDim.x * blockDim.x / LANES)
        particle_pass<VISC, MODE, SKIN, false, LANES, WIDE>(i, n, pos, vel, phat, io_pos, io_vel, io_phat, force_out, pinfo,
                                                            nlist, ncount, scenes, dyn, st, ph, acc_dt, pos_ref, pid);
}

template <int VISC, int MODE, int kBlock, int kMinBlocks, bool SKIN, int LANES, int WIDE>
__global__ void __launch_bounds__(kBlock, MODE == kForcesOnly && !SKIN ? (kMinBlocks * 2 + 2) / 3 : kMinBlocks) k_forces(
    const float4* __restrict__ pos, const float4* __restrict__ vel, const float* __restrict__ phat,
    float4* io_pos, float4* io_vel, float* io_phat, float4* __restrict__ force_out,
    const uint32_t* __restrict__ pinfo, const uint32_t* __restrict__ nlist, const uint32_t* __restrict__ ncount,
    const SceneDev* __restrict__ scenes, SceneDyn* __restrict__ dyn, DevStatus* __restrict__ st, const Phys ph,
    int acc_dt, const float4* __restrict__ pos_ref, const uint32_t* __restrict__ pid) {
    forces_body<VISC, MODE, SKIN, LANES, WIDE>(pos, vel, phat, io_pos, io_vel, io_phat, force_out, pinfo, nlist, ncount,
                                               scenes, dyn, st, ph, acc_dt, pos_ref, pid);
}

// ---------------------------------------------------------------------
// A list with a skin (rebuilt every k steps): the step's exact list, the listed pairs within the
// influence radius at x^n, in list order, in chunks of four entries.  Both passes of the step
// then run over it.  One gather and one test a listed pair; the
// predictor over the skin list itself evaluated a warp's pairs beyond the radius along with the others
// (1.65M dam break, skin 0.3 h: 640 us, now 290 for the list and 283 for the pass; bound by the gathers
// through L1).  The pairs kept are counted (DevStatus.interactions).
// A forces-only pass would use the list once: it tests the skin list's pairs itself, two pairs' gathers at a
// time, in 64 registers (the same state: 336 us; the list and a pass over it 495; one pair at a time 350; in
// 85 registers 356; with 42,120 particles 38 / 45 / 40 / 38).
// ---------------------------------------------------------------------
__global__ void __launch_bounds__(128, 8) k_exact_list(const float4* __restrict__ pos, const uint32_t* __restrict__ pinfo,
                                                       const uint32_t* __restrict__ nlist,
                                                       const uint32_t* __restrict__ ncount,
                                                       const SceneDev* __restrict__ scenes, DevStatus* __restrict__ st,
                                                       float R2, uint32_t max_neibs, uint32_t stride,
                                                       uint32_t* __restrict__ nlist_x, uint32_t* __restrict__ ncount_x) {
    const uint32_t n = st->n_active;
    uint32_t kept = 0;
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const SceneDev& sc = scenes[pinfo[i]];
        const Central ci = central_of(pos[i], sc.cell_f[0], sc.cell_f[1], sc.cell_f[2]);
        const uint32_t cnt = ncount[i];
        uint32_t nf = cnt & 0xffffu, nb = cnt >> 16;
        SPH_GUARD(nf + nb <= max_neibs, st, nf = nb = 0)
        const size_t S = stride;
        auto within = [&](uint32_t e, const float4& pj) -> bool {
            const float rx = pick(e, ci.xm, ci.x0, ci.xp) - pj.x;
            const float ry = pick(e >> 2, ci.ym, ci.y0, ci.yp) - pj.y;
            const float rz = pick(e >> 4, ci.zm, ci.z0, ci.zp) - pj.z;
            return fmaf(rx, rx, fmaf(ry, ry, rz * rz)) < R2;
        };
        auto part = [&](const uint2* lp, ptrdiff_t step, uint32_t m, ChunkWriter& w) {
            uint32_t k = 0;
            uint2 an = make_uint2(0u, 0u), bn = make_uint2(0u, 0u);
            if (m >= 4) {
                an = __ldg(lp);
                bn = __ldg(lp + step);
            }
            for (; k + 4 <= m; k += 4, lp += 2 * step) {
                const uint2 a = an, b = bn;
                if (k + 8 <= m) {  // the next iteration's chunks
                    an = __ldg(lp + 2 * step);
                    bn = __ldg(lp + 3 * step);
                }
                SPH_GUARD((max(max(a.x, a.y), max(b.x, b.y)) >> kCodeBits) < n, st, break)
                const float4 p0 = pos[a.x >> kCodeBits], p1 = pos[a.y >> kCodeBits];
                const float4 p2 = pos[b.x >> kCodeBits], p3 = pos[b.y >> kCodeBits];
                const bool h0 = within(a.x, p0), h1 = within(a.y, p1), h2 = within(b.x, p2), h3 = within(b.y, p3);
                w.put(h0, a.x);
                w.put(h1, a.y);
                w.put(h2, b.x);
                w.put(h3, b.y);
            }
            for (; k < m; k += 2, lp += step) {
                const uint2 a = __ldg(lp);
                const bool two = k + 1 < m;
                SPH_GUARD((a.x >> kCodeBits) < n && (!two || (a.y >> kCodeBits) < n), st, break)
                w.put(within(a.x, pos[a.x >> kCodeBits]), a.x);
                if (two) w.put(within(a.y, pos[a.y >> kCodeBits]), a.y);
            }
            w.flush();
        };
        const uint2* const fl = reinterpret_cast<const uint2*>(nlist) + i;
        ChunkWriter wf{make_uint4(0u, 0u, 0u, 0u), 0u, reinterpret_cast<uint4*>(nlist_x) + i, S};
        part(fl, (ptrdiff_t)S, nf, wf);
        ChunkWriter wb{make_uint4(0u, 0u, 0u, 0u), 0u,
                       reinterpret_cast<uint4*>(nlist_x) + (size_t)exact_bnd_chunk(max_neibs) * S + i, S};
        part(fl + (size_t)(list_chunks(max_neibs) - 1u) * S, -(ptrdiff_t)S, nb, wb);
        ncount_x[i] = wf.n | (wb.n << 16);
        kept += wf.n + wb.n;
    }
    const uint32_t w = __reduce_add_sync(0xffffffffu, kept);
    if ((threadIdx.x & 31) == 0 && w) atomicAdd(&st->interactions, (unsigned long long)w);
}

// Predictor update (reading C6) from forces already stored by a
// forces-only pass at the same state: the same operations as the predictor
// pass's epilogue, so the result is the same to the bit.  Used by the first
// step after a list build, whose dt0 forces pass is also its predictor's.
__global__ void k_predict_from_forces(const float4* __restrict__ pos, const float4* __restrict__ vel,
                                      const float4* __restrict__ force, const uint32_t* __restrict__ pinfo,
                                      const SceneDev* __restrict__ scenes, const SceneDyn* __restrict__ dyn,
                                      const DevStatus* __restrict__ st, const Phys ph, float4* __restrict__ pos_o,
                                      float4* __restrict__ vel_o, float* __restrict__ phat_o) {
    const uint32_t n = st->n_active;
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const uint32_t s = pinfo[i];
        const float4 pi = pos[i], vi = vel[i], a = force[i];
        const float hd = 0.5f * dyn[s].dt;
        float4 po = pi, vo = vi;
        vo.w = fmaf(hd * ph.inv_rho0, a.w, vi.w);
        if (pi.w > 0.f) {
            vo.x = fmaf(hd, a.x, vi.x);
            vo.y = fmaf(hd, a.y, vi.y);
            vo.z = fmaf(hd, a.z, vi.z);
            po.x = fmaf(hd, vi.x, pi.x);
            po.y = fmaf(hd, vi.y, pi.y);
            po.z = fmaf(hd, vi.z, pi.z);
        }
        pos_o[i] = po;
        vel_o[i] = vo;
        phat_o[i] = eos_phat(vo.w, ph, scenes[s].phat_coef);
    }
}

// the CFL dt the next step of scene 0 would take, without changing any state
__global__ void k_dt_peek(const SceneDev* __restrict__ scenes, const SceneDyn* __restrict__ dyn,
                          DevStatus* __restrict__ st, double h, double cfl, double dt_fixed) {
    if (threadIdx.x == 0) st->dt_peek = cfl_dt_of(scenes[0], dyn[0], h, cfl, dt_fixed);
}

__global__ void k_dt(const DtArgs a) { dt_body(a); }

// ---------------------------------------------------------------------
// The neighbour build and the predictor pass in one kernel: each thread writes
// its particle's list (the thread-per-particle build) and evaluates the
// predictor pass over it at once, while the list and the candidates it has
// just loaded are in cache; no separate pass re-reads the list.  The same
// list and, pair for pair in the same order, the same sums and update as the
// two kernels.  List rebuilt every step (no skin), default model.
// What it saves is the list's second reading: 1.65M dam break, 239 MB of DRAM reads against the two kernels' 238 +
// 422, the same 562M warp instructions (363M + 197M) at 67% issue (66 and 66%), 708 us against 451 + 265;
// 20.1M, 13.0 GB of traffic against 11.6 + 7.4, 9.77 ms against 6.60 + 3.53.  Per step 1.0M box 942 -> 907 us,
// 20.1M dam break 15.35 -> 14.80 ms, tanks of 2.0M 1301 -> 1320 (figures by size and block at
// default_variants, sph_api.cu).
// ---------------------------------------------------------------------
template <int VISC, int kBlockT>
__global__ void __launch_bounds__(kBlockT, 1024 / kBlockT) k_build_predict(const Buffers b, int cur, const Phys ph) {
    DevStatus* st = b.status;
    const uint32_t n = st->n_active;
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        uint32_t nfound;
        const uint32_t nent = build_particle(i, b.pos[cur], b.quads, b.cell[cur], b.pinfo[cur], b.start,
                                             b.cell_nfluid, b.scenes, b.nlist, b.ncount, ph.R2_list, ph.max_neibs, ph.stride, &nfound, st, n);
        build_stats(st, nfound, nent, ph.max_neibs, __activemask());
        asm volatile("" ::: "memory");  // the list stores above precede its loads below
        const uint32_t cnt = ld_count_fresh(b.ncount + i);
        particle_pass<VISC, kPredict, false, true>(i, n, b.pos[cur], b.vel[cur], b.phat[cur], b.pos_s, b.vel_s,
                                                   b.phat_s, nullptr, b.pinfo[cur], b.nlist, b.ncount, b.scenes,
                                                   b.dyn, st, ph, 0, nullptr, b.pid[cur], cnt);
    }
}

// ---------------------------------------------------------------------
// The whole step as one persistent kernel (batched scenes, north of the
// per-kernel graph): every block runs each phase of the step over its share
// of the particles (grid-stride loops), with a grid-wide barrier between
// phases, for nsteps steps.  A cooperative launch keeps every block resident,
// so the barriers always complete.  Phases and their arithmetic are the
// kernels of the captured step (dt, hash, scan, scatter, reorder,
// thread-per-particle list build, predictor pass, corrector pass), so the
// result is the same to the bit.  List rebuilt every step, default model.
// ---------------------------------------------------------------------
// 4 resident blocks of 256 threads per SM (64 registers): measured faster than 3 (80
// registers) and 2 (128): 12.5 / 13.9 / 16.3 ms per step on the 256-tank batch
constexpr int kPersistMinBlocks = 4;
template <int VISC>
__global__ void __launch_bounds__(kPipeBlock, kPersistMinBlocks) k_step_persistent(const Buffers b, const Geometry g, const Phys ph,
                                                                    int cur0, uint32_t nsteps) {
    cg::grid_group grid = cg::this_grid();
    const uint32_t nb = g.n_cells + 1;  // buckets: cells + the sentinel of removed particles
    const uint32_t ntiles = (nb + kScanTile - 1) / kScanTile;
    for (uint32_t s = 0; s < nsteps; ++s) {
        const int cur = (cur0 + (int)s) & 1, nxt = cur ^ 1;
        if (blockIdx.x == 0)
            dt_body(dt_args(b, g, ph, 1, 1));
        hash_body(b.pos[cur], b.cell[cur], b.pinfo[cur], b.scenes, b.status, b.key, b.slot, b.count, g.n_cells);
        grid.sync();
        for (uint32_t t = blockIdx.x; t < ntiles; t += gridDim.x) scan_reduce_tile(b.count, nb, b.bsum, t);
        grid.sync();
        if (blockIdx.x == 0) scan_bsums_body(b.bsum, ntiles);
        grid.sync();
        for (uint32_t t = blockIdx.x; t < ntiles; t += gridDim.x)
            scan_down_tile(b.count, nb, b.bsum, b.start, b.status, t);
        grid.sync();
        scatter_body(b.key, b.slot, b.start, b.status, b.unsorted, nb);
        grid.sync();
        reorder_body<kReorderCells>(b.pos[cur], b.vel[cur], b.phat[cur], b.pinfo[cur], b.pid[cur], b.start, b.unsorted, b.scenes,
                     g.n_cells, b.status, b.cell_nfluid, b.pos[nxt], b.vel[nxt], b.phat[nxt], b.cell[nxt],
                     b.pinfo[nxt], b.pid[nxt], b.quads);
        grid.sync();
        build_tpp_body(b.pos[nxt], b.quads, b.cell[nxt], b.pinfo[nxt], b.start, b.cell_nfluid, b.scenes, b.status, b.nlist,
                       b.ncount, ph.R2_list, ph.max_neibs, ph.stride);
        grid.sync();
        forces_body<VISC, kPredict, false>(b.pos[nxt], b.vel[nxt], b.phat[nxt], b.pos_s, b.vel_s, b.phat_s, nullptr,
                                           b.pinfo[nxt], b.nlist, b.ncount, b.scenes, b.dyn, b.status, ph, 0,
                                           nullptr, b.pid[nxt]);
        grid.sync();
        forces_body<VISC, kCorrect, false>(b.pos_s, b.vel_s, b.phat_s, b.pos[nxt], b.vel[nxt], b.phat[nxt], nullptr,
                                           b.pinfo[nxt], b.nlist, b.ncount, b.scenes, b.dyn, b.status, ph, 0,
                                           nullptr, b.pid[nxt]);
        grid.sync();
    }
}

template <int VISC, int B, int MB, bool SKIN, int LANES, int WIDE>
void launch_forces_s(const Buffers& b, int cur, const Geometry& g, const Phys& ph, ForceMode mode, int acc_dt,
                     cudaStream_t st) {
    const unsigned grid = g.cap ? (unsigned)(((uint64_t)g.cap * LANES + B - 1) / B) : 1;
    const bool exact = SKIN && mode != kForcesOnly;
    const uint32_t* const list = exact ? b.nlist_x : b.nlist;
    const uint32_t* const count = exact ? b.ncount_x : b.ncount;
    switch (mode) {
        case kForcesOnly:
            k_forces<VISC, kForcesOnly, B, MB, SKIN, LANES, WIDE><<<grid, B, 0, st>>>(
                b.pos[cur], b.vel[cur], b.phat[cur], nullptr, nullptr, nullptr, b.force, b.pinfo[cur], list, count,
                b.scenes, b.dyn, b.status, ph, acc_dt, nullptr, b.pid[cur]);
            break;
        case kPredict:
            k_forces<VISC, kPredict, B, MB, SKIN, LANES, WIDE><<<grid, B, 0, st>>>(
                b.pos[cur], b.vel[cur], b.phat[cur], b.pos_s, b.vel_s, b.phat_s, nullptr, b.pinfo[cur], list, count,
                b.scenes, b.dyn, b.status, ph, 0, nullptr, b.pid[cur]);
            break;
        case kCorrect:
            k_forces<VISC, kCorrect, B, MB, SKIN, LANES, WIDE><<<grid, B, 0, st>>>(
                b.pos_s, b.vel_s, b.phat_s, b.pos[cur], b.vel[cur], b.phat[cur], nullptr, b.pinfo[cur], list, count,
                b.scenes, b.dyn, b.status, ph, 0, b.pos_ref, b.pid[cur]);
            break;
    }
}

// (a skin list's passes take the plain shapes)
template <int VISC, int B, int MB, int LANES = 1, int WIDE = 0>
void launch_forces_b(const Buffers& b, int cur, const Geometry& g, const Phys& ph, ForceMode mode, int acc_dt,
                     cudaStream_t st) {
    constexpr bool kPlain = LANES == 1 && WIDE == 0;
    if (b.pos_ref)
        launch_forces_s<VISC, (kPlain ? B : 128), (kPlain ? MB : 8), true, 1, 0>(b, cur, g, ph, mode, acc_dt, st);
    else
        launch_forces_s<VISC, B, MB, false, LANES, WIDE>(b, cur, g, ph, mode, acc_dt, st);
}

// Launch shapes of the force kernels (autotuned, the corrector pass on its own): threads per block, the
// register cap implied by a minimum of resident blocks per SM, lanes per particle, list chunks
// evaluated together.  States that do not fill the GPU keep more of a particle's pairs in flight, the
// fewer particles the more.  us per step with 128 threads (1), 8 lanes (4), 16 entries a round (3),
// 8 entries a round (0):
//     4,096 particles  55.5  36.5  40.1  46.8      32,768 particles  75.4  96.6  61.9  64.2
//     8,000            64.4  40.5  42.3  47.1      46,656            89.8   126  80.2  78.1
//    12,167            65.2  54.4  44.0  50.5      64,000             101   162   111  95.2
//    19,683            70.7  72.9  51.4  56.3      97,336             134   236   140   136
// A pass over 1.65M takes 278 us with 1, 287 with 2, 315 with 0; over a 1.0M box 247 with 1, 244 with 2.
template <int VISC>
void launch_forces_v(const Buffers& b, int cur, const Geometry& g, const Phys& ph, ForceMode mode, int acc_dt,
                     cudaStream_t st) {
    switch (mode == kCorrect ? ph.forces_variant_c : mode == kPredict ? ph.forces_variant : ph.forces_variant_f) {
        case 0: launch_forces_b<VISC, 64, 10, 1, 4>(b, cur, g, ph, mode, acc_dt, st); break;
        case 2: launch_forces_b<VISC, 256, 4>(b, cur, g, ph, mode, acc_dt, st); break;
        case 3: launch_forces_b<VISC, 32, 9, 1, 8>(b, cur, g, ph, mode, acc_dt, st); break;
        case 4: launch_forces_b<VISC, 128, 4, 8>(b, cur, g, ph, mode, acc_dt, st); break;
        default: launch_forces_b<VISC, 128, 8>(b, cur, g, ph, mode, acc_dt, st); break;
    }
}

// Conservation sums (Section 2.1 invariants) over particles: momentum sum m u,
// force sum m a, sum m drho/dt, kinetic energy, total mass; |m| (boundary masses
// are stored negated).  Deterministic: a fixed grid, a fixed particle order per thread and
// fixed-order tree reductions in FP64 (per block, then over blocks).
constexpr int kConsBlocks = 304, kConsThreads = 256, kConsQ = kConservationSums;

__global__ void __launch_bounds__(kConsThreads) k_cons_partial(const float4* __restrict__ pos,
                                                               const float4* __restrict__ vel,
                                                               const float4* __restrict__ force,
                                                               const DevStatus* __restrict__ st,
                                                               double* __restrict__ part) {
    __shared__ double red[kConsQ][kConsThreads];
    double q[kConsQ] = {0, 0, 0, 0, 0, 0, 0, 0, 0};
    const uint32_t n = st->n_active;
    for (uint32_t i = blockIdx.x * kConsThreads + threadIdx.x; i < n; i += kConsBlocks * kConsThreads) {
        const double m = fabs((double)pos[i].w);
        const float4 v = vel[i], a = force[i];
        const bool fluid = pos[i].w > 0.f;
        const double ux = fluid ? v.x : 0.0, uy = fluid ? v.y : 0.0, uz = fluid ? v.z : 0.0;
        q[0] += m * ux;
        q[1] += m * uy;
        q[2] += m * uz;
        q[3] += m * a.x;
        q[4] += m * a.y;
        q[5] += m * a.z;
        q[6] += m * a.w;
        q[7] += 0.5 * m * (ux * ux + uy * uy + uz * uz);
        q[8] += m;
    }
#pragma unroll
    for (int k = 0; k < kConsQ; ++k) red[k][threadIdx.x] = q[k];
    __syncthreads();
    for (int w = kConsThreads / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w)
#pragma unroll
            for (int k = 0; k < kConsQ; ++k) red[k][threadIdx.x] += red[k][threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x < kConsQ) part[blockIdx.x * kConsQ + threadIdx.x] = red[threadIdx.x][0];
}

__global__ void k_cons_final(const double* __restrict__ part, double* __restrict__ out) {
    if (threadIdx.x < kConsQ) {
        double s = 0.0;
        for (int b = 0; b < kConsBlocks; ++b) s += part[b * kConsQ + threadIdx.x];
        out[threadIdx.x] = s;
    }
}

}  // namespace

size_t conservation_scratch_bytes() { return sizeof(double) * kConsQ * (kConsBlocks + 1); }

void launch_conservation(const Buffers& b, int cur, double* scratch, cudaStream_t st) {
    k_cons_partial<<<kConsBlocks, kConsThreads, 0, st>>>(b.pos[cur], b.vel[cur], b.force, b.status, scratch);
    k_cons_final<<<1, 32, 0, st>>>(scratch, scratch + kConsQ * kConsBlocks);
}

void launch_forces(const Buffers& b, int cur, const Geometry& g, const Phys& ph, ForceMode mode, int acc_dt,
                   cudaStream_t st) {
    if (b.pos_ref && mode == kPredict && !ph.general)  // a skin list: first the step's exact list
        k_exact_list<<<g.cap ? (g.cap + 127) / 128 : 1, 128, 0, st>>>(
            b.pos[cur], b.pinfo[cur], b.nlist, b.ncount, b.scenes, b.status, ph.R2, ph.max_neibs, ph.stride,
            b.nlist_x, b.ncount_x);
    if (ph.general) {
        launch_forces_models(b, cur, g, ph, mode, acc_dt, st);
        return;
    }
    if (ph.ddiff) {
        if (ph.visc == SPH_VISC_LAMINAR)
            launch_forces_v<SPH_VISC_LAMINAR | kDiffusion>(b, cur, g, ph, mode, acc_dt, st);
        else
            launch_forces_v<SPH_VISC_ARTIFICIAL | kDiffusion>(b, cur, g, ph, mode, acc_dt, st);
    } else if (ph.visc == SPH_VISC_LAMINAR)
        launch_forces_v<SPH_VISC_LAMINAR>(b, cur, g, ph, mode, acc_dt, st);
    else
        launch_forces_v<SPH_VISC_ARTIFICIAL>(b, cur, g, ph, mode, acc_dt, st);
}

const char* forces_variant_name(int v) {
    // (of a skin list: 128 threads but for the third)
    static const char* names[kForcesVariants] = {"64 threads, 8 entries a round", "128 threads, <=64 regs",
                                                 "256 threads, <=64 regs", "32 threads, 16 entries a round",
                                                 "8 lanes/particle"};
    return v >= 0 && v < kForcesVariants ? names[v] : "?";
}

void launch_dt(const Buffers& b, const Geometry& g, const Phys& ph, int advance_time, cudaStream_t st,
               int with_build) {
    k_dt<<<1, 256, 0, st>>>(dt_args(b, g, ph, advance_time, with_build));
}

// blocks of the persistent step kernel: all resident (a cooperative launch refuses more)
template <int VISC>
int persistent_grid() {
    int dev = 0, sms = 0, per_sm = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_step_persistent<VISC>, kPipeBlock, 0) != cudaSuccess)
        return 0;
    return sms * per_sm;
}

cudaError_t launch_step_persistent(const Buffers& b, int cur, const Geometry& g, const Phys& ph, uint32_t nsteps,
                                   cudaStream_t st) {
    const bool lam = ph.visc == SPH_VISC_LAMINAR;
    const int grid = lam ? persistent_grid<SPH_VISC_LAMINAR>() : persistent_grid<SPH_VISC_ARTIFICIAL>();
    if (grid <= 0) return cudaErrorLaunchFailure;
    Buffers bb = b;
    Geometry gg = g;
    Phys pp = ph;
    int c0 = cur;
    uint32_t ns = nsteps;
    void* args[] = {&bb, &gg, &pp, &c0, &ns};
    const void* fn = lam ? (const void*)k_step_persistent<SPH_VISC_LAMINAR>
                         : (const void*)k_step_persistent<SPH_VISC_ARTIFICIAL>;
    return cudaLaunchCooperativeKernel(fn, dim3((unsigned)grid), dim3(kPipeBlock), args, 0, st);
}

void launch_build_predict(const Buffers& b, int cur, const Geometry& g, const Phys& ph, cudaStream_t st) {
    const auto go = [&](auto kernel, unsigned block) {
        kernel<<<g.cap ? (g.cap + block - 1) / block : 1, block, 0, st>>>(b, cur, ph);
    };
    const bool laminar = ph.visc == SPH_VISC_LAMINAR;
    if (ph.fuse_predict == 256) {
        if (laminar) go(k_build_predict<SPH_VISC_LAMINAR, 256>, 256);
        else go(k_build_predict<SPH_VISC_ARTIFICIAL, 256>, 256);
    } else {
        if (laminar) go(k_build_predict<SPH_VISC_LAMINAR, 128>, 128);
        else go(k_build_predict<SPH_VISC_ARTIFICIAL, 128>, 128);
    }
}

void launch_dt_peek(const Buffers& b, const Phys& ph, cudaStream_t st) {
    k_dt_peek<<<1, 32, 0, st>>>(b.scenes, b.dyn, b.status, ph.h_d, ph.cfl, ph.dt_fixed);
}

void launch_predict_from_forces(const Buffers& b, int cur, const Geometry& g, const Phys& ph, cudaStream_t st) {
    const unsigned grid = g.cap ? (g.cap + 255) / 256 : 1;
    k_predict_from_forces<<<grid, 256, 0, st>>>(b.pos[cur], b.vel[cur], b.force, b.pinfo[cur], b.scenes, b.dyn,
                                                b.status, ph, b.pos_s, b.vel_s, b.phat_s);
}

}  // namespace sphg
