// Pair and bond forces through the Voronoi cells (arXiv 1701.02059, "Force
// Evaluation"): the quad loop over cell v_i, its neighbouring cells v_j, the
// particles of v_i and the particles of v_j, with the lipid cells reused at
// the wider search cutoff for protein pairs and the bond list for linked
// proteins.
//
// GPU design (one CTA of 4 warps per cell; what the search of the step's path
// and the FP64 forces do in its place stands at k_pair_search):
//   1. the mirrors of every neighbouring cell (contiguous after the sort) are
//      staged in shared memory by 1-D bulk async copies (TMA) completing on
//      an mbarrier, then moved into the cell's own frame: an exact int32
//      offset (wrap-around arithmetic) and, for filtering, an FP32 copy
//      (without the wrap) rotated into the cell's tangent frame (normal =
//      mean lipid director);
//   2. the cell's particles are split into compact groups of <= 32 along
//      their longer tangent extent; each group's warps cull the staged
//      particles against the group's bounding box (r_s + band) into a
//      candidate list, then every lane tests the same candidate at once
//      (broadcast reads; in the search the tests of 16 particles and 8
//      candidates are one matrix product) against its own particle,
//      appending hits to a per-lane queue in shared memory;
//   3. queued pairs are evaluated with the exact integer displacement
//      (2^-26 sigma), the type-pair cutoff decided in FP64 inside a 1e-6 sigma
//      band, and the FP32 potential; force and torque on i are
//      accumulated exactly in split integers, so the sum does not depend on
//      the order or on how candidates are split across warps;
//   4. every pair is computed from both sides (no atomics to other cells, as
//      the paper does across patch boundaries); bonds of i are added in the
//      epilogue.
#include "integrator.cuh"

#include <mutex>

namespace orbc {

constexpr int kPairThreads = 128;
constexpr int kStageCap = 624;     // staged particles per pass
constexpr int kQCap = 32;          // queued hits per lane before a flush
constexpr int kMaxNbr = 32;        // neighbouring cells per pass (one per lane of the set-up warp)
constexpr float kFilterBand = 1e-4f;

// ---------------------------------------------------------------- pair terms
// Lipid pair (see the header of orbc.h for the potential).  d = x_j - x_i.
// Returns U; adds force on i and torque on i.
__device__ inline float taylor_cos(float x) {
    // Maclaurin series of cos through x^14 on [0, pi/2]; truncation < 1e-9
    float x2 = x * x;
    float p = -1.1470745597729725e-11f;
    p = fmaf(p, x2, 2.08767569878681e-09f);
    p = fmaf(p, x2, -2.755731922398589e-07f);
    p = fmaf(p, x2, 2.48015873015873e-05f);
    p = fmaf(p, x2, -0.001388888888888889f);
    p = fmaf(p, x2, 0.041666666666666664f);
    p = fmaf(p, x2, -0.5f);
    return fmaf(p, x2, 1.0f);
}
__device__ inline float taylor_sin(float x) {
    // Maclaurin series of sin through x^15 on [0, pi/2]; truncation < 1e-10
    float x2 = x * x;
    float p = -7.647163731819816e-13f;
    p = fmaf(p, x2, 1.6059043836821613e-10f);
    p = fmaf(p, x2, -2.505210838544172e-08f);
    p = fmaf(p, x2, 2.7557319223985893e-06f);
    p = fmaf(p, x2, -0.0001984126984126984f);
    p = fmaf(p, x2, 0.008333333333333333f);
    p = fmaf(p, x2, -0.16666666666666666f);
    return x * fmaf(p, x2, 1.0f);
}

// FP32 lipid pair; Z > 0 fixes zeta at compile time (Z = 0: runtime zeta).
// S0: the spontaneous-curvature term is present (sin theta0 != 0); without
// it the terms in s0 drop out of a, w and the torque.
template <int Z, bool S0 = true, typename IC = Inst>
__device__ inline float lipid_terms_f(const IC& I, float dx, float dy, float dz, float r2, float nix, float niy,
                                      float niz, float njx, float njy, float njz, float& fx, float& fy, float& fz,
                                      float& tx, float& ty, float& tz, float* tj = nullptr) {
    const float rinv = rsqrtf(r2);
    const float r = r2 * rinv;
    // rh = r_ij / r = -(d) / r
    const float hx = -dx * rinv, hy = -dy * rinv, hz = -dz * rinv;
    const float s0 = I.s0;
    const float nin = fmaf(nix, njx, fmaf(niy, njy, niz * njz));
    const float nir = fmaf(nix, hx, fmaf(niy, hy, niz * hz));
    const float njr = fmaf(njx, hx, fmaf(njy, hy, njz * hz));
    const float a = S0 ? fmaf(s0, njr - nir, fmaf(-nir, njr, nin)) - s0 * s0 : fmaf(-nir, njr, nin);
    const float phi = fmaf(I.mu, a - 1.0f, 1.0f);
    float f, fp, g, gp;
    if (r < I.rmin) {
        const float q = I.rmin * rinv;
        const float q2 = q * q, q4 = q2 * q2;
        f = fmaf(I.eps, q4 - 2.0f * q2, I.eps);
        fp = 4.0f * I.eps * rinv * (q2 - q4);
        g = -I.eps;
        gp = 0.0f;
    } else {
        const float th = I.aw * (r - I.rmin);
        const float c = taylor_cos(th), sn = taylor_sin(th);
        // c^(2 zeta - 1) by binary powering from the low bits: the general
        // path forms the same products in the same order as the zeta = 4
        // one, so an instance gives the same bits in a batch that mixes
        // exponents (which takes the general path) as alone
        float cp;
        if (Z == 4) {
            const float c2 = c * c, c4 = c2 * c2;
            cp = (c * c2) * c4;
        } else {
            cp = 1.0f;
            float bp = c;
            for (int e = 2 * I.zeta - 1; e > 0; e >>= 1) {
                if (e & 1) cp *= bp;
                bp *= bp;
            }
        }
        f = 0.0f;
        fp = 0.0f;
        g = -I.eps * cp * c;
        gp = I.eps2z_aw * cp * sn;
    }
    const float U = fmaf(g, phi, f);
    float wx = fmaf(-njr, nix, -nir * njx), wy = fmaf(-njr, niy, -nir * njy), wz = fmaf(-njr, niz, -nir * njz);
    if (S0) {
        wx = fmaf(s0, njx - nix, wx);
        wy = fmaf(s0, njy - niy, wy);
        wz = fmaf(s0, njz - niz, wz);
    }
    const float wr = fmaf(wx, hx, fmaf(wy, hy, wz * hz));
    const float radial = fmaf(gp, phi, fp);
    const float gm = g * I.mu;
    const float gmr = gm * rinv;
    fx += -radial * hx - gmr * fmaf(-wr, hx, wx);
    fy += -radial * hy - gmr * fmaf(-wr, hy, wy);
    fz += -radial * hz - gmr * fmaf(-wr, hz, wz);
    // da/dn_i = n_j - (n_j.rh + s0) rh ; tau_i = -g mu (n_i x da/dn_i)
    const float js = S0 ? njr + s0 : njr;
    const float gx = fmaf(-js, hx, njx), gy = fmaf(-js, hy, njy), gz = fmaf(-js, hz, njz);
    tx += -gm * (niy * gz - niz * gy);
    ty += -gm * (niz * gx - nix * gz);
    tz += -gm * (nix * gy - niy * gx);
    if (tj) {
        // da/dn_j = n_i - (n_i.rh - s0) rh ; tau_j = -g mu (n_j x da/dn_j)
        const float is = nir - s0;
        const float ux = fmaf(-is, hx, nix), uy = fmaf(-is, hy, niy), uz = fmaf(-is, hz, niz);
        tj[0] = -gm * (njy * uz - njz * uy);
        tj[1] = -gm * (njz * ux - njx * uz);
        tj[2] = -gm * (njx * uy - njy * ux);
    }
    return U;
}

// WCA; d = x_j - x_i; adds the force on i.  pp: protein-protein size.
__device__ inline float wca_terms(const Inst& I, bool pp, float dx, float dy, float dz, float r2, float& fx, float& fy,
                                  float& fz) {
    const float sig = pp ? I.sig_pp : I.sig_wca;
    const float e = I.eps_wca;
    const float s2 = sig * sig / r2;
    const float s6 = s2 * s2 * s2;
    const float s12 = s6 * s6;
    const float fr = 4.0f * e * (12.0f * s12 - 6.0f * s6) / r2;
    fx -= fr * dx;
    fy -= fr * dy;
    fz -= fr * dz;
    return 4.0f * e * (s12 - s6) + e;
}

// ---------------------------------------------------------------- accumulators
struct Acc {
    // fast path: split int32 sums (|component sum| < 1000); wider values go
    // to an int64 side array with atomics (exact, rare)
    SplitAcc f[3], t[3];
    int nf, nt;
    bool used_big;
    __device__ void zero() { for (int a = 0; a < 3; a++) { f[a].zero(); t[a].zero(); } nf = 0; nt = 0; used_big = false; }
    __device__ void add3(const View& v, int p, SplitAcc* s, int& n, int c0, float x, float y, float z) {
        const float mag = fabsf(x) + fabsf(y) + fabsf(z);
        if (mag < 1000.0f) { s[0].add(x); s[1].add(y); s[2].add(z); n++; return; }
        // NaN, infinite, or a term beyond the range the 2^-32 fixed-point
        // sums hold (|component| < 2^31 after a few hundred terms)
        if (!(mag < kMaxTerm))
            flag_inst(v, v.inst[find_inst(v.inst_p0, v.B, p)], (mag == mag) ? kStatusPairForceRange : kStatusNaN);
        const size_t N = v.N;
        atomicAdd((unsigned long long*)&v.Fbig[(size_t)c0 * N + p], (unsigned long long)__float2ll_rn(x * 4294967296.0f));
        atomicAdd((unsigned long long*)&v.Fbig[(size_t)(c0 + 1) * N + p], (unsigned long long)__float2ll_rn(y * 4294967296.0f));
        atomicAdd((unsigned long long*)&v.Fbig[(size_t)(c0 + 2) * N + p], (unsigned long long)__float2ll_rn(z * 4294967296.0f));
        used_big = true;
    }
    __device__ void add_pair(const View& v, int p, float fx, float fy, float fz, float tx, float ty, float tz) {
        add3(v, p, f, nf, 0, fx, fy, fz);
        add3(v, p, t, nt, 3, tx, ty, tz);
    }
};
// exact FP64 inclusion decision for a pair inside the cutoff band; m: the
// bilayer species pair (cls 0)
__device__ inline bool exact_inside(const View& v, const Inst& I, int pi, int pj, int cls, int m = 0) {
    size_t N = v.N;
    double d2 = dist2_grid_d(v.xq[pj], v.xq[N + pj], v.xq[2 * N + pj], v.xq[pi], v.xq[N + pi], v.xq[2 * N + pi], I);
    return d2 < (cls == 0 ? I.mm_rc2[m] : (cls == 1 ? I.rc2_wca : I.rc2_pp));
}

// Pair class of two types: 0 two bilayer particles (the lipid potential), 1
// a bilayer particle and a cytoskeleton protein, 2 two cytoskeleton proteins
// (both WCA); m: the bilayer species pair 3 s_i + s_j of class 0.
__device__ inline int pair_class(int ti, int tj, int& m) {
    const bool bi = bilayer(ti), bj = bilayer(tj);
    m = (bi && bj) ? 3 * species(ti) + species(tj) : 0;
    return (bi && bj) ? 0 : ((bi || bj) ? 1 : 2);
}

// The lipid potential's FP32 constants of one bilayer species pair, in the
// field names of Inst, for the pair-term functions.
struct LipK {
    float eps, rmin, mu, s0, aw, eps2z_aw;
    int zeta;
    __device__ LipK(const Inst& I, int m)
        : eps(I.mm_eps[m]), rmin(I.rmin), mu(I.mu), s0(I.s0), aw(I.mm_aw[m]), eps2z_aw(I.mm_e2za[m]), zeta(I.zeta) {}
};

// 1-2 and 1-3 bonded pairs carry no excluded-volume term (bonded directly,
// or sharing a bond partner).  Ids are local to i's instance I; slot pj
// outside I (the partner cell set of a membrane, which no bond reaches) is
// never excluded.
__device__ inline bool is_excluded(const View& v, const Inst& I, unsigned idi, unsigned idj, int pj) {
    if ((unsigned)(pj - I.p0) >= (unsigned)I.n) return false;
    const int s = v.bptr[I.p0 + idi], e = v.bptr[I.p0 + idi + 1];
    const int s2 = v.bptr[I.p0 + idj], e2 = v.bptr[I.p0 + idj + 1];
    for (int q = s; q < e; q++) {
        const int c = v.bpartner[q];
        if ((unsigned)c == idj) return true;
        for (int w = s2; w < e2; w++)
            if (v.bpartner[w] == c) return true;
    }
    return false;
}

// ---------------------------------------------------------------- TMA helpers
__device__ inline unsigned smem_addr(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }

__device__ inline void mbar_init(unsigned long long* bar, unsigned count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ inline void mbar_expect_tx(unsigned long long* bar, unsigned bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes) : "memory");
}
__device__ inline void bulk_g2s(void* dst, const void* src, unsigned bytes, unsigned long long* bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(smem_addr(dst)),
        "l"(src), "r"(bytes), "r"(smem_addr(bar))
        : "memory");
}
__device__ inline bool mbar_try_wait(unsigned long long* bar, unsigned phase) {
    unsigned ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(smem_addr(bar)), "r"(phase)
        : "memory");
    return ok != 0;
}
// Bounded wait: gives up after `polls` polls (2^22 by default: with the
// back-off, well over a second), records a timeout in the status word and
// returns false.
__device__ inline bool mbar_wait_bounded(unsigned long long* bar, unsigned phase, unsigned* status,
                                         unsigned polls) {
    for (unsigned it = 0; it < polls; it++) {
        if (mbar_try_wait(bar, phase)) return true;
        if (it > 64) __nanosleep(256);
    }
    atomicOr(status, kStatusTimeout);
    return false;
}

// the cell's tangent frame (prepared with the cell radii)
__device__ inline Frame load_frame(const View& v, int k) {
    const float4 a = __ldg(v.cframe + 3 * (size_t)k), b = __ldg(v.cframe + 3 * (size_t)k + 1),
                 c = __ldg(v.cframe + 3 * (size_t)k + 2);
    Frame f;
    f.r[0] = a.x; f.r[1] = a.y; f.r[2] = a.z;
    f.r[3] = b.x; f.r[4] = b.y; f.r[5] = b.z;
    f.r[6] = c.x; f.r[7] = c.y; f.r[8] = c.z;
    return f;
}

// extremes over the warp in one instruction each
__device__ inline float warp_min_f32(float x) {
    float r;
    asm("redux.sync.min.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(x));
    return r;
}
__device__ inline float warp_max_f32(float x) {
    float r;
    asm("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(x));
    return r;
}

// ---------------------------------------------------------------- the kernel
struct NbrInfo {
    int base;       // first staged index
    int cnt;
    int start;      // global slot of the first particle
    int ox, oy, oz; // exact offset c_l - c_k at 2^-26 sigma (wrap-around int32)
    float fx, fy, fz;   // the same without the wrap, in sigma (FP32)
};

template <bool S0, typename IC = Inst>
__device__ inline float lipid_dispatch(const IC& I, float dx, float dy, float dz, float r2, float nix, float niy, float niz,
                                       float njx, float njy, float njz, float& fx, float& fy, float& fz, float& tx,
                                       float& ty, float& tz, int zc, float* tj) {
    if (zc == 4)
        return lipid_terms_f<4, S0, IC>(I, dx, dy, dz, r2, nix, niy, niz, njx, njy, njz, fx, fy, fz, tx, ty, tz, tj);
    return lipid_terms_f<0, true, IC>(I, dx, dy, dz, r2, nix, niy, niz, njx, njy, njz, fx, fy, fz, tx, ty, tz, tj);
}

// S0: some instance has a spontaneous-curvature term (s0 != 0).
template <bool ENERGY, bool DUMP, int Z, bool S0>
__global__ void __launch_bounds__(kPairThreads, 5) k_pairs(View v, long long* __restrict__ energy /* [B][8] */,
                                                            unsigned* __restrict__ dump,
                                                            unsigned long long* __restrict__ dump_count,
                                                            long long dump_cap) {
    // sy: staged mirrors, after staging in the cell-k frame (exact int32,
    //     2^-26 sigma), w = type
    // sY: the same particles in FP32, rotated into the tangent frame
    // so: directors, w = global slot
    __shared__ alignas(16) int4 sy[kStageCap];
    __shared__ alignas(16) float4 sY[kStageCap];
    __shared__ alignas(16) float4 so[kStageCap];
    __shared__ alignas(16) unsigned short cand[kPairThreads / 32][kStageCap];   // per-warp candidate list
    __shared__ unsigned short qbuf[kPairThreads / 32][kQCap][32];   // per-lane hit queues
    __shared__ NbrInfo nb[kMaxNbr];
    __shared__ unsigned long long bar;
    __shared__ int s_nstage, s_next, s_next_off, s_self, s_self_lo, s_self_hi, s_total;

    const int k = blockIdx.x;
    const int b = find_inst(v.inst_k0, v.B, k);
    const Inst& I = v.inst[b];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int cs = v.cell_start[k], ce = v.cell_start[k + 1];
    // the cell's neighbour row (fixed stride; rows longer than kAdjRow are
    // flagged by the adjacency pass)
    const AdjDesc* __restrict__ row = v.adjd + (size_t)k * kAdjRow;
    const int a0 = 0;
    const int a1 = min(v.adjn[k], kAdjRow);
    const float rs_b = I.rsf + kFilterBand;
    const float rs2f = rs_b * rs_b;
    const float rcl = sqrtf(I.rc2f_ll), rcw = sqrtf(I.rc2f_wca), rcp = sqrtf(I.rc2f_pp);
    const float ll_lo = (rcl - kCutBand) * (rcl - kCutBand), ll_hi = (rcl + kCutBand) * (rcl + kCutBand);
    const float w_lo = (rcw - kCutBand) * (rcw - kCutBand), w_hi = (rcw + kCutBand) * (rcw + kCutBand);
    const float p_lo = (rcp - kCutBand) * (rcp - kCutBand), p_hi = (rcp + kCutBand) * (rcp + kCutBand);
    const size_t N = v.N;
    const int zc = (Z > 0) ? Z : I.zeta;
    unsigned phase = 0;
    if (tid == 0) mbar_init(&bar, 1);
    __syncthreads();

    for (int it0 = cs; it0 < ce; it0 += kPairThreads) {
        const int nti = min(kPairThreads, ce - it0);            // particles of this i-tile
        const int groups = (nti + 31) >> 5;                     // compact groups of <= 32
        const int nsplit = (groups == 1) ? 4 : (groups == 2 ? 2 : 1);
        const int igrp = warp % groups;
        const int jsplit = warp / groups;
        const bool wactive = jsplit < nsplit;
        const int gs = (nti + groups - 1) / groups;             // balanced group size

        // staging of one pass (warp 0): neighbour descriptors, bulk copies
        auto issue = [&](const int na, const int na_off) {
                if (warp == 0) {
                    // one lane per neighbouring cell: counts, offsets, staging slots
                    const int nn = na + lane;
                    const bool has = nn < a1;
                    int l = 0, st = 0, c = 0;
                    AdjDesc d;
                    if (has) {
                        d = row[nn];
                        l = d.cell();
                        st = d.start;
                        c = d.cnt;
                        if (lane == 0) { st += na_off; c -= na_off; }
                    }
                    int incl = c;
                    for (int off = 1; off < 32; off <<= 1) {
                        const int t = __shfl_up_sync(0xffffffffu, incl, off);
                        if (lane >= off) incl += t;
                    }
                    const int excl = incl - c;
                    const bool fits = has && incl <= kStageCap;
                    const bool part = has && excl < kStageCap && incl > kStageCap;
                    const unsigned fm = __ballot_sync(0xffffffffu, fits), pm = __ballot_sync(0xffffffffu, part);
                    const int m = __popc(fm) + (pm ? 1 : 0);
                    const bool staged = fits || part;
                    const int take = part ? kStageCap - excl : c;
                    if (staged) {
                        NbrInfo inf;
                        inf.base = excl; inf.cnt = take; inf.start = st;
                        inf.ox = d.ox; inf.oy = d.oy; inf.oz = d.oz;
                        whole_offset(d, inf.fx, inf.fy, inf.fz);
                        nb[lane] = inf;
                    }
                    const unsigned selfm = __ballot_sync(0xffffffffu, staged && l == k);
                    const int total = __shfl_sync(0xffffffffu, excl + take, max(m - 1, 0));
                    // where the next pass starts: after the last fully staged
                    // neighbour, or inside the partially staged one
                    int nxt = na + __popc(fm), nxo = 0;
                    if (pm) {
                        const int p = __ffs(pm) - 1;
                        const int ex_p = __shfl_sync(0xffffffffu, excl, p);
                        nxt = na + p;
                        nxo = (p == 0 ? na_off : 0) + (kStageCap - ex_p);
                    }
                    // staged range of the own cell, and where its first particle would sit
                    int slo = -1, shi = -1, sb = 0;
                    {
                        const int p = selfm ? __ffs(selfm) - 1 : 0;
                        const int ex_p = __shfl_sync(0xffffffffu, excl, p);
                        const int tk_p = __shfl_sync(0xffffffffu, take, p);
                        if (selfm) {
                            slo = ex_p;
                            shi = ex_p + tk_p;
                            sb = ex_p - ((p == 0) ? na_off : 0);
                        }
                    }
                    if (lane == 0) {
                        s_nstage = m;
                        s_total = m > 0 ? total : 0;
                        s_next = nxt;
                        s_next_off = nxo;
                        s_self = sb; s_self_lo = slo; s_self_hi = shi;
                    }
                    if (m > 0) {
                        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                        if (lane == 0) mbar_expect_tx(&bar, (unsigned)total * 32u + v.extra_tx);
                        __syncwarp();
                        if (staged && take > 0) {
                            bulk_g2s(&sy[excl], v.mqr + st, take * 16u, &bar);
                            bulk_g2s(&so[excl], v.mor + st, take * 16u, &bar);
                        }
                    }
                }
        };
        // the first pass's copies are in flight during the tile set-up
        if (a0 < a1) issue(a0, 0);

        // ---- tangent frame of the cell; the mirrors of each tile of 128 are
        //      stored in the order of their rank along the tile's longer
        //      tangent extent (prepared with the cell radii), so that the
        //      group of rank range [g gs, (g + 1) gs) is compact
        const Frame F = load_frame(v, k);

        // ---- this lane's particle: rank r of the tile, slot pi
        const int r = igrp * gs + lane;
        const bool ivalid = wactive && lane < gs && r < nti;
        int ti = 0, pi = -1;
        int4 qi = make_int4(0, 0, 0, 0);
        float4 oi = make_float4(0, 0, 0, 0);
        float yix = 0.f, yiy = 0.f, yiz = 0.f;
        unsigned idi = 0;
        if (ivalid) {
            qi = v.mqr[it0 + r];
            oi = v.mor[it0 + r];
            pi = __float_as_int(oi.w);
            ti = qi.w & 0xff;
            F.apply(qi.x * kMirrorUnit, qi.y * kMirrorUnit, qi.z * kMirrorUnit, yix, yiy, yiz);
            if (DUMP) idi = (unsigned)I.id_base + v.id[pi];
        }
        // a lane without a particle sits far away: it passes no distance test
        if (!ivalid) { yix = 1.0e18f; yiy = 1.0e18f; yiz = 1.0e18f; }
        // group bounding box in the tangent frame, widened by the search radius
        float blo[3] = {ivalid ? yix : 3.0e38f, ivalid ? yiy : 3.0e38f, ivalid ? yiz : 3.0e38f};
        float bhi[3] = {ivalid ? yix : -3.0e38f, ivalid ? yiy : -3.0e38f, ivalid ? yiz : -3.0e38f};
        for (int a = 0; a < 3; a++) { blo[a] = warp_min_f32(blo[a]); bhi[a] = warp_max_f32(bhi[a]); }
        Acc acc;
        acc.zero();
        double up = 0, vir = 0;     // per-particle energy and virial partials, FP64 in every mode

        // passes over chunks of neighbouring cells (a cell larger than the
        // stage is split across passes)
        bool first_pass = true;
        for (int na = a0, na_off = 0; na < a1;) {
            if (!first_pass) {
                __syncthreads();
                issue(na, na_off);
            }
            first_pass = false;
            __syncthreads();
            const int m = s_nstage;
            const int total = s_total;
            const int next = s_next, next_off = s_next_off;
            if (m == 0) { na = next; na_off = next_off; continue; }
            const int sself = s_self, sslo = s_self_lo, sshi = s_self_hi;
            int selfj = (sslo >= 0 && ivalid) ? sself + (it0 + r - cs) : -1;
            if (selfj < sslo || selfj >= sshi) selfj = -1;
            bool ok = mbar_wait_bounded(&bar, phase, v.status, v.wait_polls);
            if (__syncthreads_or(!ok)) {
                // give the copies in flight a second bounded wait, then leave
                if (ok == false) mbar_wait_bounded(&bar, phase, v.status, v.wait_polls);
                return;
            }
            phase ^= 1u;

            // ---- staged particles into the cell-k frame (exact) and the
            //      tangent frame (FP32)
            for (int q = 0; q < m; q++) {
                const NbrInfo inf = nb[q];
                for (int j = inf.base + tid; j < inf.base + inf.cnt; j += kPairThreads) {
                    int4 rj = sy[j];
                    float4 y;
                    F.apply(fmaf((float)rj.x, kMirrorUnit, inf.fx), fmaf((float)rj.y, kMirrorUnit, inf.fy),
                            fmaf((float)rj.z, kMirrorUnit, inf.fz), y.x, y.y, y.z);
                    rj.x = (int)((unsigned)rj.x + (unsigned)inf.ox);
                    rj.y = (int)((unsigned)rj.y + (unsigned)inf.oy);
                    rj.z = (int)((unsigned)rj.z + (unsigned)inf.oz);
                    sy[j] = rj;
                    y.w = 0.f;
                    sY[j] = y;
                }
            }
            __syncthreads();

            if (wactive) {
                // ---- candidates: staged particles within r_s (+ band) of the
                //      group's box; the warps of a group take every nsplit-th
                //      staged particle, so that their shares of the candidates
                //      and hits stay even (whole chunks per warp left them
                //      waiting on each other at the next barrier)
                int cnt = 0;
                for (int c0 = 0; c0 < total; c0 += nsplit * 32) {
                    const int j = c0 + lane * nsplit + jsplit;
                    bool in = false;
                    if (j < total) {
                        const float4 y = sY[j];
                        const float ex = fmaxf(fmaxf(blo[0] - y.x, y.x - bhi[0]), 0.f);
                        const float ey = fmaxf(fmaxf(blo[1] - y.y, y.y - bhi[1]), 0.f);
                        const float ez = fmaxf(fmaxf(blo[2] - y.z, y.z - bhi[2]), 0.f);
                        in = fmaf(ex, ex, fmaf(ey, ey, ez * ez)) < rs2f;
                    }
                    const unsigned bal = __ballot_sync(0xffffffffu, in);
                    if (in) cand[warp][cnt + __popc(bal & ((1u << lane) - 1u))] = (unsigned short)j;
                    cnt += __popc(bal);
                }
                __syncwarp();

                int qn = 0;
                auto flush = [&]() {
                    int qmax = qn;
                    for (int off = 16; off; off >>= 1) qmax = max(qmax, __shfl_xor_sync(0xffffffffu, qmax, off));
                    for (int t = 0; t < qmax; t++) {
                        if (t >= qn) continue;
                        const int j = (int)qbuf[warp][t][lane];
                        const int4 mj = sy[j];
                        const float4 oj = so[j];
                        const int pj = __float_as_int(oj.w);
                        const int tj = mj.w & 0xff;
                        int m;
                        const int cls = pair_class(ti, tj, m);
                        const bool ll = cls == 0;
                        const int dxq = (int)((unsigned)mj.x - (unsigned)qi.x);
                        const int dyq = (int)((unsigned)mj.y - (unsigned)qi.y);
                        const int dzq = (int)((unsigned)mj.z - (unsigned)qi.z);
                        const float dxf = (float)dxq * kMirrorUnit, dyf = (float)dyq * kMirrorUnit,
                                    dzf = (float)dzq * kMirrorUnit;
                        const float r2f = fmaf(dxf, dxf, fmaf(dyf, dyf, dzf * dzf));
                        const float lo = cls == 0 ? (I.has_mp ? I.mm_lo[m] : ll_lo) : (cls == 1 ? w_lo : p_lo);
                        const float hi = cls == 0 ? (I.has_mp ? I.mm_hi[m] : ll_hi) : (cls == 1 ? w_hi : p_hi);
                        if (r2f >= hi) continue;
                        bool in = r2f < lo;
                        if (!in) in = exact_inside(v, I, pi, pj, cls, m);
                        if (in && cls != 0 && is_excluded(v, I, v.id[pi], v.id[pj], pj)) in = false;
                        if (!in) continue;
                        float fx = 0, fy = 0, fz = 0, tx = 0, ty = 0, tz = 0, U;
                        const float dx = dxf, dy = dyf, dz = dzf, r2 = r2f;
                        if (ll && I.has_mp)
                            U = lipid_dispatch<S0, LipK>(LipK(I, m), dx, dy, dz, r2, oi.x, oi.y, oi.z, oj.x, oj.y, oj.z, fx,
                                                         fy, fz, tx, ty, tz, zc, (float*)nullptr);
                        else if (ll)
                            U = lipid_dispatch<S0>(I, dx, dy, dz, r2, oi.x, oi.y, oi.z, oj.x, oj.y, oj.z, fx, fy, fz, tx, ty,
                                                   tz, zc, (float*)nullptr);
                        else
                            U = wca_terms(I, cls == 2, dx, dy, dz, r2, fx, fy, fz);
                        acc.add_pair(v, pi, fx, fy, fz, tx, ty, tz);
                        if (ENERGY) {
                            up += 0.5 * (double)U;
                            vir += -0.5 * ((double)dx * (double)fx + (double)dy * (double)fy + (double)dz * (double)fz);
                        }
                        if (DUMP) {
                            const unsigned idj =
                                (unsigned)v.inst[find_inst(v.inst_p0, v.B, pj)].id_base + v.id[pj];
                            if (idi < idj) {
                                unsigned long long slot = atomicAdd(dump_count, 1ull);
                                if ((long long)slot < dump_cap) { dump[2 * slot] = idi; dump[2 * slot + 1] = idj; }
                            }
                        }
                    }
                    qn = 0;
                    __syncwarp();
                };
                // ---- every lane tests the same candidate (broadcast reads)
                static_assert(kStageCap % 8 == 0, "candidate lists are read 8 at a time");
                for (int c = 0; c < cnt; c += 8) {
                    if (__any_sync(0xffffffffu, qn > kQCap - 8)) flush();
                    const uint4 c8 = *reinterpret_cast<const uint4*>(&cand[warp][c]);   // 8 indices, broadcast
                    const unsigned cw[4] = {c8.x, c8.y, c8.z, c8.w};
#pragma unroll
                    for (int u = 0; u < 8; u++) {
                        if (c + u < cnt) {
                            const int j = (int)((cw[u >> 1] >> (16 * (u & 1))) & 0xffffu);
                            const float4 y = sY[j];
                            const float ex = y.x - yix, ey = y.y - yiy, ez = y.z - yiz;
                            const float d2 = fmaf(ex, ex, fmaf(ey, ey, ez * ez));
                            if (d2 < rs2f && j != selfj) { qbuf[warp][qn][lane] = (unsigned short)j; qn++; }
                        }
                    }
                }
                flush();
            }
            na = next;
            na_off = next_off;
        }

        // combine the warps of a group (exact integer sums) and write; rows
        // are indexed by the rank r.  The red rows of the later splits
        // ((nsplit - 1) x nti <= 96 rows of 56 bytes) fit in sY, which no
        // warp reads any more.
        __syncthreads();
        {
            // the warps of a group hold partial sums of the same particles:
            // the later splits hand theirs over by plain stores, split 0 adds
            // them and writes the particle
            static_assert(3 * 32 * 14 * sizeof(int) <= kStageCap * sizeof(float4), "split rows must fit in sY");
            int (*red)[14] = reinterpret_cast<int (*)[14]>(&sY[0]);
            if (ivalid && jsplit > 0) {
                int* d = red[(jsplit - 1) * nti + r];
                d[0] = acc.f[0].h; d[1] = acc.f[0].l; d[2] = acc.f[1].h; d[3] = acc.f[1].l;
                d[4] = acc.f[2].h; d[5] = acc.f[2].l; d[6] = acc.t[0].h; d[7] = acc.t[0].l;
                d[8] = acc.t[1].h; d[9] = acc.t[1].l; d[10] = acc.t[2].h; d[11] = acc.t[2].l;
                d[12] = acc.nf; d[13] = acc.nt;
            }
            const bool any_big = __syncthreads_or(ivalid && acc.used_big);
            if (ivalid && jsplit == 0) {
                int sm[14] = {acc.f[0].h, acc.f[0].l, acc.f[1].h, acc.f[1].l, acc.f[2].h, acc.f[2].l,
                              acc.t[0].h, acc.t[0].l, acc.t[1].h, acc.t[1].l, acc.t[2].h, acc.t[2].l, acc.nf, acc.nt};
                for (int q = 1; q < nsplit; q++) {
                    const int* d = red[(q - 1) * nti + r];
    #pragma unroll
                    for (int c = 0; c < 14; c++) sm[c] += d[c];
                }
                const int p = pi;
    #pragma unroll
                for (int a = 0; a < 3; a++) {
                    SplitAcc f; f.h = sm[2 * a]; f.l = sm[2 * a + 1];
                    SplitAcc t; t.h = sm[6 + 2 * a]; t.l = sm[6 + 2 * a + 1];
                    long long fb = 0, tb = 0;
                    if (any_big) {
                        fb = __ldcg(&v.Fbig[(size_t)a * N + p]);
                        tb = __ldcg(&v.Fbig[(size_t)(3 + a) * N + p]);
                        v.Fbig[(size_t)a * N + p] = 0; v.Fbig[(size_t)(3 + a) * N + p] = 0;
                    }
                    v.F[a * N + p] = f.finish(sm[12]) + fb;
                    v.T[a * N + p] = t.finish(sm[13]) + tb;
                }
            }
        }
        if (ENERGY) {
            // per-particle energies to fixed point, exact integer sums per instance
            long long eu = 0, ew = 0;
            if (ivalid) {
                eu = __double2ll_rn(up * 4294967296.0);
                ew = __double2ll_rn(vir * 4294967296.0);
            }
            for (int off = 16; off; off >>= 1) {
                eu += __shfl_xor_sync(0xffffffffu, eu, off);
                ew += __shfl_xor_sync(0xffffffffu, ew, off);
            }
            if (lane == 0) {
                atomicAdd((unsigned long long*)&energy[b * 8 + 0], (unsigned long long)eu);
                atomicAdd((unsigned long long*)&energy[b * 8 + 4], (unsigned long long)ew);
            }
        }
        __syncthreads();
    }
}

// ================================================================ split pair path
// The quad loop in two launches: a per-cell search that lists, for every
// particle, the staged particles of its neighbouring cells within its
// type-pair cutoff (+ two skins + a rounding band), and an evaluation with
// one thread per particle over its list, which takes the exact inclusion
// decision and the pair terms.  The search keeps only what the filter needs
// (no evaluation, queues or combine), so it runs with more resident warps;
// the evaluation has no barriers and full lanes.  Forces are the same exact
// integer sums as in the one-launch kernel, whatever order the list holds.
//
// List entry: (row << 26) | q, where q indexes the rank-ordered mirrors (in a
// batch of more than 2^26 particles from the membrane's first slot on: FAR; a
// membrane has no more, see Ensemble::setup) and row is the neighbouring cell's
// place in the row of the particle's cell, whose exact offset c_l - c_k the
// search writes to rowoff.  Lists hold
// kListCap entries per particle (t-major: entry t of particle q at t N + q);
// further entries go to an overflow list evaluated with integer atomics.
constexpr int kSearchStage = 640;
constexpr int kFragRow = 12;        // floats between fragment rows (48 B: no bank conflicts)
constexpr int kListCap = 32;
constexpr int kRowShift = kListBits;

// The slot that the list entries of instance I count from in a FAR batch: the
// first one of its membrane (of both its cell sets).  A form of its own: in
// every batch, one more register and addition a pair make the steps of 400,000
// particles in twelve membranes 1 per cent slower.
inline __host__ __device__ bool far_batch(int N) { return N > 1 << kListBits; }
__device__ inline int list_base(const View& v, const Inst& I) {
    return I.partner < 0 ? I.p0 : min(I.p0, v.inst[I.partner].p0);
}

struct SNbr {
    int base, cnt, start, row;
    float ox, oy, oz;       // c_l - c_k without the wrap, in sigma
};

// The FP32 constants of the pair terms, held in registers by the evaluation.
struct PairC {
    float eps, rmin, mu, s0, aw, eps2z_aw, eps_wca, sig_wca, sig_pp;
    int zeta;
    float ll_lo, ll_hi, w_lo, w_hi, p_lo, p_hi;   // squared cutoffs -+ the FP64 decision band
    __device__ explicit PairC(const Inst& I)
        : eps(I.eps), rmin(I.rmin), mu(I.mu), s0(I.s0), aw(I.aw), eps2z_aw(I.eps2z_aw), eps_wca(I.eps_wca),
          sig_wca(I.sig_wca), sig_pp(I.sig_pp), zeta(I.zeta), ll_lo(I.ll_lo), ll_hi(I.ll_hi), w_lo(I.w_lo), w_hi(I.w_hi),
          p_lo(I.p_lo), p_hi(I.p_hi) {}
};

// ================================================================ FP64 pair forces
// The quad loop with FP64 terms: the neighbour search below (its DIRECT form)
// evaluates the pairs it finds instead of listing them.  GB300 issues one
// FP64 instruction per 16 cycles and SM, so it is bound by their number:
//   - each pair is evaluated once, by the particle of the lower id (so the
//     result does not depend on the cell list), and both sides get their
//     force and torque as 2^-32 integers by atomics: integer sums, any order;
//   - a warp collects its interacting pairs in shared memory (integer and
//     FP32 work) and evaluates 32 at a time, with all lanes full (no list, so
//     no limit to the partners of a particle either);
//   - the terms are arranged for few FP64 operations (about 120 a pair): one
//     reciprocal square root by a third-order step from the FP32 one, no
//     division, sine and cosine from their series about pi/4, positions and
//     directors in grid units with the powers of two folded into constants.
// The one-launch kernel that it replaces (both sides, six divisions, sqrt and
// sincos per pair, lanes idle when their queues ran dry) took 6.30 ms for the
// 250k vesicle, this one 0.54 ms, its FP64 pipe 81% busy; 55.0 and 9.4 ms for the 4M
// cell.
constexpr int kQueue64 = 64;      // a warp's queued pairs: fewer than 32 left over and up to 32 new ones
constexpr double kTwo40 = 1099511627776.0, kTwo80 = kTwo40 * kTwo40;
constexpr double kTwo32 = 4294967296.0;

// 1/sqrt(x) for 0 < x < 2^127: y from the FP32 estimate (error below 2^-21)
// with the third-order step y (1 + e/2 + 3 e^2/8), e = 1 - x y^2 (error e^3).
__device__ inline double rsqrt_d(double x) {
    const double y = (double)rsqrtf((float)x);
    const double e = fma(-(x * y), y, 1.0);
    return fma(y * e, fma(e, 0.375, 0.5), y);
}

// sine and cosine of pi/4 + x, |x| <= pi/4: Maclaurin series through x^15 and
// x^16 (truncation below 5e-17), combined by the addition theorem.
__device__ inline void sincos_quarter(double x, double& s, double& c) {
    const double x2 = x * x;
    double p = -7.6471637318198164759e-13;          // -1/15!
    p = fma(p, x2, 1.6059043836821614599e-10);      // 1/13!
    p = fma(p, x2, -2.5052108385441718775e-08);     // -1/11!
    p = fma(p, x2, 2.7557319223985890653e-06);      // 1/9!
    p = fma(p, x2, -1.9841269841269841270e-04);     // -1/7!
    p = fma(p, x2, 8.3333333333333333333e-03);      // 1/5!
    p = fma(p, x2, -1.6666666666666666667e-01);     // -1/3!
    const double sx = fma(p * x2, x, x);
    double q = 4.7794773323873852974e-14;           // 1/16!
    q = fma(q, x2, -1.1470745597729724714e-11);     // -1/14!
    q = fma(q, x2, 2.0876756987868098979e-09);      // 1/12!
    q = fma(q, x2, -2.7557319223985890653e-07);     // -1/10!
    q = fma(q, x2, 2.4801587301587301587e-05);      // 1/8!
    q = fma(q, x2, -1.3888888888888888889e-03);     // -1/6!
    q = fma(q, x2, 4.1666666666666666667e-02);      // 1/4!
    q = fma(q, x2, -0.5);
    const double cx = fma(q, x2, 1.0);
    const double h = 0.70710678118654752440;        // sqrt(1/2)
    s = h * (cx + sx);
    c = h * (cx - sx);
}

// One interacting pair from the side of pi: d = x_j - x_i and the directors in
// grid units.  F on i (the reaction is its negative) and the torques on both,
// as 2^-32 fixed point before rounding; the potential energy when EN.
template <bool Z4, bool S0, bool EN>
__device__ inline void pair_terms_d(const Inst& I, int cls, int m, const double D[3], const double A[3], const double B[3],
                                    double f[3], double ti[3], double tj[3], double& U) {
    const double R2 = fma(D[2], D[2], fma(D[1], D[1], D[0] * D[0]));
    const double ri = rsqrt_d(R2 * (1.0 / kTwo80)) * (1.0 / kTwo40);      // 1/r, grid units
    if (cls != 0) {
        const double sig = cls == 2 ? I.sig_pp_d : I.sig_wca_d, e = I.eps_wca_d;
        const double i2 = ri * ri, s2 = (sig * sig * kTwo80) * i2;
        const double s6 = s2 * s2 * s2;
        const double K = (-48.0 * e * kTwo32 * kTwo40) * (s6 * (s6 - 0.5)) * i2;
        for (int a = 0; a < 3; a++) { f[a] = K * D[a]; ti[a] = 0.0; tj[a] = 0.0; }
        U = EN ? fma(4.0 * e, s6 * (s6 - 1.0), e) : 0.0;
        return;
    }
    const double r = R2 * ri;                                             // grid units
    const double h[3] = {-D[0] * ri, -D[1] * ri, -D[2] * ri};
    const double nn = fma(A[2], B[2], fma(A[1], B[1], A[0] * B[0]));      // n_i.n_j 2^80
    const double ir = fma(A[2], h[2], fma(A[1], h[1], A[0] * h[0]));      // n_i.h 2^40
    const double jr = fma(B[2], h[2], fma(B[1], h[1], B[0] * h[0]));
    const double s0 = S0 ? I.s0_d * kTwo40 : 0.0;
    double av = fma(-ir, jr, nn);                                         // a 2^80
    if (S0) av += fma(s0, jr - ir, -s0 * s0);
    const double mu = I.mu_d;
    const double phi = fma(mu * (1.0 / kTwo80), av, 1.0 - mu);
    const double eps = I.mm_eps_d[m];
    double g, rad;                                                        // g, (f' + g' phi) 2^32
    double fu = 0.0;
    if (r < I.rmin_d * kTwo40) {
        const double q = (I.rmin_d * kTwo40) * ri, q2 = q * q;
        rad = (4.0 * eps * kTwo32 * kTwo40) * ri * fma(-q2, q2, q2);
        if (EN) fu = fma(eps, fma(q2, q2, -2.0 * q2), eps);
        g = -eps;
    } else {
        const double w = I.mm_w_d[m];
        double c, s;
        sincos_quarter(fma(w * (1.0 / kTwo40), r, fma(-w, I.rmin_d, -0.78539816339744830962)), s, c);
        double cp;
        if (Z4) {
            const double c2 = c * c;
            cp = (c * c2) * (c2 * c2);
        } else {
            cp = 1.0;
            double bp = c;
            for (int e = 2 * I.zeta - 1; e > 0; e >>= 1) {
                if (e & 1) cp *= bp;
                bp *= bp;
            }
        }
        g = -eps * (cp * c);
        rad = (I.mm_e2zw_d[m] * kTwo32) * (cp * s) * phi;
    }
    U = EN ? fma(g, phi, fu) : 0.0;
    const double gm = g * (mu * kTwo32 / kTwo80);      // g mu 2^32, per product of two grid directors
    const double gr = gm * (ri * kTwo40);              // ... / r
    const double js = S0 ? jr + s0 : jr, is = S0 ? ir - s0 : ir;
    // F = -(radial - g mu wr / r) h - (g mu / r) w with w = -js n_i - is n_j,
    // wr = w.h = -(js ir + is jr)
    const double ca = fma(gr, fma(js, ir, is * jr), rad);
    const double cb = gr * js, cc = gr * is;
    double gi[3], gj[3];
    for (int a = 0; a < 3; a++) {
        f[a] = fma(-ca, h[a], fma(cb, A[a], cc * B[a]));
        gi[a] = fma(-js, h[a], B[a]);                  // da/dn_i
        gj[a] = fma(-is, h[a], A[a]);                  // da/dn_j
    }
    for (int a = 0; a < 3; a++) {
        const int u = a == 2 ? 0 : a + 1, w = a == 0 ? 2 : a - 1;
        ti[a] = -gm * fma(A[u], gi[w], -(A[w] * gi[u]));
        tj[a] = -gm * fma(B[u], gj[w], -(B[w] * gj[u]));
    }
}

// Does the found particle interact with particle pi (mirror displacement d:
// FP32 outside the cutoff band, exact inside it, exclusions), and is the pair
// pi's to evaluate?  Returns the pair's class and species in code, its other
// slot in pj.
__device__ inline bool own_pair_d(const View& v, const Inst& I, const PairC& C, int4 qi, int pi, unsigned idi, int qj,
                                  int ox, int oy, int oz, int& pj, int& code) {
    const int4 mj = __ldg(v.mqr + qj);
    int m;
    const int cls = pair_class(qi.w & 0xff, mj.w & 0xff, m);
    const float dx = (float)(int)((unsigned)mj.x + (unsigned)ox - (unsigned)qi.x) * kMirrorUnit,
                dy = (float)(int)((unsigned)mj.y + (unsigned)oy - (unsigned)qi.y) * kMirrorUnit,
                dz = (float)(int)((unsigned)mj.z + (unsigned)oz - (unsigned)qi.z) * kMirrorUnit;
    const float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
    const float lo = cls == 0 ? I.mm_lo[m] : (cls == 1 ? C.w_lo : C.p_lo);
    const float hi = cls == 0 ? I.mm_hi[m] : (cls == 1 ? C.w_hi : C.p_hi);
    if (r2 >= hi) return false;
    pj = __float_as_int(__ldg(&v.mor[qj].w));
    const Inst& J = (unsigned)(pj - I.p0) < (unsigned)I.n ? I : v.inst[I.partner];
    if (idi > (unsigned)J.id_base + v.id[pj]) return false;
    if (!(r2 < lo) && !exact_inside(v, I, pi, pj, cls, m)) return false;
    if (cls != 0 && (qi.w & mj.w & kMirrorBonded) && is_excluded(v, I, v.id[pi], v.id[pj], pj)) return false;
    code = cls | (m << 2);
    return true;
}

// One pair's terms into F and T of both particles.
template <bool Z4, bool S0, bool EN>
__device__ inline void eval_pair_d(const View& v, const Inst& I, int pi, int pj, int code, long long& eu, long long& ew) {
    const size_t N = v.N;
    const int cls = code & 3, m = code >> 2;
    double D[3], A[3], B[3], f[3], ti[3], tj[3], U;
    for (int a = 0; a < 3; a++)
        D[a] = __ll2double_rn(minimg_q(v.xq[a * N + pj] - v.xq[a * N + pi], I.boxq[a], I.periodic[a]));
    if (cls == 0)
        for (int a = 0; a < 3; a++) {
            A[a] = __ll2double_rn(v.nq[a * N + pi]);
            B[a] = __ll2double_rn(v.nq[a * N + pj]);
        }
    pair_terms_d<Z4, S0, EN>(I, cls, m, D, A, B, f, ti, tj, U);
    // (a conversion saturates and turns a NaN into the most negative integer,
    // so one integer test finds terms beyond the range and NaN)
    const long long lim = (long long)((double)kMaxTerm * kTwo32);
    long long q[9];
    for (int a = 0; a < 3; a++) { q[a] = __double2ll_rn(f[a]); q[3 + a] = __double2ll_rn(ti[a]); q[6 + a] = __double2ll_rn(tj[a]); }
    bool big = false;
    for (int a = 0; a < 9; a++) big |= !below(q[a], lim - 1);
    if (big) {
        const double s = f[0] + f[1] + f[2] + ti[0] + ti[1] + ti[2] + tj[0] + tj[1] + tj[2];
        flag_inst(v, I, s == s ? kStatusPairForceRange : kStatusNaN);
    }
    for (int a = 0; a < 3; a++) {
        atomicAdd((unsigned long long*)&v.F[a * N + pi], (unsigned long long)q[a]);
        atomicAdd((unsigned long long*)&v.F[a * N + pj], (unsigned long long)(-q[a]));
    }
    if (cls == 0)
        for (int a = 0; a < 3; a++) {
            atomicAdd((unsigned long long*)&v.T[a * N + pi], (unsigned long long)q[3 + a]);
            atomicAdd((unsigned long long*)&v.T[a * N + pj], (unsigned long long)q[6 + a]);
        }
    if (EN) {
        // energy and virial at 2^-38 (|U| < 2^25): exact sums per cell, one
        // rounding to 2^-32 at its end
        eu += __double2ll_rn(U * 274877906944.0);
        ew += __double2ll_rn(fma(D[2], f[2], fma(D[1], f[1], D[0] * f[0])) * (-64.0 / kTwo40));
    }
}

// ---- distance tests on the tensor cores (TF32, FP32 accumulation)
// A warp tests its 32 particles against 32 candidates as the product of a
// 32 x 8 and an 8 x 32 matrix,
//   d^2 - cut = -2 x_i.x_j + |x_j|^2 + (|x_i|^2 - cut_i) - (cut of the class)_i,
// whose sign is the hit: eight m16n8k8 products and one funnel shift per
// result instead of about ten FP32 instructions per test (159M -> 126M
// instructions on the 1M cell; 0.66 -> 0.61 ms on the 4M cell, its species-pair
// form 195 -> 169 us at 1M).  Coordinates are
// rounded to TF32 first (and the squares taken of the rounded ones, split in
// two TF32 terms), so the result is the distance of points moved by at most
// 2^-11 of their distance from the cell's centre: the cutoffs grow by
// filter_band, and a list holds up to a few pairs more, which the exact
// decision drops.
__device__ inline float tf32_rna(float x) {
    unsigned r;
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
    return __uint_as_float(r);
}
__device__ inline float tf32_down(float x) {      // towards minus infinity
    const float r = __uint_as_float(__float_as_uint(x) & 0xffffe000u);
    return r <= x ? r : __uint_as_float(__float_as_uint(r) + 0x2000u);
}
__device__ inline void mma_tf32(float d[4], const float a[4], float b0, float b1) {
    asm("mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
        "{%10, %10, %10, %10};"
        : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
        : "r"(__float_as_uint(a[0])), "r"(__float_as_uint(a[1])), "r"(__float_as_uint(a[2])), "r"(__float_as_uint(a[3])),
          "r"(__float_as_uint(b0)), "r"(__float_as_uint(b1)), "f"(0.f));
}

// Eight CTAs per SM: 0.608 ms on the 4M cell against 0.613 at seven or nine.
// MP (band-3 or glycophorin in the batch): the staged particles carry three
// partner classes (lipid 0, cytoskeleton 1, bilayer protein 2) and each
// particle culls them at its own cutoff for that class, so that a lipid's
// list is not widened to the cutoff of its widest protein pair.
// DIRECT (FP64 forces): the pairs found are evaluated at once (pair_terms_d);
// F and T are zero before the launch.  EN adds U_pair and the virial of the
// cell's instance to energy [B][8].
template <bool MP, bool DIRECT = false, bool Z4 = true, bool S0 = false, bool EN = false, bool ONE = false, bool FAR = false>
__global__ void __launch_bounds__(kPairThreads, DIRECT ? 4 : 8)
    k_pair_search(View v, int* __restrict__ nlist, int* __restrict__ ncnt, int cap, int2* __restrict__ ovf,
                  int* __restrict__ novf, int ovf_cap, int4* __restrict__ rowoff, long long* __restrict__ energy,
                  const __grid_constant__ Inst one) {
    // sY: staged mirrors (int4 by the bulk copy), then in the tangent frame
    //     (FP32), w = 0 for a bilayer particle and 1 for a cytoskeleton protein
    // sQ: the list entry of each staged particle (DIRECT: its slot in the
    //     rank-ordered mirrors, its row in sR)
    // cand: per warp, the byte offsets (16 j) in sY of the culled candidates
    __shared__ alignas(16) float4 sY[kSearchStage];
    __shared__ int sQ[kSearchStage];
    __shared__ unsigned char sR[DIRECT ? kSearchStage : 1];
    __shared__ alignas(16) unsigned short cand[kPairThreads / 32][kSearchStage];
    __shared__ SNbr nb[kMaxNbr];
    __shared__ int s_cnt[kPairThreads];
    __shared__ alignas(16) float frag[kPairThreads / 32][32 * kFragRow];   // per warp: fragment rows
    __shared__ int2 wq[DIRECT ? kPairThreads / 32 : 1][DIRECT ? kQueue64 : 1];       // queued pairs: slots
    __shared__ unsigned char wc[DIRECT ? kPairThreads / 32 : 1][DIRECT ? kQueue64 : 1];   // class and species
    __shared__ long long s_e[2];
    __shared__ unsigned long long bar;
    __shared__ int s_nstage, s_next, s_next_off, s_self, s_self_lo, s_self_hi, s_total;

    const int k = blockIdx.x;
    const int b = ONE ? 0 : find_inst(v.inst_k0, v.B, k);
    const Inst& I = ONE ? one : v.inst[b];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int cs = v.cell_start[k], ce = v.cell_start[k + 1];
    const AdjDesc* __restrict__ row = v.adjd + (size_t)k * kAdjRow;
    const int a1 = min(v.adjn[k], kAdjRow);
    const size_t N = v.N;
    // (a list outlives the mirrors it was made from by up to a skin's move)
    const float sk = (DIRECT ? 0.0f : 2.0f * I.skinf) + kFilterBand;
    long long eu = 0, ew = 0;
    int nq = 0;                       // the warp's queued pairs
    auto drain = [&]() {              // evaluates the last 32 of them
        __syncwarp();
        nq -= 32;
        const int2 pr = wq[warp][nq + lane];
        eval_pair_d<Z4, S0, EN>(v, I, pr.x, pr.y, wc[warp][nq + lane], eu, ew);
        __syncwarp();
    };
    const float rsb = I.rsf + sk, rs2f = rsb * rsb;
    const int qbase = FAR ? list_base(v, I) : 0;
    const float cw = I.rcf_wca + sk, cp = I.rcf_pp + sk;
    // candidate c of 32 goes to the fragment column whose hit is bit c; the
    // byte transpose within four lanes that brings a row's hits to one lane
    const int fcol = (((lane >> 1) & 3) * 8 + 2 * (lane >> 3) + (lane & 1)) * kFragRow;
    const unsigned q4 = lane & 3;
    const unsigned selA = q4 | ((4 + q4) << 4), selC = 0x5410u,
                   selD = (0 ^ q4) | ((1 ^ q4) << 4) | ((2 ^ q4) << 8) | ((3 ^ q4) << 12);
    unsigned phase = 0;
    if (tid == 0) mbar_init(&bar, 1);
    __syncthreads();

    for (int it0 = cs; it0 < ce; it0 += kPairThreads) {
        const int nti = min(kPairThreads, ce - it0);
        const int groups = (nti + 31) >> 5;
        const int lsplit = (groups == 1) ? 2 : (groups == 2 ? 1 : 0), nsplit = 1 << lsplit;
        // (groups is 1 to 4: no divisions)
        const int jsplit = groups == 1 ? warp : (groups == 2 ? warp >> 1 : (groups == 3 ? (warp == 3) : 0));
        const int igrp = warp - jsplit * groups;
        const bool wactive = jsplit < nsplit;
        const int gs = groups == 1 ? nti : (groups == 2 ? (nti + 1) >> 1 : (groups == 3 ? (nti + 2) / 3 : (nti + 3) >> 2));
        s_cnt[tid] = 0;

        auto issue = [&](const int na, const int na_off) {
            if (warp == 0) {
                const int nn = na + lane;
                const bool has = nn < a1;
                int l = 0, st = 0, c = 0;
                AdjDesc d;
                if (has) {
                    d = row[nn];
                    l = d.cell();
                    st = d.start;
                    c = d.cnt;
                    // each row's exact offset, written where the row is first
                    // staged (lane 0 of a pass that continues a split row
                    // was written in the pass before)
                    if (!DIRECT && it0 == cs && !(lane == 0 && na_off > 0))
                        rowoff[(size_t)k * kAdjRow + nn] = make_int4(d.ox, d.oy, d.oz, 0);
                    if (lane == 0) { st += na_off; c -= na_off; }
                }
                int incl = c;
                for (int off = 1; off < 32; off <<= 1) {
                    const int t = __shfl_up_sync(0xffffffffu, incl, off);
                    if (lane >= off) incl += t;
                }
                const int excl = incl - c;
                const bool fits = has && incl <= kSearchStage;
                const bool part = has && excl < kSearchStage && incl > kSearchStage;
                const unsigned fm = __ballot_sync(0xffffffffu, fits), pm = __ballot_sync(0xffffffffu, part);
                const int m = __popc(fm) + (pm ? 1 : 0);
                const bool staged = fits || part;
                const int take = part ? kSearchStage - excl : c;
                if (staged) {
                    SNbr inf;
                    inf.base = excl; inf.cnt = take; inf.start = st; inf.row = nn;
                    whole_offset(d, inf.ox, inf.oy, inf.oz);
                    nb[lane] = inf;
                }
                const unsigned selfm = __ballot_sync(0xffffffffu, staged && l == k);
                const int total = __shfl_sync(0xffffffffu, excl + take, max(m - 1, 0));
                int nxt = na + __popc(fm), nxo = 0;
                if (pm) {
                    const int p = __ffs(pm) - 1;
                    const int ex_p = __shfl_sync(0xffffffffu, excl, p);
                    nxt = na + p;
                    nxo = (p == 0 ? na_off : 0) + (kSearchStage - ex_p);
                }
                int slo = -1, shi = -1, sb = 0;
                {
                    const int p = selfm ? __ffs(selfm) - 1 : 0;
                    const int ex_p = __shfl_sync(0xffffffffu, excl, p);
                    const int tk_p = __shfl_sync(0xffffffffu, take, p);
                    if (selfm) {
                        slo = ex_p;
                        shi = ex_p + tk_p;
                        sb = ex_p - ((p == 0) ? na_off : 0);
                    }
                }
                if (lane == 0) {
                    s_nstage = m;
                    s_total = m > 0 ? total : 0;
                    s_next = nxt;
                    s_next_off = nxo;
                    s_self = sb; s_self_lo = slo; s_self_hi = shi;
                }
                if (m > 0) {
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    if (lane == 0) mbar_expect_tx(&bar, (unsigned)total * 16u + v.extra_tx);
                    __syncwarp();
                    if (staged && take > 0) bulk_g2s(&sY[excl], v.mqr + st, take * 16u, &bar);
                }
            }
        };
        if (0 < a1) issue(0, 0);

        const Frame F = load_frame(v, k);
        const int r = igrp * gs + lane;
        const bool ivalid = wactive && lane < gs && r < nti;
        int ti = 0, pi = 0;
        unsigned idi = 0;
        int4 qi = make_int4(0, 0, 0, 0);
        float yix = 1.0e18f, yiy = 1.0e18f, yiz = 1.0e18f;
        if (ivalid) {
            qi = v.mqr[it0 + r];
            ti = qi.w & 0xff;
            if (DIRECT) {
                pi = __float_as_int(v.mor[it0 + r].w);
                idi = (unsigned)I.id_base + v.id[pi];
            }
            F.apply(qi.x * kMirrorUnit, qi.y * kMirrorUnit, qi.z * kMirrorUnit, yix, yiy, yiz);
        }
        // squared search radius for a bilayer and for a cytoskeleton partner
        // (for a bilayer particle the widest cutoff of its species; with MP
        // the lipid partners' and the bilayer proteins' apart), widened by
        // what the rounded coordinates may move: 2^-11 (|x_i| + |x_j|) with
        // |x_i| <= R_k (plus what it moved since), |x_j| <= |x_i| + r_s, and
        // the rounding of the products' sum
        const bool bi = bilayer(ti);
        const int si = species(ti);
        const float reach = 2.0f * (v.Rf[k] + 2.0f * I.skinf) + rsb;
        const float fb = sk + 5.0e-4f * reach, fb2 = 1.0e-5f * reach * reach + 1.0e-4f;
        const float cl = (MP ? I.mm_rcp[3 * si] : I.mm_rcf[si]) + fb;
        const float cwb = I.rcf_wca + fb, cpb = I.rcf_pp + fb;
        const float cutL = (bi ? cl * cl : cwb * cwb) + fb2;
        const float cutP = (bi ? cwb * cwb : cpb * cpb) + fb2;
        float cutM = cutP;
        if (MP) {
            const float cm = fmaxf(I.mm_rcp[3 * si + 1], I.mm_rcp[3 * si + 2]) + fb;
            cutM = (bi ? cm * cm : cwb * cwb) + fb2;
        }
        // A fragments: lane l's particle is row (l >> 2) + 8 (l & 3), which is
        // the row whose hits the lane ends up with
        float af[2][4];
        float* const fr = frag[warp];
        {
            const float x = tf32_rna(yix), y = tf32_rna(yiy), z = tf32_rna(yiz);
            float c = fmaf(x, x, fmaf(y, y, z * z)) - cutL;
            float ax = -2.0f * x, ay = -2.0f * y, az = -2.0f * z;
            if (!ivalid) { c = 1.0e30f; ax = ay = az = 0.f; }
            const float ch = tf32_rna(c);
            float* w = fr + ((lane >> 2) + 8 * (lane & 3)) * kFragRow;
            *reinterpret_cast<float4*>(w) = make_float4(ax, ay, az, 1.0f);
            *reinterpret_cast<float4*>(w + 4) = make_float4(MP ? tf32_down(cutL - cutP) : 1.0f, ch, ivalid ? c - ch : 0.f,
                                                            tf32_down(cutL - (MP ? cutM : cutP)));
            __syncwarp();
            const float* p = fr + (lane >> 2) * kFragRow + (lane & 3);
            for (int h = 0; h < 2; h++) {
                af[h][0] = p[16 * h * kFragRow];
                af[h][1] = p[(16 * h + 8) * kFragRow];
                af[h][2] = p[16 * h * kFragRow + 4];
                af[h][3] = p[(16 * h + 8) * kFragRow + 4];
            }
            __syncwarp();
        }
        // the group box's cull radius: the search cutoff, or for a group
        // without bilayer particles (a protein cell) the larger of its two
        // cutoffs
        const bool glip = __any_sync(0xffffffffu, ivalid && bi);
        const float rcull2 = glip ? rs2f : fmaxf(cw, cp) * fmaxf(cw, cp);
        float blo[3] = {ivalid ? yix : 3.0e38f, ivalid ? yiy : 3.0e38f, ivalid ? yiz : 3.0e38f};
        float bhi[3] = {ivalid ? yix : -3.0e38f, ivalid ? yiy : -3.0e38f, ivalid ? yiz : -3.0e38f};
        for (int a = 0; a < 3; a++) { blo[a] = warp_min_f32(blo[a]); bhi[a] = warp_max_f32(bhi[a]); }
        const int qi_idx = it0 + r;

        bool first_pass = true;
        for (int na = 0, na_off = 0; na < a1;) {
            if (!first_pass) {
                __syncthreads();
                issue(na, na_off);
            }
            first_pass = false;
            __syncthreads();
            const int m = s_nstage;
            const int total = s_total;
            const int next = s_next, next_off = s_next_off;
            if (m == 0) { na = next; na_off = next_off; continue; }
            const int sself = s_self, sslo = s_self_lo, sshi = s_self_hi;
            int selfj = (sslo >= 0 && ivalid) ? sself + (it0 + r - cs) : -1;
            if (selfj < sslo || selfj >= sshi) selfj = -1;
            bool ok = mbar_wait_bounded(&bar, phase, v.status, v.wait_polls);
            if (__syncthreads_or(!ok)) {
                if (ok == false) mbar_wait_bounded(&bar, phase, v.status, v.wait_polls);
                return;
            }
            phase ^= 1u;
            // staged particles into the cell's tangent frame (FP32), with
            // their list entries
            // (a warp per neighbouring cell: with the whole CTA on one cell
            // after the other, half of its warps found nothing to do; the
            // whole CTA for the few cells of a pass that large ones fill,
            // where warps would go without one: the search of eight cells of
            // 1,359 particles 0.9 ms against 1.0)
            const bool wide = m < kPairThreads / 32;
            for (int q = wide ? 0 : warp; q < m; q += wide ? 1 : kPairThreads / 32) {
                const SNbr inf = nb[q];
                for (int j = inf.base + (wide ? tid : lane); j < inf.base + inf.cnt; j += wide ? kPairThreads : 32) {
                    const int4 rj = reinterpret_cast<const int4*>(sY)[j];
                    float4 w;
                    F.apply(fmaf((float)rj.x, kMirrorUnit, inf.ox), fmaf((float)rj.y, kMirrorUnit, inf.oy),
                            fmaf((float)rj.z, kMirrorUnit, inf.oz), w.x, w.y, w.z);
                    const int tj = rj.w & 0xff;
                    w.w = MP ? (tj == kLipid ? 0.0f : (bilayer(tj) ? 2.0f : 1.0f)) : (bilayer(tj) ? 0.0f : 1.0f);
                    sY[j] = w;
                    const int at = inf.start + (j - inf.base);
                    if (DIRECT) sR[j] = (unsigned char)inf.row;
                    sQ[j] = DIRECT ? at : (inf.row << kRowShift) | (at - qbase);
                }
            }
            __syncthreads();

            if (wactive) {
                int cnt = 0, p0 = 0;
                // the warp's first own particle in this pass: the group's
                // particles are staged one after the other and lie in its
                // box, so they follow each other in the candidate list too
                const int self0 = sself + (it0 + igrp * gs - cs);
                int jf = max(self0, sslo);
                jf += (jsplit - jf) & (nsplit - 1);
                for (int c0 = 0; c0 < total; c0 += nsplit * 32) {
                    const int j = c0 + lane * nsplit + jsplit;
                    bool in = false;
                    if (j < total) {
                        const float4 y = sY[j];
                        const float ex = fmaxf(fmaxf(blo[0] - y.x, y.x - bhi[0]), 0.f);
                        const float ey = fmaxf(fmaxf(blo[1] - y.y, y.y - bhi[1]), 0.f);
                        const float ez = fmaxf(fmaxf(blo[2] - y.z, y.z - bhi[2]), 0.f);
                        in = fmaf(ex, ex, fmaf(ey, ey, ez * ez)) < rcull2;
                    }
                    const unsigned bal = __ballot_sync(0xffffffffu, in);
                    if ((unsigned)(jf - c0) < (unsigned)(nsplit * 32))
                        p0 = cnt + __popc(bal & ((1u << ((jf - jsplit - c0) >> lsplit)) - 1u));
                    if (in) cand[warp][cnt + __popc(bal & ((1u << lane) - 1u))] = (unsigned short)(j << 4);   // byte offset of sY[j]
                    cnt += __popc(bal);
                }
                __syncwarp();
                // the own particle's place in this warp's list (-1: the other warps')
                const int sp = selfj >= 0 && ((selfj - jsplit) & (nsplit - 1)) == 0 ? p0 + ((selfj - jf) >> lsplit) : -1;
                // 32 candidates at a time (past the list: far away, no hit)
                static_assert(kSearchStage * 16 <= 65536, "candidate byte offsets fit 16 bits");
                for (int c0 = 0; c0 < cnt; c0 += 32) {
                    {
                        float4 y = make_float4(0.f, 0.f, 0.f, 0.f);
                        float n = 1.0e30f;
                        if (c0 + lane < cnt) {
                            y = *reinterpret_cast<const float4*>(reinterpret_cast<const char*>(sY) + cand[warp][c0 + lane]);
                            y.x = tf32_rna(y.x); y.y = tf32_rna(y.y); y.z = tf32_rna(y.z);
                            n = fmaf(y.x, y.x, fmaf(y.y, y.y, y.z * y.z));
                        }
                        // (MP has no room for the square's second term: rounded down)
                        const float nh = MP ? __uint_as_float(__float_as_uint(n) & 0xffffe000u) : tf32_rna(n);
                        float* w = fr + fcol;
                        *reinterpret_cast<float4*>(w) = make_float4(y.x, y.y, y.z, nh);
                        *reinterpret_cast<float4*>(w + 4) =
                            make_float4(MP ? (y.w == 1.0f ? 1.0f : 0.f) : n - nh, 1.0f, 1.0f, MP ? (y.w == 2.0f ? 1.0f : 0.f) : y.w);
                    }
                    __syncwarp();
                    unsigned m0 = 0, m1 = 0, m2 = 0, m3 = 0;       // rows g, g + 8, g + 16, g + 24
                    const float* p = fr + (lane >> 2) * kFragRow + (lane & 3);
#pragma unroll
                    for (int nt = 3; nt >= 0; nt--) {
                        const float b0 = p[8 * nt * kFragRow], b1 = p[8 * nt * kFragRow + 4];
                        float d[4];
                        mma_tf32(d, af[0], b0, b1);
                        m0 = __funnelshift_l(__float_as_uint(d[1]), m0, 1);
                        m0 = __funnelshift_l(__float_as_uint(d[0]), m0, 1);
                        m1 = __funnelshift_l(__float_as_uint(d[3]), m1, 1);
                        m1 = __funnelshift_l(__float_as_uint(d[2]), m1, 1);
                        mma_tf32(d, af[1], b0, b1);
                        m2 = __funnelshift_l(__float_as_uint(d[1]), m2, 1);
                        m2 = __funnelshift_l(__float_as_uint(d[0]), m2, 1);
                        m3 = __funnelshift_l(__float_as_uint(d[3]), m3, 1);
                        m3 = __funnelshift_l(__float_as_uint(d[2]), m3, 1);
                    }
                    __syncwarp();
                    // bytes (row, lane of four) -> (lane, row): byte u of the
                    // result is this lane's row in lane u of the four
                    const unsigned mm = m0 | (m1 << 8) | (m2 << 16) | (m3 << 24);
                    const unsigned w1 = __shfl_xor_sync(0xffffffffu, mm, 1), w2 = __shfl_xor_sync(0xffffffffu, mm, 2),
                                   w3 = __shfl_xor_sync(0xffffffffu, mm, 3);
                    // own, lane ^ 1, lane ^ 2, lane ^ 3 in this order, then by lane
                    unsigned hits = __byte_perm(__byte_perm(mm, w1, selA), __byte_perm(w2, w3, selA), selC);
                    hits = __byte_perm(hits, 0u, selD);
                    if ((unsigned)(sp - c0) < 32u) hits &= ~(1u << (sp - c0));
                    if constexpr (DIRECT) {
                        const PairC C(I);
                        while (__any_sync(0xffffffffu, hits)) {
                            bool in = false;
                            int pj = 0, code = 0;
                            if (hits) {
                                const int u = __ffs(hits) - 1;
                                hits &= hits - 1u;
                                const int j = cand[warp][c0 + u] >> 4;
                                const AdjDesc& d = row[sR[j]];
                                in = own_pair_d(v, I, C, qi, pi, idi, sQ[j], d.ox, d.oy, d.oz, pj, code);
                            }
                            const unsigned m2 = __ballot_sync(0xffffffffu, in);
                            if (in) {
                                const int at = nq + __popc(m2 & ((1u << lane) - 1u));
                                wq[warp][at] = make_int2(pi, pj);
                                wc[warp][at] = (unsigned char)code;
                            }
                            nq += __popc(m2);
                            if (nq >= 32) drain();
                        }
                    }
                    if constexpr (!DIRECT) {
                        // places in the list for all hits of the chunk at once
                        // (the warps of a group share the particle's list)
                        const int nh = __popc(hits);
                        int pos = nh ? atomicAdd(&s_cnt[r], nh) : 0;
                        if (pos + nh <= cap) {
                            int* at = nlist + (size_t)pos * N + qi_idx;
                            while (hits) {
                                const int u = __ffs(hits) - 1;
                                hits &= hits - 1u;
                                *at = sQ[cand[warp][c0 + u] >> 4];
                                at += N;
                            }
                        } else {
                            while (hits) {
                                const int u = __ffs(hits) - 1;
                                hits &= hits - 1u;
                                const int e = sQ[cand[warp][c0 + u] >> 4];
                                if (pos < cap) {
                                    nlist[(size_t)pos * N + qi_idx] = e;
                                } else {
                                    const int o = atomicAdd(novf, 1);
                                    if (o < ovf_cap) ovf[o] = make_int2(qi_idx, e);
                                    else atomicOr(v.status, kStatusListOverflow);
                                }
                                pos++;
                            }
                        }
                    }
                }
            }
            na = next;
            na_off = next_off;
        }
        __syncthreads();
        if (!DIRECT && tid < nti) ncnt[it0 + tid] = s_cnt[tid];
        __syncthreads();
    }
    if constexpr (DIRECT) {
        // the warps' remainders (fewer than 32 pairs each) together: the
        // warps move theirs behind the first one's (room for 4 x 31 in the
        // four queues), which saves two of four nearly empty rounds per cell
        __shared__ int s_left[kPairThreads / 32];
        int2 pr = make_int2(0, 0);
        unsigned char code = 0;
        __syncwarp();
        if (lane < nq) { pr = wq[warp][lane]; code = wc[warp][lane]; }
        if (lane == 0) s_left[warp] = nq;
        __syncthreads();
        int base = 0, total = 0;
        for (int w = 0; w < kPairThreads / 32; w++) { base += w < warp ? s_left[w] : 0; total += s_left[w]; }
        if (lane < nq) { (&wq[0][0])[base + lane] = pr; (&wc[0][0])[base + lane] = code; }
        __syncthreads();
        if (tid < total) {
            pr = (&wq[0][0])[tid];
            eval_pair_d<Z4, S0, EN>(v, I, pr.x, pr.y, (&wc[0][0])[tid], eu, ew);
        }
        if (EN) {
            if (tid < 2) s_e[tid] = 0;
            __syncthreads();
            atomicAdd((unsigned long long*)&s_e[0], (unsigned long long)eu);
            atomicAdd((unsigned long long*)&s_e[1], (unsigned long long)ew);
            __syncthreads();
            if (tid == 0) {
                atomicAdd((unsigned long long*)&energy[b * 8 + 0], (unsigned long long)((s_e[0] + 32) >> 6));
                atomicAdd((unsigned long long*)&energy[b * 8 + 4], (unsigned long long)((s_e[1] + 32) >> 6));
            }
        }
    }
}

// One listed pair: exact integer displacement (2^-26 sigma), the type-pair
// cutoff decided in FP32 outside a 1e-6 sigma band and in FP64 inside it,
// bonded exclusions, then the FP32 pair terms.  Returns false when the pair
// does not interact.
template <int Z, bool S0>
__device__ inline bool listed_pair(const View& v, const Inst& I, int zc, int pi, int ti, int4 qi, float4 oi, int4 mj,
                                   float4 oj, int4 o, float ll_lo, float ll_hi, float w_lo, float w_hi, float p_lo,
                                   float p_hi, float& fx, float& fy, float& fz, float& tx, float& ty, float& tz, float& U,
                                   float d[3]) {
    const int pj = __float_as_int(oj.w);
    const int tj = mj.w & 0xff;
    int m;
    const int cls = pair_class(ti, tj, m);
    const bool ll = cls == 0;
    const int dxq = (int)((unsigned)mj.x + (unsigned)o.x - (unsigned)qi.x);
    const int dyq = (int)((unsigned)mj.y + (unsigned)o.y - (unsigned)qi.y);
    const int dzq = (int)((unsigned)mj.z + (unsigned)o.z - (unsigned)qi.z);
    const float dx = (float)dxq * kMirrorUnit, dy = (float)dyq * kMirrorUnit, dz = (float)dzq * kMirrorUnit;
    const float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
    const float lo = cls == 0 ? (I.has_mp ? I.mm_lo[m] : ll_lo) : (cls == 1 ? w_lo : p_lo);
    const float hi = cls == 0 ? (I.has_mp ? I.mm_hi[m] : ll_hi) : (cls == 1 ? w_hi : p_hi);
    if (r2 >= hi) return false;
    bool in = r2 < lo;
    if (!in) in = exact_inside(v, I, pi, pj, cls, m);
    if (in && cls != 0 && is_excluded(v, I, v.id[pi], v.id[pj], pj)) in = false;
    if (!in) return false;
    d[0] = dx; d[1] = dy; d[2] = dz;
    if (ll && I.has_mp)
        U = lipid_dispatch<S0, LipK>(LipK(I, m), dx, dy, dz, r2, oi.x, oi.y, oi.z, oj.x, oj.y, oj.z, fx, fy, fz, tx, ty, tz,
                                     zc, (float*)nullptr);
    else if (ll)
        U = lipid_dispatch<S0>(I, dx, dy, dz, r2, oi.x, oi.y, oi.z, oj.x, oj.y, oj.z, fx, fy, fz, tx, ty, tz, zc,
                               (float*)nullptr);
    else
        U = wca_terms(I, cls == 2, dx, dy, dz, r2, fx, fy, fz);
    return true;
}

// One particle's list (the thread of rank q): the listed particles' mirrors
// read from global memory (L1/L2), the constants of the pair terms in
// registers, the force and torque summed as exact split integers; terms of
// 1000 or more go to the int64 side array (big = true).
// MP: the batch holds band-3 or glycophorin, whose pairs take the constants
// of their bilayer species pair (the lipid-only instantiation tests the
// lipid type alone).
// EN: also the energies and virials of the particle's sides of its pairs
// (11 FP64-pipe instructions a pair in FP64, at 16 cycles each and SM; split
// integer sums take about 60 FP32 ones: forces and energies of the 1M cell in
// one call 1.17 ms with the one-launch kernel, 0.45 with the lists), as exact
// sums (hi 2^-32 + lo 2^-52) in es: U, then d . F, both over all listed
// pairs (each pair counted from both sides).
// The list's entries t0, t0 + dt, ... (dt > 1: several threads share a
// particle).
template <int Z, bool S0, bool MP = false, bool EN = false, bool FAR = false>
__device__ __forceinline__ void eval_list(const View& v, int q, const int* __restrict__ nlist,
                                          const int* __restrict__ ncnt, int cap, const int4* __restrict__ rowoff,
                                          SplitAcc af[3], SplitAcc at[3], int& nterm, bool& big, int& pi_out,
                                          const Inst* one, long long* es = nullptr, int t0 = 0, int dt = 1) {
    const size_t N = v.N;
    const int4 qi = v.mqr[q];
    const float4 oi = v.mor[q];
    const int pi = __float_as_int(oi.w);
    pi_out = pi;
    const int ti = qi.w & 0xff;
    const int k = v.cell[pi];
    const Inst& I = one ? *one : v.inst[find_inst(v.inst_p0, v.B, pi)];
    const PairC C(I);
    const int zc = (Z > 0) ? Z : C.zeta;
    const int4* __restrict__ ro = rowoff + (size_t)k * kAdjRow;
    const int qbase = FAR ? list_base(v, I) : 0;
    const int n = min(ncnt[q], cap);
    // a particle without bonds has no excluded pair: its list skips the test
    // (the lipid-only instantiation runs only when no bilayer particle has a
    // bond, so that only pairs of cytoskeleton proteins can be excluded)
    const bool ibond = (qi.w & kMirrorBonded) != 0;
    for (int a = 0; a < 3; a++) { af[a].zero(); at[a].zero(); }
    nterm = 0;
    big = false;
    SplitAcc3 eu, ew;
    int ne = 0;
    if (EN) {
        eu.zero();
        ew.zero();
        for (int a = 0; a < 4; a++) es[a] = 0;
    }
    // the next list entry is in flight while a pair is evaluated; the
    // mirrors are read through the read-only data path
    int e_next = t0 < n ? __ldcs(nlist + (size_t)t0 * N + q) : 0;
    for (int t = t0; t < n; t += dt) {
        const int e = e_next;
        if (t + dt < n) e_next = __ldcs(nlist + (size_t)(t + dt) * N + q);
        const int qj = qbase + (e & ((1 << kRowShift) - 1));
        const int4 o = __ldg(ro + ((unsigned)e >> kRowShift));
        const int4 mj = __ldg(v.mqr + qj);
        const float4 oj = __ldg(v.mor + qj);
        const int tj = mj.w & 0xff;
        int m = 0;
        int cls;
        if constexpr (MP) {
            cls = pair_class(ti, tj, m);
        } else {
            const bool l2 = (ti == kLipid) && (tj == kLipid);
            cls = l2 ? 0 : ((ti == kLipid || tj == kLipid) ? 1 : 2);
        }
        const bool ll = cls == 0;
        const int dxq = (int)((unsigned)mj.x + (unsigned)o.x - (unsigned)qi.x);
        const int dyq = (int)((unsigned)mj.y + (unsigned)o.y - (unsigned)qi.y);
        const int dzq = (int)((unsigned)mj.z + (unsigned)o.z - (unsigned)qi.z);
        const float dx = (float)dxq * kMirrorUnit, dy = (float)dyq * kMirrorUnit, dz = (float)dzq * kMirrorUnit;
        const float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
        // (a lipid pair, m = 0, keeps the constants held in registers)
        const bool tab = MP && m != 0;
        const float lo = cls == 0 ? (tab ? I.mm_lo[m] : C.ll_lo) : (cls == 1 ? C.w_lo : C.p_lo);
        const float hi = cls == 0 ? (tab ? I.mm_hi[m] : C.ll_hi) : (cls == 1 ? C.w_hi : C.p_hi);
        if (r2 >= hi) continue;
        if (!(r2 < lo) && !exact_inside(v, I, pi, __float_as_int(oj.w), cls, m)) continue;
        if ((MP ? (cls != 0 && ibond) : cls == 2) &&
            is_excluded(v, I, v.id[pi], v.id[__float_as_int(oj.w)], __float_as_int(oj.w)))
            continue;
        float f[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        float U = 0.f;
        if (ll && MP) {
            // one code path for every species pair (lanes with different
            // pairs stay converged): the pair's constants picked first
            PairC Cm = C;
            if (tab) {
                Cm.eps = I.mm_eps[m];
                Cm.aw = I.mm_aw[m];
                Cm.eps2z_aw = I.mm_e2za[m];
            }
            if (zc == 4)
                U = lipid_terms_f<4, S0>(Cm, dx, dy, dz, r2, oi.x, oi.y, oi.z, oj.x, oj.y, oj.z, f[0], f[1], f[2], f[3],
                                     f[4], f[5]);
            else
                U = lipid_terms_f<0, true>(Cm, dx, dy, dz, r2, oi.x, oi.y, oi.z, oj.x, oj.y, oj.z, f[0], f[1], f[2],
                                       f[3], f[4], f[5]);
        } else if (ll) {
            if (zc == 4)
                U = lipid_terms_f<4, S0>(C, dx, dy, dz, r2, oi.x, oi.y, oi.z, oj.x, oj.y, oj.z, f[0], f[1], f[2], f[3],
                                     f[4], f[5]);
            else
                U = lipid_terms_f<0, true>(C, dx, dy, dz, r2, oi.x, oi.y, oi.z, oj.x, oj.y, oj.z, f[0], f[1], f[2], f[3],
                                       f[4], f[5]);
        } else {
            const float sig = cls == 2 ? C.sig_pp : C.sig_wca;
            const float s2 = sig * sig / r2;
            const float s6 = s2 * s2 * s2;
            const float s12 = s6 * s6;
            const float fr = 4.0f * C.eps_wca * (12.0f * s12 - 6.0f * s6) / r2;
            f[0] = -fr * dx; f[1] = -fr * dy; f[2] = -fr * dz;
            U = 4.0f * C.eps_wca * (s12 - s6) + C.eps_wca;
        }
        if (EN) {
            // the products with their rounding errors (fused multiply-adds),
            // so that the virial's sum is as exact as the energy's
            const float w0 = dx * f[0], w1 = dy * f[1], w2 = dz * f[2];
            const float we = fmaf(dx, f[0], -w0) + fmaf(dy, f[1], -w1) + fmaf(dz, f[2], -w2);
            if (fabsf(U) < 1000.0f && fabsf(w0) + fabsf(w1) + fabsf(w2) < 1000.0f) {
                eu.add(U);
                ew.add(w0); ew.add(w1); ew.add(w2); ew.add(we);
                ne++;
            } else {
                es[0] += __double2ll_rn((double)U * 4294967296.0);
                es[2] += __double2ll_rn(((double)w0 + (double)w1 + (double)w2 + (double)we) * 4294967296.0);
            }
        }
        const float mag = fabsf(f[0]) + fabsf(f[1]) + fabsf(f[2]) + fabsf(f[3]) + fabsf(f[4]) + fabsf(f[5]);
        if (mag < 1000.0f) {
            for (int a = 0; a < 3; a++) { af[a].add(f[a]); at[a].add(f[3 + a]); }
            nterm++;
        } else {
            // terms of 1000 or more go to the int64 side array (exact, rare)
            if (!(mag < kMaxTerm))
                flag_inst(v, v.inst[find_inst(v.inst_p0, v.B, pi)], (mag == mag) ? kStatusPairForceRange : kStatusNaN);
            for (int a = 0; a < 6; a++)
                atomicAdd((unsigned long long*)&v.Fbig[(size_t)a * N + pi],
                          (unsigned long long)__float2ll_rn(f[a] * 4294967296.0f));
            big = true;
        }
    }
    if (EN) {
        long long h, l;
        eu.finish(ne, h, l);
        es[0] += h; es[1] += l;
        ew.finish(4 * ne, h, l);
        es[2] += h; es[3] += l;
    }
}

// The block's particles by the length of their lists, the longest first:
// thread t takes the particle of the returned rank.  A warp lasts as long as
// its longest list, and a cell's beads have a few partners where its lipids
// have twenty.
__device__ __forceinline__ int by_length(const int* __restrict__ ncnt, int cap, int N) {
    __shared__ int bin_n[64];           // by list length + 1, 0: no particle; counts, then starts
    __shared__ unsigned char order[kPairThreads];
    static_assert(kListCap + 2 <= 64 && kPairThreads <= 256, "a bin per length, a byte per thread");
    const int t = threadIdx.x, q = blockIdx.x * kPairThreads + t;
    if (t < 64) bin_n[t] = 0;
    __syncthreads();
    const int bin = q < N ? min(ncnt[q], cap) + 1 : 0;
    const int r = atomicAdd(&bin_n[bin], 1);
    __syncthreads();
    if (t < 32) {
        const int c0 = bin_n[63 - 2 * t], c1 = bin_n[62 - 2 * t];
        int x = c0 + c1;
        for (int off = 1; off < 32; off <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, x, off);
            if (t >= off) x += y;
        }
        bin_n[63 - 2 * t] = x - c0 - c1;
        bin_n[62 - 2 * t] = x - c1;
    }
    __syncthreads();
    order[bin_n[bin] + r] = (unsigned char)t;
    __syncthreads();
    return blockIdx.x * kPairThreads + order[t];
}

// Evaluation: one thread per particle over its list (see eval_list), the
// block's particles by the length of their lists (4M cell 0.62 ms against
// 0.65 in rank order, with a skin of 0.3 at 1M 0.236 against 0.254; blocks of
// 256 are slower, 0.68).  (Evaluating from mirrors staged in shared memory per
// cell, with each list split over two or four threads, took 1.31 ms against
// 1.06 ms of an earlier form of this kernel.)
// Compiled for 5 and 7 CTAs per SM (the autotuner's second dimension), 72
// registers at seven; at six 0.70 ms on the 4M cell, at eight (64 registers,
// more spills) 0.66.
// MP: the batch holds band-3 or glycophorin (eval_list).
template <int Z, bool S0, int MINB, bool MP = false, bool EN = false, bool ONE = false, bool FAR = false>
__global__ void __launch_bounds__(kPairThreads, MINB)
    k_pair_eval(View v, const int* __restrict__ nlist, const int* __restrict__ ncnt, int cap,
                const int4* __restrict__ rowoff, long long* __restrict__ energy, const __grid_constant__ Inst one) {
    const int q = by_length(ncnt, cap, v.N);
    if (!EN && q >= v.N) return;
    const size_t N = v.N;
    SplitAcc af[3], at[3];
    int nterm, pi;
    bool big;
    if constexpr (EN) {
        // the block's sums (exact), halved (each pair has two sides) and
        // rounded to 2^-32 once; energy [B][8] is summed over the instances
        // of a membrane, so the block's go to its first particle's
        __shared__ long long s_e[4];
        if (threadIdx.x < 4) s_e[threadIdx.x] = 0;
        __syncthreads();
        long long es[4] = {0, 0, 0, 0};
        if (q < v.N) eval_list<Z, S0, MP, true>(v, q, nlist, ncnt, cap, rowoff, af, at, nterm, big, pi, ONE ? &one : nullptr, es);
        for (int a = 0; a < 4; a++) {
            for (int off = 16; off; off >>= 1) es[a] += __shfl_xor_sync(0xffffffffu, es[a], off);
            if ((threadIdx.x & 31) == 0) atomicAdd((unsigned long long*)&s_e[a], (unsigned long long)es[a]);
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            auto half = [](long long hi, long long lo) {
                return (hi >> 1) + ((((hi & 1) << 20) + lo + (1ll << 20)) >> 21);
            };
            long long* e = energy + 8 * find_inst(v.inst_p0, v.B, blockIdx.x * blockDim.x);
            atomicAdd((unsigned long long*)&e[0], (unsigned long long)half(s_e[0], s_e[1]));
            atomicAdd((unsigned long long*)&e[4], (unsigned long long)half(-s_e[2], -s_e[3]));
        }
        if (q >= v.N) return;
    } else {
        eval_list<Z, S0, MP, false, FAR>(v, q, nlist, ncnt, cap, rowoff, af, at, nterm, big, pi, ONE ? &one : nullptr);
    }
#pragma unroll
    for (int a = 0; a < 3; a++) {
        long long fb = 0, tb = 0;
        if (big) {
            fb = __ldcg(&v.Fbig[(size_t)a * N + pi]);
            tb = __ldcg(&v.Fbig[(size_t)(3 + a) * N + pi]);
            v.Fbig[(size_t)a * N + pi] = 0;
            v.Fbig[(size_t)(3 + a) * N + pi] = 0;
        }
        v.F[a * N + pi] = af[a].finish(nterm) + fb;
        v.T[a * N + pi] = at[a].finish(nterm) + tb;
    }
}

// The same with 2^sh threads per particle (neighbouring lanes), for batches
// that one thread per particle spreads too thinly: a thread's chain of
// gathers and pair terms is what such a launch lasts (2,304 particles 20.5 us
// with one thread, 14.3 with four; 20k 26.2 and 18.0; 62k 32.7 and 26.6 with
// two; 145k are better off with one, 44.7 against 45.9).  The partial sums
// are integers, so the result is the same.
template <int Z, bool S0, bool MP, bool ONE>
__global__ void __launch_bounds__(128, 7)
    k_pair_eval_split(View v, const int* __restrict__ nlist, const int* __restrict__ ncnt, int cap,
                      const int4* __restrict__ rowoff, int sh, const __grid_constant__ Inst one) {
    const long long x = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const int q = (int)(x >> sh), part = (int)(x & ((1 << sh) - 1));
    const unsigned live = __ballot_sync(0xffffffffu, q < v.N);
    if (q >= v.N) return;
    const size_t N = v.N;
    SplitAcc af[3], at[3];
    int nterm, pi;
    bool big;
    eval_list<Z, S0, MP>(v, q, nlist, ncnt, cap, rowoff, af, at, nterm, big, pi, ONE ? &one : nullptr, nullptr, part,
                         1 << sh);
    __syncwarp(live);
    for (int off = 1 << (sh - 1); off; off >>= 1) {
        for (int a = 0; a < 3; a++) {
            af[a].h += __shfl_xor_sync(live, af[a].h, off);
            af[a].l += __shfl_xor_sync(live, af[a].l, off);
            at[a].h += __shfl_xor_sync(live, at[a].h, off);
            at[a].l += __shfl_xor_sync(live, at[a].l, off);
        }
        nterm += __shfl_xor_sync(live, nterm, off);
    }
    // (the large terms of the other lanes are in the side array before it is read)
    const unsigned anybig = __ballot_sync(live, big);
    if (anybig) {
        __threadfence();
        __syncwarp(live);
    }
    if (part != 0) return;
    const int lane = threadIdx.x & 31;
    const bool mine = (anybig >> lane) & ((1u << (1 << sh)) - 1u);
#pragma unroll
    for (int a = 0; a < 3; a++) {
        long long fb = 0, tb = 0;
        if (mine) {
            fb = __ldcg(&v.Fbig[(size_t)a * N + pi]);
            tb = __ldcg(&v.Fbig[(size_t)(3 + a) * N + pi]);
            v.Fbig[(size_t)a * N + pi] = 0;
            v.Fbig[(size_t)(3 + a) * N + pi] = 0;
        }
        v.F[a * N + pi] = af[a].finish(nterm) + fb;
        v.T[a * N + pi] = at[a].finish(nterm) + tb;
    }
}

// The evaluation of one step with the next step's update in its epilogue:
// each particle's force and torque are complete once its own list is done
// (the bonds, the listed pairs beyond the lists' capacity and the large
// terms were added beforehand to the side array, flagged per particle; the
// volume constraint's pressure is added here), and its B-A-O-A update (with
// the final B of this step) needs nothing else, so the FP64 update of one
// warp overlaps the FP32 pair terms of the others.  The updated state goes
// to the other state buffer (o): the exact inclusion decisions of the other
// threads still read this step's positions.  D: FP64 increments.
template <int Z, bool S0, bool D>
__global__ void __launch_bounds__(128, 4)
    k_pair_eval_step(View v, View o, const int* __restrict__ nlist, const int* __restrict__ ncnt, int cap,
                     const int4* __restrict__ rowoff, unsigned char* __restrict__ sflag,
                     const long long* __restrict__ steps, long long* __restrict__ msum, int* __restrict__ mcnt,
                     int* __restrict__ rot_list, int* __restrict__ rot_n) {
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    const unsigned live = __ballot_sync(0xffffffffu, q < v.N);
    if (q >= v.N) return;
    const size_t N = v.N;
    SplitAcc af[3], at[3];
    int nterm, pi;
    bool big;
    eval_list<Z, S0>(v, q, nlist, ncnt, cap, rowoff, af, at, nterm, big, pi, nullptr);
    const bool side = big || sflag[pi];
    long long F[3], Tq[3];
#pragma unroll
    for (int a = 0; a < 3; a++) {
        long long fb = 0, tb = 0;
        if (side) {
            fb = __ldcg(&v.Fbig[(size_t)a * N + pi]);
            tb = __ldcg(&v.Fbig[(size_t)(3 + a) * N + pi]);
            v.Fbig[(size_t)a * N + pi] = 0;
            v.Fbig[(size_t)(3 + a) * N + pi] = 0;
        }
        F[a] = af[a].finish(nterm) + fb;
        Tq[a] = at[a].finish(nterm) + tb;
    }
    if (side) sflag[pi] = 0;
    const Inst& I = v.inst[find_inst(v.inst_p0, v.B, pi)];
    if (I.vol_on && bilayer(v.type[pi])) {
        // the volume constraint's pressure on the lipid's area element, as
        // the constraint's own launch computes it
        const double V = I.a3 * volume_of(__ldg(&v.vol[2 * (&I - v.inst)]), __ldg(&v.vol[2 * (&I - v.inst) + 1]));
        const float pa = (float)(-I.kv * (V - I.v0) * I.avol);
        for (int a = 0; a < 3; a++) {
            const float f = pa * (ll_to_float(v.nq[a * N + pi]) * (float)kGridInv);
            if (!(fabsf(f) < kMaxTerm)) flag_inst(v, I, f == f ? kStatusPairForceRange : kStatusNaN);
            else F[a] += __float2ll_rn(f * 4294967296.0f);
        }
    }
    for (int a = 0; a < 3; a++) { v.F[a * N + pi] = F[a]; v.T[a * N + pi] = Tq[a]; }
    __syncwarp(live);
    if (D) baoa_d_body<true>(v, o, pi, F, Tq, steps, msum, mcnt, live, true, rot_list, rot_n, nullptr);
    else baoa_body<float, true>(v, o, pi, F, Tq, steps, msum, mcnt, live, true);
}

// Listed pairs beyond kListCap: the same terms, added to F and T by 64-bit
// integer atomics (each term rounded to 2^-32 exactly as the split sums do,
// so the totals are the same integers).
// sflag (nullable): add to the side array instead, and flag the particle
// (the evaluation with the update in its epilogue collects it).
template <int Z, bool S0, bool EN = false>
__device__ inline void pair_overflow(const View& v, const int2* __restrict__ ovf, const int* __restrict__ novf,
                                     int ovf_cap, const int4* __restrict__ rowoff, unsigned char* __restrict__ sflag,
                                     int at, int threads, long long* __restrict__ energy = nullptr) {
    const int n = min(*novf, ovf_cap);
    const size_t N = v.N;
    for (int x = at; x < n; x += threads) {
        const int2 pr = ovf[x];
        const int q = pr.x, e = pr.y;
        const int4 qi = v.mqr[q];
        const float4 oi = v.mor[q];
        const int pi = __float_as_int(oi.w);
        const int ti = qi.w & 0xff;
        const int k = v.cell[pi];
        const int b = find_inst(v.inst_p0, v.B, pi);
        const Inst& I = v.inst[b];
        const int zc = (Z > 0) ? Z : I.zeta;
        const float rcl = sqrtf(I.rc2f_ll), rcw = sqrtf(I.rc2f_wca), rcp = sqrtf(I.rc2f_pp);
        const int qj = (far_batch(v.N) ? list_base(v, I) : 0) + (e & ((1 << kRowShift) - 1));
        const int4 o = rowoff[(size_t)k * kAdjRow + ((unsigned)e >> kRowShift)];
        float f[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f}, U, d[3];
        if (!listed_pair<Z, S0>(v, I, zc, pi, ti, qi, oi, v.mqr[qj], v.mor[qj], o, (rcl - kCutBand) * (rcl - kCutBand),
                                (rcl + kCutBand) * (rcl + kCutBand), (rcw - kCutBand) * (rcw - kCutBand),
                                (rcw + kCutBand) * (rcw + kCutBand), (rcp - kCutBand) * (rcp - kCutBand),
                                (rcp + kCutBand) * (rcp + kCutBand), f[0], f[1], f[2], f[3], f[4], f[5], U, d))
            continue;
        const float mag = fabsf(f[0]) + fabsf(f[1]) + fabsf(f[2]) + fabsf(f[3]) + fabsf(f[4]) + fabsf(f[5]);
        if (!(mag < kMaxTerm)) flag_inst(v, I, (mag == mag) ? kStatusPairForceRange : kStatusNaN);
        long long* const Ft = sflag ? v.Fbig : v.F;
        long long* const Tt = sflag ? v.Fbig + 3 * N : v.T;
        for (int a = 0; a < 3; a++) {
            atomicAdd((unsigned long long*)&Ft[a * N + pi], (unsigned long long)__float2ll_rn(f[a] * 4294967296.0f));
            atomicAdd((unsigned long long*)&Tt[a * N + pi], (unsigned long long)__float2ll_rn(f[3 + a] * 4294967296.0f));
        }
        if (sflag) sflag[pi] = 1;
        if (EN) {
            const double w = (double)d[0] * (double)f[0] + (double)d[1] * (double)f[1] + (double)d[2] * (double)f[2];
            atomicAdd((unsigned long long*)&energy[b * 8 + 0], (unsigned long long)__double2ll_rn((double)U * 2147483648.0));
            atomicAdd((unsigned long long*)&energy[b * 8 + 4], (unsigned long long)__double2ll_rn(w * -2147483648.0));
        }
    }
}

template <int Z, bool S0>
__global__ void k_pair_overflow(View v, const int2* __restrict__ ovf, const int* __restrict__ novf, int ovf_cap,
                                const int4* __restrict__ rowoff, unsigned char* __restrict__ sflag) {
    pair_overflow<Z, S0>(v, ovf, novf, ovf_cap, rowoff, sflag, blockIdx.x * blockDim.x + threadIdx.x,
                         gridDim.x * blockDim.x);
}

// Harmonic bonds ("Force Evaluation": a list of bonds between proteins is
// maintained): one thread per bond, after the pair kernel wrote F.  The bond
// force is rounded to the 2^-32 grid once and added to both ends with
// opposite signs by 64-bit integer atomics: integer sums do not depend on
// the order, and the result equals evaluating the bond from each end.
// sflag (nullable): add to the side array instead, and flag both ends.
template <typename T, bool ENERGY>
__device__ inline void bond_one(const View& v, int q, long long* __restrict__ energy /* [B][8] */,
                                unsigned char* __restrict__ sflag) {
    int b = -1;
    long long eb = 0, ew = 0;
    if (q < v.nbond) {
        b = v.binst[q];
        const Inst& I = v.inst[b];
        const size_t N = v.N;
        const int2 e = v.bij[q];
        const int pi = v.slot_of_id[e.x], pj = v.slot_of_id[e.y];
        const long long ddx = minimg_q(v.xq[pj] - v.xq[pi], I.boxq[0], I.periodic[0]);
        const long long ddy = minimg_q(v.xq[N + pj] - v.xq[N + pi], I.boxq[1], I.periodic[1]);
        const long long ddz = minimg_q(v.xq[2 * N + pj] - v.xq[2 * N + pi], I.boxq[2], I.periodic[2]);
        T dx, dy, dz, r0, kb;
        if constexpr (sizeof(T) == 4) {
            dx = ll_to_float(ddx) * (float)kGridInv; dy = ll_to_float(ddy) * (float)kGridInv;
            dz = ll_to_float(ddz) * (float)kGridInv;
            const float2 kf = v.bkf[q];
            r0 = kf.x; kb = kf.y;
        } else {
            dx = grid_to_double(ddx); dy = grid_to_double(ddy); dz = grid_to_double(ddz);
            const double2 kd = v.bkd[q];
            r0 = kd.x; kb = kd.y;
        }
        const T r = sqrt(dx * dx + dy * dy + dz * dz);
        const T dr = r - r0;
        const T c = kb * dr / r;
        const T g[3] = {c * dx, c * dy, c * dz};     // force on the first end
        for (int a = 0; a < 3; a++) {
            long long f;
            if constexpr (sizeof(T) == 4) f = __float2ll_rn(g[a] * 4294967296.0f);
            else f = __double2ll_rn(g[a] * 4294967296.0);
            if (!(fabs(g[a]) < (T)kMaxTerm)) flag_inst(v, I, (g[a] == g[a]) ? kStatusPairForceRange : kStatusNaN);
            long long* const Ft = sflag ? v.Fbig : v.F;
            atomicAdd((unsigned long long*)&Ft[a * N + pi], (unsigned long long)f);
            atomicAdd((unsigned long long*)&Ft[a * N + pj], (unsigned long long)(-f));
        }
        if (sflag) { sflag[pi] = 1; sflag[pj] = 1; }
        if (ENERGY) {
            // energy and virial partials in FP64 from the exact displacement
            const double ex = grid_to_double(ddx), ey = grid_to_double(ddy), ez = grid_to_double(ddz);
            const double r2d = ex * ex + ey * ey + ez * ez;
            const double rd = sqrt(r2d);
            const double r0d = (double)r0, kbd = (double)kb;
            const double drd = rd - r0d;
            eb = __double2ll_rn(0.5 * kbd * drd * drd * 4294967296.0);
            ew = __double2ll_rn(-(kbd * drd * rd) * 4294967296.0);
        }
    }
    if (ENERGY) {
        // warp-aggregate per instance, then one atomic per instance and warp
        const unsigned grp = __match_any_sync(0xffffffffu, b);
        long long sb = 0, sw = 0;
        unsigned m = grp;
        while (m) {
            const int src = __ffs(m) - 1;
            m &= m - 1;
            sb += __shfl_sync(grp, eb, src);
            sw += __shfl_sync(grp, ew, src);
        }
        if (b >= 0 && (int)(threadIdx.x & 31) == __ffs(grp) - 1) {
            atomicAdd((unsigned long long*)&energy[b * 8 + 1], (unsigned long long)sb);
            atomicAdd((unsigned long long*)&energy[b * 8 + 4], (unsigned long long)sw);
        }
    }
}

template <typename T, bool ENERGY>
__global__ void k_bonds(View v, long long* __restrict__ energy, unsigned char* __restrict__ sflag) {
    bond_one<T, ENERGY>(v, blockIdx.x * blockDim.x + threadIdx.x, energy, sflag);
}

// The bonds and the listed pairs beyond the lists' capacity (blocks from
// ovf_block on) in one launch: both add to F by integer atomics after the
// evaluation wrote it.
template <int Z, bool S0, bool EN = false>
__global__ void k_bonds_overflow(View v, int ovf_block, const int2* __restrict__ ovf, const int* __restrict__ novf,
                                 int ovf_cap, const int4* __restrict__ rowoff, long long* __restrict__ energy) {
    if ((int)blockIdx.x < ovf_block)
        bond_one<float, EN>(v, blockIdx.x * blockDim.x + threadIdx.x, energy, nullptr);
    else
        pair_overflow<Z, S0, EN>(v, ovf, novf, ovf_cap, rowoff, nullptr, (blockIdx.x - ovf_block) * blockDim.x + threadIdx.x,
                                 (gridDim.x - ovf_block) * blockDim.x, energy);
}

// The pair kernel runs five CTAs per SM only with the whole unified L1 /
// shared memory given to shared memory; ask for that once per process.
template <typename Kern> static void prefer_shared(Kern k) {
    CK(cudaFuncSetAttribute((const void*)k, cudaFuncAttributePreferredSharedMemoryCarveout,
                            (int)cudaSharedmemCarveoutMaxShared));
}
static void prefer_shared_all() {
    static std::once_flag once;
    std::call_once(once, [] {
        prefer_shared(k_pairs<false, true, 0, true>);
        prefer_shared(k_pairs<true, false, 4, true>);
        prefer_shared(k_pairs<true, false, 4, false>);
        prefer_shared(k_pairs<true, false, 0, true>);
    });
}

void Ensemble::alloc_lists() {
    list_cap = kListCap;
    // the overflow list and the unranked mirrors of large cells share their
    // memory: the mirrors are read by the launch that writes them or the next
    // one of the rebuild, the overflow list is written by the search after it.
    // So the list holds the pairs that the tests' margin adds (up to about one
    // a particle) beside the N / 4 it is meant for
    ovf_cap = (int)std::min<long long>(std::max(N / 4, 4096) + 2ll * N, 0x7fffffff);
    d_nlist = alloc<int>((size_t)list_cap * N);
    d_ncnt = alloc<int>(N);
    d_novf = alloc<int2>(ovf_cap);
    d_mq = (int4*)d_novf;
    d_novf_n = alloc<int>(1);
    d_rowoff = alloc<int4>(adj_cap);
    d_sflag = alloc<unsigned char>(N);
    list_valid = false;
}

// The search's overflow count starts at zero: the rebuild before it left it
// so, unless the lists are searched again without a rebuild.
void Ensemble::clear_overflow() {
    if (!ovf_clean_) CK(cudaMemsetAsync(d_novf_n, 0, sizeof(int), stream));
    ovf_clean_ = false;
}

// The neighbour lists, once per cell reorder.
void Ensemble::launch_search() {
    if (list_valid) return;
    tic("pair_search");
    clear_overflow();
#define ORBC_SEARCH(MP, ONE, FAR)                                                                                         \
    k_pair_search<MP, false, true, false, false, ONE, FAR><<<Ktot, kPairThreads, 0, stream>>>(                                 \
        view(), d_nlist, d_ncnt, list_cap, d_novf, d_novf_n, ovf_cap, d_rowoff, nullptr, inst_h[0])
    if (any_mp()) {
        if (B == 1) ORBC_SEARCH(true, true, false);
        else if (far_batch(N)) ORBC_SEARCH(true, false, true);
        else ORBC_SEARCH(true, false, false);
    } else {
        if (B == 1) ORBC_SEARCH(false, true, false);
        else if (far_batch(N)) ORBC_SEARCH(false, false, true);
        else ORBC_SEARCH(false, false, false);
    }
#undef ORBC_SEARCH
    launches++;
    CK(cudaGetLastError());
    toc();
    list_valid = true;
}

void Ensemble::launch_pairs(bool energies, bool dump, bool one_launch) {
    View v = view();
    if (energies) CK(cudaMemsetAsync(d_energy, 0, sizeof(long long) * 8 * B, stream));
    bool z4 = true, s0z = true;
    for (auto& I : inst_h) { z4 = z4 && I.zeta == 4; s0z = s0z && I.s0_d == 0.0; }
    const dim3 g(Ktot), t(kPairThreads);
    prefer_shared_all();
    if (!force_f64() && !one_launch && !dump) {
        // split path: neighbour lists (once per cell reorder), evaluation,
        // listed pairs beyond the lists' capacity
        launch_search();
        tic("pairs");
        const int ng = (int)((N + kPairThreads - 1) / kPairThreads);
        // the batch's launch shape: the choice of its largest instance
        int ctas = prm_h[0].eval_ctas, nmax = -1;
        for (int b = 0; b < B; b++)
            if (inst_h[b].n > nmax) { nmax = inst_h[b].n; ctas = prm_h[b].eval_ctas; }
        // threads per particle: as many as fit the chip at once (seven CTAs
        // of 128 on each of 152 SMs), up to four (eight gain nothing more on
        // 2,304 particles and lose 2.6 us on 20,000)
        int sh = 0;
        while (sh < 2 && ((long long)N << (sh + 1)) <= 152ll * 7 * 128) sh++;
        const int nsp = (int)((((long long)N << sh) + 127) / 128);
        // (with energies: five CTAs per SM, for their registers)
        // one instance: its constants as a kernel argument (ONE)
#define ORBC_EVAL_N(Z, S, MP, ONE)                                                                                          \
    do {                                                                                                                    \
        if (energies)                                                                                                       \
            k_pair_eval<Z, S, 5, MP, true, ONE><<<ng, kPairThreads, 0, stream>>>(v, d_nlist, d_ncnt, list_cap, d_rowoff, d_energy, inst_h[0]); \
        else if (sh > 0)                                                                                                    \
            k_pair_eval_split<Z, S, MP, ONE><<<nsp, 128, 0, stream>>>(v, d_nlist, d_ncnt, list_cap, d_rowoff, sh, inst_h[0]); \
        else if (ctas == 5)                                                                                                 \
            k_pair_eval<Z, S, 5, MP, false, ONE><<<ng, kPairThreads, 0, stream>>>(v, d_nlist, d_ncnt, list_cap, d_rowoff, nullptr, inst_h[0]); \
        else                                                                                                                \
            k_pair_eval<Z, S, 7, MP, false, ONE><<<ng, kPairThreads, 0, stream>>>(v, d_nlist, d_ncnt, list_cap, d_rowoff, nullptr, inst_h[0]); \
    } while (0)
#define ORBC_EVAL(Z, S, MP)                                                                                                 \
    do {                                                                                                                    \
        if (B == 1) ORBC_EVAL_N(Z, S, MP, true);                                                                            \
        else if (far_batch(N)) /* (an arena's: no energies) */                                                              \
            k_pair_eval<Z, S, 7, MP, false, false, true><<<ng, kPairThreads, 0, stream>>>(v, d_nlist, d_ncnt, list_cap, d_rowoff, nullptr, inst_h[0]); \
        else ORBC_EVAL_N(Z, S, MP, false);                                                                                  \
    } while (0)
        if (any_mp()) {
            // band-3 or glycophorin present (or a bonded bilayer particle):
            // the evaluation with the bilayer species pairs' constants
            if (z4 && s0z) ORBC_EVAL(4, false, true);
            else ORBC_EVAL(0, true, true);
        } else if (z4 && s0z) {
            ORBC_EVAL(4, false, false);
        } else if (z4) {
            ORBC_EVAL(4, true, false);
        } else {
            ORBC_EVAL(0, true, false);
        }
#undef ORBC_EVAL
#undef ORBC_EVAL_N
        launches++;
        CK(cudaGetLastError());
        toc();
        tic("bonds");
        const int nbb = (nbond + 255) / 256, nov = 76;
#define ORBC_BONDS(Z, S)                                                                                              \
    do {                                                                                                              \
        if (energies) k_bonds_overflow<Z, S, true><<<nbb + nov, 256, 0, stream>>>(v, nbb, d_novf, d_novf_n, ovf_cap, d_rowoff, d_energy); \
        else k_bonds_overflow<Z, S><<<nbb + nov, 256, 0, stream>>>(v, nbb, d_novf, d_novf_n, ovf_cap, d_rowoff, nullptr); \
    } while (0)
        if (any_mp()) ORBC_BONDS(0, true);
        else if (z4 && s0z) ORBC_BONDS(4, false);
        else if (z4) ORBC_BONDS(4, true);
        else ORBC_BONDS(0, true);
#undef ORBC_BONDS
        launches++;
        CK(cudaGetLastError());
        toc();
        launch_volume(energies);
        return;
    }
    if (dump || !force_f64()) {
        // (the pair set is the same at every precision)
        tic("pairs");
        if (dump) k_pairs<false, true, 0, true><<<g, t, 0, stream>>>(v, d_energy, d_dump, d_dump_count, dump_cap);
        else if (z4 && s0z) k_pairs<true, false, 4, false><<<g, t, 0, stream>>>(v, d_energy, nullptr, nullptr, 0);
        else if (z4) k_pairs<true, false, 4, true><<<g, t, 0, stream>>>(v, d_energy, nullptr, nullptr, 0);
        else k_pairs<true, false, 0, true><<<g, t, 0, stream>>>(v, d_energy, nullptr, nullptr, 0);
        launches++;
        CK(cudaGetLastError());
        toc();
    }
    if (force_f64()) {
        tic("pairs");
        CK(cudaMemsetAsync(d_F, 0, sizeof(long long) * 3 * (size_t)N, stream));
        CK(cudaMemsetAsync(d_T, 0, sizeof(long long) * 3 * (size_t)N, stream));
#define ORBC_PAIRS_D(MP, Z4, S, EN)                                                                                   \
    k_pair_search<MP, true, Z4, S, EN><<<g, t, 0, stream>>>(v, nullptr, nullptr, 0, nullptr, nullptr, 0, nullptr, d_energy, inst_h[0])
        if (!any_mp() && z4 && s0z) { if (energies) ORBC_PAIRS_D(false, true, false, true); else ORBC_PAIRS_D(false, true, false, false); }
        else { if (energies) ORBC_PAIRS_D(true, false, true, true); else ORBC_PAIRS_D(true, false, true, false); }
#undef ORBC_PAIRS_D
        launches++;
        CK(cudaGetLastError());
        toc();
    }
    tic("bonds");
    const int nb = (int)((std::max(nbond, 1) + 255) / 256);
    if (!force_f64()) {
        if (energies) k_bonds<float, true><<<nb, 256, 0, stream>>>(v, d_energy, nullptr);
        else k_bonds<float, false><<<nb, 256, 0, stream>>>(v, d_energy, nullptr);
    } else {
        if (energies) k_bonds<double, true><<<nb, 256, 0, stream>>>(v, d_energy, nullptr);
        else k_bonds<double, false><<<nb, 256, 0, stream>>>(v, d_energy, nullptr);
    }
    launches++;
    CK(cudaGetLastError());
    toc();
    // (also after a dump: it writes F and T anew, and the next step starts
    // from them)
    launch_volume(energies);
}

void Ensemble::launch_pairs_step(bool msums) {
    View v = view();
    bool z4 = true, s0z = true;
    for (auto& I : inst_h) { z4 = z4 && I.zeta == 4; s0z = s0z && I.s0_d == 0.0; }
    prefer_shared_all();
    launch_search();
    tic("pairs_step");
    // what the epilogue cannot compute from a particle's own list goes to
    // the side array first: bonds, listed pairs beyond the lists' capacity;
    // then the constrained volume
    const int nb = (int)((std::max(nbond, 1) + 255) / 256);
    k_bonds<float, false><<<nb, 256, 0, stream>>>(v, d_energy, d_sflag);
    if (z4 && s0z) k_pair_overflow<4, false><<<152, 128, 0, stream>>>(v, d_novf, d_novf_n, ovf_cap, d_rowoff, d_sflag);
    else if (z4) k_pair_overflow<4, true><<<152, 128, 0, stream>>>(v, d_novf, d_novf_n, ovf_cap, d_rowoff, d_sflag);
    else k_pair_overflow<0, true><<<152, 128, 0, stream>>>(v, d_novf, d_novf_n, ovf_cap, d_rowoff, d_sflag);
    launches += 2;
    launch_volume_sum();
    long long* ms = msums ? d_msum : nullptr;
    int* mc = msums ? d_mcnt : nullptr;
    const View o = view_alt();
    const int ng = (int)((N + 127) / 128);
    const bool d = !step_f32();
#define ORBC_EVAL_STEP(Z, S, D) \
    k_pair_eval_step<Z, S, D><<<ng, 128, 0, stream>>>(v, o, d_nlist, d_ncnt, list_cap, d_rowoff, d_sflag, d_step, ms, mc, \
                                                     d_cell_tmp, d_rot_n)
    if (z4 && s0z) { if (d) ORBC_EVAL_STEP(4, false, true); else ORBC_EVAL_STEP(4, false, false); }
    else if (z4) { if (d) ORBC_EVAL_STEP(4, true, true); else ORBC_EVAL_STEP(4, true, false); }
    else { if (d) ORBC_EVAL_STEP(0, true, true); else ORBC_EVAL_STEP(0, true, false); }
#undef ORBC_EVAL_STEP
    launches++;
    CK(cudaGetLastError());
    toc();
    if (d) {
        k_rot_rest<<<152, 128, 0, stream>>>(v, o, d_step, 1, d_cell_tmp, d_rot_n);
        launches++;
    }
    swap_state();
    k_step_advance<<<1, 64, 0, stream>>>(d_step, B, 1, d_rot_n);
    launches++;
    CK(cudaGetLastError());
    forces_valid = false;   // F and T belong to the positions before the update
}

}  // namespace orbc
