// labf_dyn.cuh -- per-term, per-walker and per-stage device work shared by
// the separate kernels (k_dyn.cu) and the fused pair launch (k_pairs.cu).
#pragma once
#include "labf_internal.cuh"

namespace labf {

// -------------------------------------------------------------------------
// gate of the batched step, after the integrator: a walker whose pruning was
// requested is re-pruned by this step's pair pass (prune_now = 1 + step
// counter; the next integrator step takes the positions it starts from as the
// walker's new reference).  When some walker must rebuild, the walkers whose
// systems are due soon (near flags) join it (coalescing).  Inside a CUDA
// graph one thread also sets the step's conditional handle to "some walker
// must rebuild", so that the graph skips the list kernels otherwise; such
// steps are counted in counters[6].
// -------------------------------------------------------------------------
__device__ __forceinline__ void coalesce_rebuilds(const Dev &d, int w0, int w1, int any) {
    if (!any) return;
    for (int w = w0 + threadIdx.x; w < w1; w += blockDim.x)
        if (__ldcg(d.near + w)) d.rebuild[w] = 1;
}

// by one block; the flags may come from other SMs of the launch: read past L1
__device__ __forceinline__ void gate_work(const Dev &d, int w0, int w1, cudaGraphConditionalHandle handle,
                                          int conditional) {
    __shared__ int any;
    if (threadIdx.x == 0) any = 0;
    __syncthreads();
    for (int w = w0 + threadIdx.x; w < w1; w += blockDim.x) {
        const int p = __ldcg(d.prune + w);
        d.prune_now[w] = p ? d.step[w] + 1ull : 0ull;
        if (p) {
            d.prune[w] = 0;
            atomicAdd(&d.counters[10], 1ull);
        }
        if (__ldcg(d.rebuild + w)) any = 1;
    }
    __syncthreads();
    coalesce_rebuilds(d, w0, w1, any);
    if (conditional && threadIdx.x == 0) {
        cudaGraphSetConditional(handle, any ? 1u : 0u);
        if (any) atomicAdd(&d.counters[6], 1ull);
    }
}

// ---------------------------------------------------------------------------
// bonds (1/2 k (r - r0)^2), angles (1/2 k (theta - theta0)^2) and positional
// restraints (1/2 k |x - x0|^2): term t of the bonded items of walkers
// [w0, w1); with ENERGY the term's energy in fixed point and its index
// ---------------------------------------------------------------------------
template <bool ENERGY>
__device__ __forceinline__ void bonded_term(const Dev &d, int t, int w0, int w1, long long &fix, int &key) {
    int lo = w0, hi = w1 - 1;  // walker owning item t
    while (lo < hi) {
        int mid = (lo + hi + 1) >> 1;
        if (d.walk[mid].bo_off <= t) lo = mid; else hi = mid - 1;
    }
    const int w = lo;
    const WalkerDev &W = d.walk[w];
    const SysDev &S = d.sys[W.sys];
    const int *soa = d.slot_of_atom + W.atom_base;
    int k = t - W.bo_off;
    float e = 0.f;
    int eterm = 4;
    if (k < S.n_bonds) {
        const int2 ij = d.bond_ij[S.bond_off + k];
        const float2 p = d.bond_p[S.bond_off + k];
        const int gi = checked_slot(d, soa[ij.x]), gj = checked_slot(d, soa[ij.y]);
        const float4 xi = d.xq[gi], xj = d.xq[gj];
        float dx = min_image(xi.x - xj.x, S.boxf, S.box_invf);
        float dy = min_image(xi.y - xj.y, S.boxf, S.box_invf);
        float dz = min_image(xi.z - xj.z, S.boxf, S.box_invf);
        float r = sqrtf(dx * dx + dy * dy + dz * dz);
        float dr = r - p.x;
        float fs = -p.y * dr / r;
        add_force(d, gi, fs * dx, fs * dy, fs * dz);
        add_force(d, gj, -fs * dx, -fs * dy, -fs * dz);
        if (ENERGY) e = 0.5f * p.y * dr * dr;
    } else if ((k -= S.n_bonds) < S.n_angles) {
        const int4 ijk = d.angle_ijk[S.angle_off + k];
        const float2 p = d.angle_p[S.angle_off + k];
        const int gi = checked_slot(d, soa[ijk.x]), gj = checked_slot(d, soa[ijk.y]), gk = checked_slot(d, soa[ijk.z]);
        const float4 xi = d.xq[gi], xj = d.xq[gj], xk = d.xq[gk];
        float ux = min_image(xi.x - xj.x, S.boxf, S.box_invf);
        float uy = min_image(xi.y - xj.y, S.boxf, S.box_invf);
        float uz = min_image(xi.z - xj.z, S.boxf, S.box_invf);
        float vx = min_image(xk.x - xj.x, S.boxf, S.box_invf);
        float vy = min_image(xk.y - xj.y, S.boxf, S.box_invf);
        float vz = min_image(xk.z - xj.z, S.boxf, S.box_invf);
        float nu2 = ux * ux + uy * uy + uz * uz, nv2 = vx * vx + vy * vy + vz * vz;
        float inu = rsqrtf(nu2), inv = rsqrtf(nv2);
        float cs = (ux * vx + uy * vy + uz * vz) * inu * inv;
        cs = fminf(1.f, fmaxf(-1.f, cs));
        float th = acosf(cs);
        float dth = th - p.x;
        float sn = sqrtf(fmaxf(1.f - cs * cs, 1e-12f));
        float g = p.y * dth / sn;  // dU/dtheta / sin(theta)
        float a11 = g * inu * inv, a12 = g * cs * inu * inu, a22 = g * cs * inv * inv;
        float fix = a11 * vx - a12 * ux, fiy = a11 * vy - a12 * uy, fiz = a11 * vz - a12 * uz;
        float fkx = a11 * ux - a22 * vx, fky = a11 * uy - a22 * vy, fkz = a11 * uz - a22 * vz;
        add_force(d, gi, fix, fiy, fiz);
        add_force(d, gk, fkx, fky, fkz);
        add_force(d, gj, -fix - fkx, -fiy - fky, -fiz - fkz);
        if (ENERGY) {
            e = 0.5f * p.y * dth * dth;
            eterm = 5;
        }
    } else {
        k -= S.n_angles;
        const int ai = d.posres_idx[S.posres_off + k];
        const float4 x0 = d.posres_x0[S.posres_off + k];
        const int gi = checked_slot(d, soa[ai]);
        const float4 xi = d.xq[gi];
        float dx = min_image(xi.x - x0.x, S.boxf, S.box_invf);
        float dy = min_image(xi.y - x0.y, S.boxf, S.box_invf);
        float dz = min_image(xi.z - x0.z, S.boxf, S.box_invf);
        add_force(d, gi, -S.posres_k * dx, -S.posres_k * dy, -S.posres_k * dz);
        if (ENERGY) {
            e = 0.5f * S.posres_k * (dx * dx + dy * dy + dz * dz);
            eterm = 6;
        }
    }
    if (ENERGY) {
        fix = __double2ll_rn((double)e * E_TO_FIX);
        key = N_ETERMS * w + eterm;
    }
}

// adds the lanes' fixed-point energies (key: index of eterm, -1: none) with
// one atomic per warp and kind of term; integer sums give the same bits in any
// order.  Per-term atomics on one address took 14-22 us for 16 k-33 k terms.
__device__ __forceinline__ void add_energies(const Dev &d, long long fix, int key) {
    constexpr unsigned ALL = 0xffffffffu;
    for (unsigned rest = __ballot_sync(ALL, key >= 0); rest;) {
        const int k0 = __shfl_sync(ALL, key, __ffs(rest) - 1);
        const bool in = key == k0;
        // 26-bit pieces: 32 of them fit a 32-bit sum
        const unsigned lo = __reduce_add_sync(ALL, in ? (unsigned)fix & 0x3ffffffu : 0u);
        const unsigned mid = __reduce_add_sync(ALL, in ? (unsigned)(fix >> 26) & 0x3ffffffu : 0u);
        const int hi = __reduce_add_sync(ALL, in ? (int)(fix >> 52) : 0);
        if ((threadIdx.x & 31) == 0)
            atomicAdd((unsigned long long *)&d.eterm[k0],
                      ((unsigned long long)(long long)hi << 52) + ((unsigned long long)mid << 26) + lo);
        rest &= ~__ballot_sync(ALL, in);
    }
}

// ---------------------------------------------------------------------------
// per walker, one warp: flat-bottom COM restraint, lambda-dependent distance
// restraint and lambda-switched well.  Their forces are added, and their
// dU/dlambda, energy and k1 derivatives go to wdir (lane-strided loops and
// fixed shuffle trees: the result is deterministic).  They need only the
// positions and lambda, so the fused launch runs them beside the alchemical
// items instead of after them.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void walker_restraints(const Dev &d, int w, int lane) {
    const WalkerDev &W = d.walk[w];
    const SysDev &S = d.sys[W.sys];
    double2 *out = reinterpret_cast<double2 *>(d.wdir + 4 * (size_t)w);
    if (!(S.n_fb_a > 0 && S.n_fb_b > 0) && S.n_lr <= 0 && S.n_lh <= 0) {
        if (lane < 2) out[lane] = make_double2(0.0, 0.0);
        return;
    }
    const int *soa = d.slot_of_atom + W.atom_base;
    double e_rest = 0.0;

    // ---- flat-bottom restraint on |COM_a - COM_b| ----
    if (S.n_fb_a > 0 && S.n_fb_b > 0) {
        double com[2][4];
        for (int grp = 0; grp < 2; ++grp) {
            const int off = S.fb_off + (grp ? S.n_fb_a : 0);
            const int ng = grp ? S.n_fb_b : S.n_fb_a;
            const float4 r0 = d.xq[checked_slot(d, soa[d.fb_idx[off]])];
            double acc[4] = {0, 0, 0, 0};
            for (int k = lane; k < ng; k += 32) {
                const int a = d.fb_idx[off + k];
                const float4 xa = d.xq[checked_slot(d, soa[a])];
                const double m = 1.0 / (double)d.ap[S.atom_off + a].w;
                acc[0] += m * min_image(xa.x - r0.x, S.boxf, S.box_invf);
                acc[1] += m * min_image(xa.y - r0.y, S.boxf, S.box_invf);
                acc[2] += m * min_image(xa.z - r0.z, S.boxf, S.box_invf);
                acc[3] += m;
            }
            for (int c = 0; c < 4; ++c) com[grp][c] = warp_sum(acc[c]);
            com[grp][0] = r0.x + com[grp][0] / com[grp][3];
            com[grp][1] = r0.y + com[grp][1] / com[grp][3];
            com[grp][2] = r0.z + com[grp][2] / com[grp][3];
        }
        double dv[3];
        for (int c = 0; c < 3; ++c) {
            const double t = com[0][c] - com[1][c];
            dv[c] = t - S.box * nearbyint(t * S.box_inv);
        }
        const double dd = sqrt(dv[0] * dv[0] + dv[1] * dv[1] + dv[2] * dv[2]);
        if (dd > S.fb_d0) {
            const double ex = dd - S.fb_d0;
            const double fmag = S.fb_k * ex / dd;
            for (int grp = 0; grp < 2; ++grp) {
                const int off = S.fb_off + (grp ? S.n_fb_a : 0);
                const int ng = grp ? S.n_fb_b : S.n_fb_a;
                const double sgn = grp ? 1.0 : -1.0;
                const double mt = com[grp][3];
                for (int k = lane; k < ng; k += 32) {
                    const int a = d.fb_idx[off + k];
                    const double wgt = (1.0 / (double)d.ap[S.atom_off + a].w) / mt;
                    add_force(d, checked_slot(d, soa[a]), (float)(sgn * fmag * dv[0] * wgt), (float)(sgn * fmag * dv[1] * wgt),
                              (float)(sgn * fmag * dv[2] * wgt));
                }
            }
            e_rest = 0.5 * S.fb_k * ex * ex;
        }
    }

    double dl_dir = 0.0, e_lh = 0.0, dk1 = 0.0, d2k1 = 0.0;
    // ---- lambda-dependent distance restraint (Sec. 4.2): pairs kept at
    // least d_min = delta/2 (1 - cos 2 pi lambda) apart ----
    if (S.n_lr > 0) {
        const double lam = d.lam[w];
        const double dmin = 0.5 * S.lr_delta * (1.0 - cospi(2.0 * lam));
        const double ddmin = S.lr_delta * 3.14159265358979323846 * sinpi(2.0 * lam);
        for (int k = lane; k < S.n_lr; k += 32) {
            const int2 ab = d.lr_ij[S.lr_off + k];
            const int ga = checked_slot(d, soa[ab.x]), gb = checked_slot(d, soa[ab.y]);
            const float4 xa = d.xq[ga], xb = d.xq[gb];
            const float dx = min_image(xa.x - xb.x, S.boxf, S.box_invf);
            const float dy = min_image(xa.y - xb.y, S.boxf, S.box_invf);
            const float dz = min_image(xa.z - xb.z, S.boxf, S.box_invf);
            const double r = sqrt((double)dx * dx + (double)dy * dy + (double)dz * dz);
            if (r < dmin) {
                const double ex = r - dmin;
                e_lh += 0.5 * S.lr_k * ex * ex;
                dl_dir += -S.lr_k * ex * ddmin;
                const float fs = (float)(-S.lr_k * ex / r);
                add_force(d, ga, fs * dx, fs * dy, fs * dz);
                add_force(d, gb, -fs * dx, -fs * dy, -fs * dz);
            }
        }
    }
    // ---- lambda-switched harmonic well (uses lambda itself) ----
    if (S.n_lh > 0) {
        const double lam = d.lam[w];
        const double kl = (1.0 - lam) * S.lh_k0 + lam * S.lh_k1;
        for (int k = lane; k < S.n_lh; k += 32) {
            const int a = d.lh_idx[S.lh_off + k];
            const int g = checked_slot(d, soa[a]);
            const float4 xa = d.xq[g], x0 = d.lh_x0[S.lh_off + k];
            float dx = min_image(xa.x - x0.x, S.boxf, S.box_invf);
            float dy = min_image(xa.y - x0.y, S.boxf, S.box_invf);
            float dz = min_image(xa.z - x0.z, S.boxf, S.box_invf);
            if (S.lh_dims < 3) dz = 0.f;
            if (S.lh_dims < 2) dy = 0.f;
            const double r2 = (double)dx * dx + (double)dy * dy + (double)dz * dz;
            add_force(d, g, (float)(-kl * dx), (float)(-kl * dy), (float)(-kl * dz));
            dl_dir += 0.5 * (S.lh_k1 - S.lh_k0) * r2;
            e_lh += 0.5 * kl * r2;
            dk1 += 0.5 * lam * r2;
            d2k1 += 0.5 * r2;
        }
    }
    const double v0 = warp_sum(dl_dir), v1 = warp_sum(e_lh) + e_rest, v2 = warp_sum(dk1), v3 = warp_sum(d2k1);
    if (lane == 0) {
        out[0] = make_double2(v0, v1);
        out[1] = make_double2(v2, v3);
    }
}

// dU/dlambda from the partials (one expression for every form of the step)
__device__ __forceinline__ double sample_of(double dlv, double sv, double dle, double se, double direct) {
    return __dadd_rn(__fma_rn(dlv, sv, __dmul_rn(dle, se)), direct);
}

// Sum over the walker's alchemical atoms of component c of their partial sums
// (written by other SMs of the launch: read past L1), by four neighbouring
// lanes: lane q of the four adds the atoms r = q mod 4 in order, then the
// four are added as (0 + 1) + (2 + 3).  Every form of the step adds so, hence
// the same bits.  Four short chains of FP64 adds and loads instead of one.
__device__ __forceinline__ double alch_sum4(const Dev &d, int alch_base, int n_alch, int c, int q, bool on) {
    const double *o = d.alch_out + 4 * (size_t)alch_base + c;
    double v = 0.0;
    if (on) {
#pragma unroll 4
        for (int r = q; r < n_alch; r += 4) v += __ldcg(o + 4 * r);
    }
    v += __shfl_xor_sync(0xffffffffu, v, 1);
    return v + __shfl_xor_sync(0xffffffffu, v, 2);
}

// value and lambda derivative of theta parameter p (3 per alchemical atom,
// then k1) of walker w
__device__ __forceinline__ void theta_terms(const Dev &d, const WalkerDev &W, const SysDev &S, int w, int p, double dlv,
                                            double dle, double &th, double &d2) {
    if (p == S.P - 1) {
        const double2 k1 = __ldcg(reinterpret_cast<const double2 *>(d.wdir + 4 * (size_t)w) + 1);
        th = k1.x;
        d2 = k1.y;
        return;
    }
    const int r = p / 3, c = p - 3 * r;
    const double *o = d.alch_th + 6 * (size_t)(W.alch_base + r) + c;
    th = __ldcg(o);
    d2 = (c < 2 ? dlv : dle) * __ldcg(o + 3);
}

// the walker's sample from the partial sums of its alchemical atoms and its
// restraints, one warp; with ENERGY also the energy terms and the theta
// derivatives
template <bool ENERGY>
__device__ __forceinline__ void walker_sample(const Dev &d, int w, int lane) {
    const WalkerDev &W = d.walk[w];
    const SysDev &S = d.sys[W.sys];
    double lv, le, dlv, dle;
    lambda_path(d.lam[w], S.b_v, S.b_e, lv, le, dlv, dle);
    // four lanes per component
    const double v = alch_sum4(d, W.alch_base, S.n_alch, (lane >> 2) & 3, lane & 3, lane < (ENERGY ? 16 : 8));
    const double se = __shfl_sync(0xffffffffu, v, 4), usc = __shfl_sync(0xffffffffu, v, 8),
                 urf = __shfl_sync(0xffffffffu, v, 12);
    const double *dir = d.wdir + 4 * (size_t)w;
    if (lane == 0) {
        d.s[w] = sample_of(dlv, v, dle, se, __ldcg(dir));
        if (ENERGY) {
            long long *et = d.eterm + N_ETERMS * w;
            atomicAdd((unsigned long long *)&et[2], (unsigned long long)__double2ll_rn(usc * E_TO_FIX));
            atomicAdd((unsigned long long *)&et[3], (unsigned long long)__double2ll_rn(urf * E_TO_FIX));
            atomicAdd((unsigned long long *)&et[6], (unsigned long long)__double2ll_rn(__ldcg(dir + 1) * E_TO_FIX));
        }
    }
    if (ENERGY) {
        double *th = d.wth + (size_t)w * 2 * d.P_max;
        for (int p = lane; p < S.P; p += 32) theta_terms(d, W, S, w, p, dlv, dle, th[p], th[d.P_max + p]);
    }
}

// restraints and sample of a walker, one warp (one-task launches)
__device__ __forceinline__ void walker_work(const Dev &d, int w, int lane) {
    walker_restraints(d, w, lane);
    __syncwarp();
    walker_sample<false>(d, w, lane);
}

// ---------------------------------------------------------------------------
// ABF: fold the samples of a stage's walkers, merge every shared_freq steps,
// bias = min(1, n/n_full) * mean, final B of lambda.  One warp per stage,
// lane = walker, 32 walkers at a time.
// prime = 1: only G = -s + bias (no sample, no step).
// SAMPLE: the samples are computed here from the alchemical partials (fused
// launch), otherwise walker_work has left them in s.
// ---------------------------------------------------------------------------
__device__ __forceinline__ double abf_bias(const SysDev &S, double sum, double cnt) {
    if (!S.abf_on || cnt <= 0.0) return 0.0;
    return fmin(1.0, cnt / S.n_full) * sum / cnt;
}

template <bool SAMPLE>
__device__ __forceinline__ void lambda_work(const Dev &d, int si, int prime, int lane) {
    constexpr unsigned ALL = 0xffffffffu;
    const StageDev &st = d.stage[si];
    const int w0 = st.w0, nw = st.w1 - st.w0;
    if (nw <= 0) return;  // (create refuses stages without walkers)
    const SysDev &S = d.sys[st.sys];
    const int K = S.shared_freq;  // 0: merged only by the host (la_abf_import)
    const bool one = nw <= 32;    // the walkers' values stay in registers
    double s = 0.0, sum = 0.0, plam = 0.0;
    unsigned long long cnt = 0, stepn = 0;
    int k = -1;
    if (!prime) {
        for (int b = 0; b < nw; b += 32) {
            const int w = w0 + b + lane;
            const bool on = b + lane < nw;
            double dlv = 0.0, dle = 0.0;
            k = -1;
            s = 0.0;
            double sv = 0.0, se = 0.0;
            if (SAMPLE) {  // four lanes per walker, eight walkers at a time
                for (int q = 0; q < 32 && b + q < nw; q += 8) {
                    const int v = b + q + (lane >> 2);
                    const bool von = v < nw;
                    const int base = von ? d.walk[w0 + v].alch_base : 0;
                    const double a = alch_sum4(d, base, S.n_alch, 0, lane & 3, von);
                    const double e = alch_sum4(d, base, S.n_alch, 1, lane & 3, von);
                    const double a8 = __shfl_sync(ALL, a, 4 * (lane & 7)), e8 = __shfl_sync(ALL, e, 4 * (lane & 7));
                    if ((lane & 24) == q) {
                        sv = a8;
                        se = e8;
                    }
                }
            }
            if (on) {
                const double lam = d.lam[w];
                plam = d.plam[w];
                stepn = d.step[w];
                if (SAMPLE || S.theta_stats) {
                    double lv, le;
                    lambda_path(lam, S.b_v, S.b_e, lv, le, dlv, dle);
                }
                if (SAMPLE) {
                    s = sample_of(dlv, sv, dle, se, __ldcg(d.wdir + 4 * (size_t)w));
                    d.s[w] = s;
                } else {
                    s = __ldcg(d.s + w);
                }
                k = bin_of(lam, st);
            }
            if (K == 1) {
                // every step merges: the walker-local statistics are zero before
                // the fold and again after it, so the samples go straight to the
                // shared ones, a bin's walkers in order by the bin's first lane
                const unsigned grp = __match_any_sync(ALL, k);
                const int lead = __ffs(grp) - 1;
                const bool mine = on && lane == lead;
                double s2 = 0.0;
                if (mine) {
                    sum = d.abf_sum[st.bin_off + k];
                    s2 = d.abf_sumsq[st.bin_off + k];
                    cnt = d.abf_count[st.bin_off + k];
                }
                for (unsigned rest = grp; __any_sync(ALL, mine && rest); rest &= rest - 1u) {
                    const double v = __shfl_sync(ALL, s, rest ? __ffs(rest) - 1 : 0);
                    if (mine && rest) {
                        sum = __dadd_rn(sum, v);
                        s2 = __dadd_rn(s2, __dmul_rn(v, v));
                        ++cnt;
                    }
                }
                if (mine) {
                    d.abf_sum[st.bin_off + k] = sum;
                    d.abf_sumsq[st.bin_off + k] = s2;
                    d.abf_count[st.bin_off + k] = cnt;
                }
                sum = __shfl_sync(ALL, sum, lead);
                cnt = __shfl_sync(ALL, cnt, lead);
            } else if (on) {  // each walker's own statistics
                const size_t lk = (size_t)w * d.max_bins + k;
                d.dl_sum[lk] = __dadd_rn(d.dl_sum[lk], s);
                d.dl_sumsq[lk] = __dadd_rn(d.dl_sumsq[lk], __dmul_rn(s, s));
                d.dl_count[lk] += 1ull;
            }
            if (S.theta_stats) {
                // per parameter (lane), walkers in order; a run of walkers in one
                // bin keeps the bin's sums in registers
                const int n = min(32, nw - b);
                for (int p0 = 0; p0 < S.P; p0 += 32) {
                    const int p = p0 + lane;
                    int cur = -1;
                    double t2 = 0.0, t1 = 0.0, ts = 0.0;
                    for (int j = 0; j < n; ++j) {
                        const int kj = __shfl_sync(ALL, k, j);
                        const double sj = __shfl_sync(ALL, s, j), vj = __shfl_sync(ALL, dlv, j),
                                     ej = __shfl_sync(ALL, dle, j);
                        if (p >= S.P) continue;
                        double th, d2;
                        theta_terms(d, d.walk[w0 + b + j], S, w0 + b + j, p, vj, ej, th, d2);
                        if (kj != cur) {
                            if (cur >= 0) {
                                const size_t q = (size_t)(st.bin_off + cur) * d.P_max + p;
                                d.th_d2[q] = t2;
                                d.th_d[q] = t1;
                                d.th_sd[q] = ts;
                            }
                            const size_t q = (size_t)(st.bin_off + kj) * d.P_max + p;
                            t2 = d.th_d2[q];
                            t1 = d.th_d[q];
                            ts = d.th_sd[q];
                            cur = kj;
                        }
                        t2 += d2;
                        t1 += th;
                        ts += sj * th;
                    }
                    if (cur >= 0) {
                        const size_t q = (size_t)(st.bin_off + cur) * d.P_max + p;
                        d.th_d2[q] = t2;
                        d.th_d[q] = t1;
                        d.th_sd[q] = ts;
                    }
                }
            }
            // the next 32 walkers' leaders, and the merge below, read what these
            // lanes stored (shuffles and votes do not order memory)
            __syncwarp();
        }
        if (K > 1 && (d.step[w0] + 1ull) % (unsigned long long)K == 0ull) {
            for (int q = lane; q < st.n_bins; q += 32) {
                double s1 = d.abf_sum[st.bin_off + q], s2 = d.abf_sumsq[st.bin_off + q];
                unsigned long long c = d.abf_count[st.bin_off + q];
                for (int w = w0; w < st.w1; ++w) {
                    const size_t lk = (size_t)w * d.max_bins + q;
                    s1 += d.dl_sum[lk];
                    s2 += d.dl_sumsq[lk];
                    c += d.dl_count[lk];
                    d.dl_sum[lk] = 0.0;
                    d.dl_sumsq[lk] = 0.0;
                    d.dl_count[lk] = 0ull;
                }
                d.abf_sum[st.bin_off + q] = s1;
                d.abf_sumsq[st.bin_off + q] = s2;
                d.abf_count[st.bin_off + q] = c;
            }
        }
        __syncwarp();
    }
    for (int b = 0; b < nw; b += 32) {
        const int w = w0 + b + lane;
        if (b + lane >= nw) continue;
        if (prime || !one) {
            s = __ldcg(d.s + w);
            k = bin_of(d.lam[w], st);
            plam = d.plam[w];
            stepn = d.step[w];
        }
        if (prime || !one || K != 1) {
            const size_t lk = (size_t)w * d.max_bins + k;
            sum = d.abf_sum[st.bin_off + k] + d.dl_sum[lk];
            cnt = d.abf_count[st.bin_off + k] + d.dl_count[lk];
        }
        const double G = -s + abf_bias(S, sum, (double)cnt);
        d.G[w] = G;
        if (!prime) {
            if (S.lambda_dynamics) d.plam[w] = plam + 0.5 * S.dt_d * G;
            d.step[w] = stepn + 1ull;
            d.pending[w] = 1;
        }
    }
}

}  // namespace labf
