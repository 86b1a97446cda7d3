// k_io.cu -- state and force transfer between the slot layout and the
// system's atom order, and the lambda-path evaluator.
#include "labf_dyn.cuh"
#include "labf_internal.cuh"
#include "labf_launch.h"

namespace labf {

// to_slots = 0: x, v (atom order) <- slots;  1: slots <- x, v
__global__ void k_state_io(Dev d, int w, int n, float *x, float *v, int to_slots) {
    const WalkerDev &W = d.walk[w];
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const int g = checked_slot(d, d.slot_of_atom[W.atom_base + i]);
        if (to_slots) {
            float4 xq = d.xq[g];
            xq.x = x[3 * i];
            xq.y = x[3 * i + 1];
            xq.z = x[3 * i + 2];
            d.xq[g] = xq;
            d.vv[g] = make_float4(v[3 * i], v[3 * i + 1], v[3 * i + 2], 0.f);
        } else {
            const float4 xq = d.xq[g], vv = d.vv[g];
            x[3 * i] = xq.x;
            x[3 * i + 1] = xq.y;
            x[3 * i + 2] = xq.z;
            v[3 * i] = vv.x;
            v[3 * i + 1] = vv.y;
            v[3 * i + 2] = vv.z;
        }
    }
}

// every walker's x and v in one launch (rows: walkers in order, atom order
// inside; a NULL array is left out).  One launch and one copy per array took
// the place of a launch and two copies per walker: 2.0 ms of a 7.0 ms pass for
// 144 walkers x 772 atoms went to those.
__global__ void k_states_io(Dev d, int rows, float *x, float *v, int to_slots) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < rows; i += gridDim.x * blockDim.x) {
        const int g = checked_slot(d, d.slot_of_atom[i]);
        const size_t o = 3 * (size_t)i;
        if (to_slots) {
            if (x) {
                float4 xq = d.xq[g];
                xq.x = x[o];
                xq.y = x[o + 1];
                xq.z = x[o + 2];
                d.xq[g] = xq;
            }
            if (v) d.vv[g] = make_float4(v[o], v[o + 1], v[o + 2], 0.f);
        } else {
            if (x) {
                const float4 xq = d.xq[g];
                x[o] = xq.x;
                x[o + 1] = xq.y;
                x[o + 2] = xq.z;
            }
            if (v) {
                const float4 vv = d.vv[g];
                v[o] = vv.x;
                v[o + 1] = vv.y;
                v[o + 2] = vv.z;
            }
        }
    }
}

__global__ void k_lambda_path(const double *lam, int n, double bv, double be, double *out) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        double lv, le, dlv, dle;
        lambda_path(lam[i], bv, be, lv, le, dlv, dle);
        out[4 * i] = lv;
        out[4 * i + 1] = le;
        out[4 * i + 2] = dlv;
        out[4 * i + 3] = dle;
    }
}

// -------------------------------------------------------------------------
// One energy evaluation of a walker is [k_ef_in][rebuild chain][pairs, bonded
// terms and restraints][k_ef_out]: every input in the first launch, every
// read-out in the last.  Sixteen smaller launches and copies took 35% more
// host time than the GPU needed for its work on 12 300 atoms.
// -------------------------------------------------------------------------

// before the evaluation: forces and energies cleared; optionally the walker's
// positions (atom order) and lambda, the system's alchemical parameters
// (epsilon, sigma, q; every walker of the system then rebuilds, the per-slot
// copies of the parameters are refreshed there) from device arrays.  rebuild:
// the walker's lists are rebuilt before its forces are evaluated.  Negative or
// non-finite epsilon or sigma: the atom keeps its parameters and
// LA_STATUS_BAD_PARAM is set.
__global__ void k_ef_in(Dev d, int w, int n, const float *x, const double *theta, const double *lam, int rebuild) {
    const WalkerDev &W = d.walk[w];
    const SysDev &S = d.sys[W.sys];
    const int nthr = gridDim.x * blockDim.x, t0 = blockIdx.x * blockDim.x + threadIdx.x;
    unsigned long long *F = d.F + 3 * (size_t)W.slot_off;
    for (int i = t0; i < 3 * W.sc_cap * SC; i += nthr) F[i] = 0ull;
    if (x)
        for (int i = t0; i < n; i += nthr) {
            const int g = checked_slot(d, d.slot_of_atom[W.atom_base + i]);
            float4 xq = d.xq[g];
            xq.x = x[3 * (size_t)i];
            xq.y = x[3 * (size_t)i + 1];
            xq.z = x[3 * (size_t)i + 2];
            d.xq[g] = xq;
        }
    if (blockIdx.x != 0) return;
    if (threadIdx.x < N_ETERMS) d.eterm[(size_t)N_ETERMS * w + threadIdx.x] = 0;
    if (threadIdx.x == 0) {
        if (x || rebuild) d.rebuild[w] = 1;
        if (lam) d.lam[w] = *lam;
    }
    if (!theta) return;
    for (int r = threadIdx.x; r < S.n_alch; r += blockDim.x) {
        const double eps = theta[3 * r], sig = theta[3 * r + 1], q = theta[3 * r + 2];
        if (!(eps >= 0.0) || !(sig >= 0.0) || !(eps < 1e30) || !(sig < 1e30) || !(fabs(q) < 1e30)) {
            set_status(d, LA_STATUS_BAD_PARAM);
            continue;
        }
        const int a = d.alch_atoms[S.alch_off + r];
        float4 p = d.aparam_mut[S.atom_off + a];
        p.x = (float)(q * (double)S.sqrt_coul);
        p.y = (float)(0.5 * sig);
        p.z = (float)(2.0 * sqrt(eps));
        d.aparam_mut[S.atom_off + a] = p;
    }
    for (int v = S.w_first + threadIdx.x; v < S.w_first + S.w_count; v += blockDim.x) d.rebuild[v] = 1;
}

// after the evaluation: block 0 sums the walker's sample, refreshes its
// stage's lambda forces and writes the energies and derivatives to `out` ([0,
// LA_N_TERMS) the energy terms, then U, dU/dlambda, dU/dtheta [P],
// d2U/dlambda dtheta [P]; NULL: left in the engine's arrays); the other
// blocks write the forces in atom order (NULL: none)
__global__ void k_ef_out(Dev d, int w, int n, int P, double *out, float *forces) {
    const WalkerDev &W = d.walk[w];
    if (blockIdx.x != 0) {
        const int nthr = (gridDim.x - 1) * blockDim.x;
        for (int i = (blockIdx.x - 1) * blockDim.x + threadIdx.x; i < n; i += nthr) {
            const int g = checked_slot(d, d.slot_of_atom[W.atom_base + i]);
            const unsigned long long *F = d.F + 3 * (size_t)g;
            const float fx = fix_to_float(F[0]), fy = fix_to_float(F[1]), fz = fix_to_float(F[2]);
            forces[3 * (size_t)i] = fx;
            forces[3 * (size_t)i + 1] = fy;
            forces[3 * (size_t)i + 2] = fz;
            if (fabsf(fx) > FIX_LIMIT || fabsf(fy) > FIX_LIMIT || fabsf(fz) > FIX_LIMIT)
                set_status(d, LA_STATUS_FIXED_OVERFLOW);
        }
        return;
    }
    if (threadIdx.x < 32) {
        walker_sample<true>(d, w, threadIdx.x);
        __syncwarp();
        lambda_work<false>(d, W.stage, 1, threadIdx.x);
        __threadfence();
    }
    __syncthreads();
    if (!out) return;
    const int t = threadIdx.x;
    if (t == 0) {
        double u = 0.0;
        for (int k = 0; k < LA_N_TERMS; ++k) {
            const double e = (double)__ldcg(d.eterm + N_ETERMS * w + k) / E_TO_FIX;
            out[k] = e;
            u += e;
        }
        out[LA_N_TERMS] = u;
        out[LA_N_TERMS + 1] = d.s[w];
    }
    const double *th = d.wth + (size_t)w * 2 * d.P_max;
    for (int p = t; p < P; p += blockDim.x) {
        out[LA_N_TERMS + 2 + p] = th[p];
        out[LA_N_TERMS + 2 + P + p] = th[d.P_max + p];
    }
}

void launch_ef_in(const Dev &d, int w, int n, int slots, const float *x, const double *theta, const double *lam,
                  bool rebuild, cudaStream_t s) {
    k_ef_in<<<(3 * slots + 1023) / 1024, 256, 0, s>>>(d, w, n, x, theta, lam, rebuild ? 1 : 0);
}

void launch_ef_out(const Dev &d, int w, int n, int P, double *out, float *forces, cudaStream_t s) {
    k_ef_out<<<1 + (forces ? (n + 255) / 256 : 0), 256, 0, s>>>(d, w, n, P, out, forces);
}

void launch_state_io(const Dev &d, int w, int n, float *x, float *v, bool to_slots, cudaStream_t s) {
    k_state_io<<<(n + 255) / 256, 256, 0, s>>>(d, w, n, x, v, to_slots ? 1 : 0);
}

void launch_states_io(const Dev &d, int rows, float *x, float *v, bool to_slots, cudaStream_t s) {
    k_states_io<<<(rows + 255) / 256, 256, 0, s>>>(d, rows, x, v, to_slots ? 1 : 0);
}

void launch_lambda_path(const double *lam, int n, double bv, double be, double *out, cudaStream_t s) {
    k_lambda_path<<<(n + 255) / 256, 256, 0, s>>>(lam, n, bv, be, out);
}

}  // namespace labf
