// labf_launch.h -- host-side launchers shared by the translation units.
#pragma once

#include <cuda_runtime.h>

#include "labf_internal.cuh"

#define LA_MAX_WALKERS_PER_LAUNCH LA_MAX_WALKERS

namespace labf {

// Host copies of the per-walker offsets the launchers size grids with.
struct HostView {
    int n_walkers = 0, n_sm = 0, pair_blocks = 0;
    int pair_variant = 0;  // 0: 8 warps/CTA, 80 regs; 1: 4 warps, 72; 2: 4 warps, 64
    const int *slot_off = nullptr, *slot_cap = nullptr, *sc_cap = nullptr, *n_cols = nullptr;
    const int *alch_base = nullptr, *n_alch = nullptr;
    const int *bo_off = nullptr, *n_bo = nullptr;
    const volatile int *items = nullptr;  // pair work items per walker, as the last integrator launch met them
};

void launch_integrate(const Dev &d, const HostView &hv, int w0, int w1, cudaStream_t s);
void launch_finish(const Dev &d, const HostView &hv, int w0, int w1, cudaStream_t s);
// batched: the batched step's chain (fresh lists are pruned by its pair pass)
void launch_rebuild(const Dev &d, const HostView &hv, int w0, int w1, cudaStream_t s, bool batched = false);
void launch_items(const Dev &d, const HostView &hv, int w0, int w1, cudaStream_t s);
// conditional: also set the graph's conditional handle (false outside graphs)
void launch_gate(const Dev &d, int w0, int w1, cudaGraphConditionalHandle handle, bool conditional,
                 cudaStream_t s);
// integrator and gate in one launch (gate_in_integrate) or two
bool gate_in_integrate(const HostView &hv, int w0, int w1);
void launch_integrate_gate(const Dev &d, const HostView &hv, int w0, int w1, cudaGraphConditionalHandle handle,
                           bool conditional, cudaStream_t s);
int rebuild_kernel_count(const HostView &hv, int w0, int w1);
// rebuild coalescing of the one-walker-per-launch form (the batched step's
// gate does the same)
void launch_coalesce(const Dev &d, int w0, int w1, cudaStream_t s);
void launch_pairs(const Dev &d, const HostView &hv, int w0, int w1, cudaStream_t s);
// pairs, bonded terms and restraints of one walker with energies and derivatives
void launch_pairs_energy(const Dev &d, const HostView &hv, int w, cudaStream_t s);
// whether a pair launch of walkers [w0, w1) takes the latency form now
bool pairs_latency(const HostView &hv, int w0, int w1);
// pairs + bonded + walker terms + lambda update of all walkers in one launch
void launch_pairs_fused(const Dev &d, const HostView &hv, bool latency, cudaStream_t s);
void launch_bonded(const Dev &d, const HostView &hv, int w0, int w1, cudaStream_t s);
void launch_walker(const Dev &d, int w0, int w1, cudaStream_t s);
void launch_lambda(const Dev &d, int s0, int s1, bool prime, cudaStream_t s);
void launch_state_io(const Dev &d, int w, int n, float *x, float *v, bool to_slots, cudaStream_t s);
void launch_states_io(const Dev &d, int rows, float *x, float *v, bool to_slots, cudaStream_t s);
void launch_lambda_path(const double *lam, int n, double bv, double be, double *out, cudaStream_t s);
void launch_ef_in(const Dev &d, int w, int n, int slots, const float *x, const double *theta, const double *lam,
                  bool rebuild, cudaStream_t s);
void launch_ef_out(const Dev &d, int w, int n, int P, double *out, float *forces, cudaStream_t s);

}  // namespace labf
