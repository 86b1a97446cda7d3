// k_static.cu -- la_alch_pairs_static: the alchemical part of the pair pass
// with its scratch in a file-scope static device array, for callers that
// cannot allocate device memory (a plugin inside a program that owns the
// GPU memory, or a deployment with a fixed device footprint).
//
// One launch does the pass.  Environment blocks: a thread per atom runs over
// the alchemical atoms (staged in shared memory) and writes the atom's force,
// summed in 64-bit fixed point in registers.  Alchemical blocks: one per
// (group of alchemical atoms, chunk of atoms), whose FP64 partial sums and
// fixed-point forces go to the scratch; the last block of a group adds its
// chunks and the last group its atoms, in fixed orders, so results do not
// depend on the order of the blocks.  The
// distances are computed twice (about 20 instructions per pair of a few
// hundred bytes per atom), which costs less than per-pair atomics and lets
// both sides fill the chip: one warp per alchemical atom over all atoms, as
// before, left 12 warps on 152 SMs.  The pass is bound by instruction issue
// (largest shapes) or by launch latency: 120 200 atoms x 200 alchemical atoms
// 2.29 -> 0.12 ms per call, 12 300 x 12 260 -> 17 us.
//
// The scratch holds the partial sums, the arrival counter and one status word
// (LA_STATUS_* bits: a bad alchemical index, a non-finite distance or force,
// a force beyond the fixed-point range), reported in out[5].  Every call
// clears the last two first.  All calls on a device share the array: calls
// whose GPU work overlaps race, so callers must serialise them.
#include <cuda_runtime.h>

#include <cmath>
#include <cstdio>
#include <mutex>
#include <string>

#include "labf_internal.cuh"

// per alchemical atom 4 doubles and 3 int64 forces of each chunk of atoms, and
// the 4 sums over its chunks; then the status word, the count of finished
// groups and, per group of alchemical atoms, that of finished chunks
#define LA_STATIC_CHUNKS 32
#define LA_STATIC_PART_WORDS (7ull * LA_STATIC_CHUNKS * LA_STATIC_MAX_ALCH)
#define LA_STATIC_SUM_WORDS (4ull * LA_STATIC_MAX_ALCH)
#define LA_STATIC_COUNT_WORDS ((2ull + LA_STATIC_MAX_ALCH) / 2)

// The scratch array (about 1.8 MB on every device that loads the library).
// Host code must not take its address directly: the name is a host-side
// stand-in; the device address comes from cudaGetSymbolAddress.
static __device__ __align__(256) unsigned char g_static_scratch[8 * (LA_STATIC_PART_WORDS + LA_STATIC_SUM_WORDS + LA_STATIC_COUNT_WORDS)];

namespace labf {
namespace {

constexpr int MAX_DEVICES = 64;
std::mutex g_setup_mutex;
void *g_scratch_addr[MAX_DEVICES] = {nullptr};
thread_local std::string g_static_err;

struct StaticParams {
    int n, n_alch;
    float L, Linv, rc2, krf, crf, sqrt_coul;
    float le, lvn, dlvn, sa, dsdl;
};

struct StaticIn {
    const float *x, *q, *sig, *eps;
    const uint8_t *alch;
    const int *grp, *alch_idx;
};

// an alchemical atom; a < 0: not an alchemical atom of this system
struct StaticAlch {
    float x, y, z, q, half_sig, eps2;
    int a, grp;
};

__device__ __forceinline__ StaticAlch load_alch(const StaticParams &p, const StaticIn &in, int r, unsigned *status) {
    StaticAlch A;
    A.a = in.alch_idx[r];
    if ((unsigned)A.a >= (unsigned)p.n || !in.alch[A.a]) {
        atomicOr(status, LA_STATUS_BAD_INDEX);
        A.a = -1;
        A.x = A.y = A.z = A.q = A.half_sig = A.eps2 = 0.f;
        A.grp = -1;
        return A;
    }
    A.x = in.x[3 * (size_t)A.a];
    A.y = in.x[3 * (size_t)A.a + 1];
    A.z = in.x[3 * (size_t)A.a + 2];
    A.q = in.q[A.a] * p.sqrt_coul;
    A.half_sig = 0.5f * in.sig[A.a];
    A.eps2 = 2.0f * sqrtf(fmaxf(in.eps[A.a], 0.f));
    A.grp = in.grp[A.a];
    return A;
}

// largest magnitude of a force's components
__device__ __forceinline__ float static_top(float fx, float fy, float fz) {
    return fmaxf(fabsf(fx), fmaxf(fabsf(fy), fabsf(fz)));
}
// a force that fits the 64-bit fixed-point range, else a status bit
__device__ __forceinline__ bool static_force_ok(float m, unsigned *status) {
    if (m < FIX_LIMIT) return true;
    atomicOr(status, m == m ? LA_STATUS_FIXED_OVERFLOW : LA_STATUS_NONFINITE);
    return false;
}

// minimum image; the nearest integer by adding and taking away 1.5 x 2^23
// (round to nearest even below 2^22, as rintf): the conversion instruction
// runs on the special-function unit at an eighth of the rate (128 -> 119 us
// at the largest shapes)
__device__ __forceinline__ float static_image(float dx, float L, float Linv) {
    constexpr float M = 12582912.0f;
    return dx - L * (fmaf(dx, Linv, M) - M);
}

constexpr int ST_THREADS = 128, ST_WARPS = ST_THREADS / 32;
constexpr int ST_TILE = 64;  // alchemical atoms staged at a time

// Range of an atom's whole force.  Sums of fixed-point forces may wrap: modulo
// 2^64 they are exact whenever the whole force is in range, whatever the parts
// are.  Whether it is in range is asked only of atoms with a part so large that
// their number could carry the sum out of range (BIG_PAIR: at most
// LA_STATIC_MAX_ALCH pairs; BIG_SHARE: warps of a group), and answered by
// adding the pairs once more in FP32.  An environment atom is asked about by its
// own thread, for its force, and by the groups that meet its big pairs, for the
// status: they are through before the status is read (arrivals of the
// environment blocks took 3% of the largest shapes' time).
constexpr float BIG_PAIR = FIX_LIMIT / LA_STATIC_MAX_ALCH, BIG_SHARE = FIX_LIMIT / (LA_STATIC_CHUNKS * ST_WARPS);

struct StaticPair {
    float fs, dx, dy, dz, top, dsc, rf_u, usc;
};

// the pair (A, environment atom b at xb..zb); false when out of reach or skipped
__device__ __forceinline__ bool static_pair(const StaticParams &p, const StaticIn &in, const StaticAlch &A, int b, float xb,
                                            float yb, float zb, int gb, unsigned *status, StaticPair &o) {
    o.dx = static_image(A.x - xb, p.L, p.Linv);
    o.dy = static_image(A.y - yb, p.L, p.Linv);
    o.dz = static_image(A.z - zb, p.L, p.Linv);
    const float r2 = o.dx * o.dx + o.dy * o.dy + o.dz * o.dz;
    if (r2 >= p.rc2 || A.a < 0 || (A.grp >= 0 && gb == A.grp)) return false;
    if (r2 != r2) {
        atomicOr(status, LA_STATUS_NONFINITE);
        return false;
    }
    const float rinv = rsqrtf(r2);
    const float r2inv = rinv * rinv;
    const float qq = A.q * in.q[b] * p.sqrt_coul;
    o.rf_u = qq * (rinv + p.krf * r2 - p.crf);
    const float rf_f = qq * (rinv * r2inv - 2.0f * p.krf);
    const float sg = A.half_sig + 0.5f * in.sig[b];
    const float e4 = A.eps2 * 2.0f * sqrtf(fmaxf(in.eps[b], 0.f));
    float sc_f = 0.f;
    o.usc = o.dsc = 0.f;
    if (e4 > 0.f) {
        const float q2 = r2 / (sg * sg);
        const float rho6 = q2 * q2 * q2;
        const float is = 1.0f / (p.sa + rho6);
        const float g = is * is - is;
        const float g1 = is * is - 2.0f * is * is * is;
        o.usc = p.lvn * e4 * g;
        sc_f = -p.lvn * e4 * g1 * 6.0f * rho6 * r2inv;
        o.dsc = p.dlvn * e4 * g + p.lvn * e4 * g1 * p.dsdl;
    }
    o.fs = sc_f + p.le * rf_f;
    o.top = static_top(o.fs * o.dx, o.fs * o.dy, o.fs * o.dz);
    return static_force_ok(o.top, status);
}

// f 2^32 modulo 2^64 (f2fix clamps at 2^31; a warp's share may be 2^40), by
// shifting the mantissa: the conversion to 64-bit integers runs on the FP64
// pipe (2.5% of the time of 27 100 x 100 atoms)
__device__ __forceinline__ unsigned long long f2fix_wrap(float f) {
    if (fabsf(f) < FIX_LIMIT) return f2fix(f);
    const unsigned bits = __float_as_uint(fabsf(f));
    const unsigned long long v = (unsigned long long)((bits & 0x7fffffu) | 0x800000u) << (((int)(bits >> 23) - 118) & 63);
    return f < 0.f ? 0ull - v : v;
}

// the whole force on environment atom b, by its thread
__device__ __forceinline__ bool env_force_ok(const StaticParams &p, const StaticIn &in, int b, float xb, float yb, float zb,
                                          int gb, unsigned *status) {
    float f[3] = {0.f, 0.f, 0.f};
    for (int r = 0; r < p.n_alch; ++r) {
        StaticPair o;
        if (!static_pair(p, in, load_alch(p, in, r, status), b, xb, yb, zb, gb, status, o)) continue;
        f[0] = fmaf(-o.fs, o.dx, f[0]);
        f[1] = fmaf(-o.fs, o.dy, f[1]);
        f[2] = fmaf(-o.fs, o.dz, f[2]);
    }
    return static_force_ok(static_top(f[0], f[1], f[2]), status);
}

// the whole force on alchemical atom A, by the block; also those on the
// environment atoms of A's big pairs
__device__ __forceinline__ bool alch_force_ok(const StaticParams &p, const StaticIn &in, const StaticAlch &A,
                                           float (&share)[ST_WARPS][3], unsigned *status) {
    float f[3] = {0.f, 0.f, 0.f};
    for (int b = threadIdx.x; b < p.n; b += ST_THREADS) {
        StaticPair o;
        if (in.alch[b] || !static_pair(p, in, A, b, in.x[3 * (size_t)b], in.x[3 * (size_t)b + 1], in.x[3 * (size_t)b + 2],
                                       in.grp[b], status, o))
            continue;
        f[0] = fmaf(o.fs, o.dx, f[0]);
        f[1] = fmaf(o.fs, o.dy, f[1]);
        f[2] = fmaf(o.fs, o.dz, f[2]);
        if (!(o.top < BIG_PAIR))
            env_force_ok(p, in, b, in.x[3 * (size_t)b], in.x[3 * (size_t)b + 1], in.x[3 * (size_t)b + 2], in.grp[b], status);
    }
    __syncthreads();  // share free
    for (int c = 0; c < 3; ++c) {
        const float v = warp_sumf(f[c]);
        if ((threadIdx.x & 31) == 0) share[threadIdx.x >> 5][c] = v;
    }
    __syncthreads();
    for (int c = 0; c < 3; ++c) {
        f[c] = 0.f;
        for (int q = 0; q < ST_WARPS; ++q) f[c] += share[q][c];
    }
    return static_force_ok(static_top(f[0], f[1], f[2]), status);
}

// sum over the warp, on every lane
__device__ __forceinline__ double static_sum(double v, bool any) { return any ? warp_sum(v) : 0.0; }

// RA: alchemical atoms per alchemical block (4 once the grid is full: their
// atoms' loads are shared)
template <int RA>
__global__ void __launch_bounds__(ST_THREADS) k_static(const __grid_constant__ StaticParams p,
                                                       const __grid_constant__ StaticIn in, int n_env_blocks,
                                                       int chunks, unsigned long long *part, double *sums, unsigned *status,
                                                       double dlv, double dle, float *forces, double *out) {
    __shared__ StaticAlch tile[ST_TILE];
    __shared__ double wsum[ST_WARPS][RA][4];
    __shared__ unsigned long long wfix[ST_WARPS][RA][3];
    __shared__ float wforce[ST_WARPS][3];
    __shared__ int last;
    const int tid = threadIdx.x, lane = tid & 31, wib = tid >> 5;
    if ((int)blockIdx.x < n_env_blocks) {
        // ---- environment atoms: force of one atom per thread ----
        const int b = blockIdx.x * ST_THREADS + tid;
        const bool on = b < p.n, env = on && !in.alch[b];
        float xb = 0.f, yb = 0.f, zb = 0.f;
        int gb = -1;
        if (on) {
            xb = in.x[3 * (size_t)b];
            yb = in.x[3 * (size_t)b + 1];
            zb = in.x[3 * (size_t)b + 2];
            gb = in.grp[b];
        }
        unsigned long long f[3] = {0ull, 0ull, 0ull};
        float top = 0.f;
        bool listed = false;  // an alchemical atom whose group writes its force
        for (int r0 = 0; r0 < p.n_alch; r0 += ST_TILE) {
            __syncthreads();
            if (tid < ST_TILE && r0 + tid < p.n_alch) tile[tid] = load_alch(p, in, r0 + tid, status);
            __syncthreads();
            const int nr = min(ST_TILE, p.n_alch - r0);
            for (int r = 0; r < nr; ++r) {
                StaticPair o;
                if (!env) {
                    listed = listed || tile[r].a == b;
                } else if (static_pair(p, in, tile[r], b, xb, yb, zb, gb, status, o)) {
                    f[0] += f2fix(-o.fs * o.dx);
                    f[1] += f2fix(-o.fs * o.dy);
                    f[2] += f2fix(-o.fs * o.dz);
                    top = fmaxf(top, o.top);
                }
            }
        }
        const bool ok = top < BIG_PAIR || env_force_ok(p, in, b, xb, yb, zb, gb, status);
        if (on && !listed)
            for (int c = 0; c < 3; ++c) forces[3 * (size_t)b + c] = ok ? fix_to_float(f[c]) : 0.f;
        return;
    }
    {
        // ---- alchemical atoms [r0, r0 + RA) against one chunk of atoms ----
        const int k = blockIdx.x - n_env_blocks, chunk = k % chunks, r0 = (k / chunks) * RA;
        if (tid < RA && r0 + tid < p.n_alch) tile[tid] = load_alch(p, in, r0 + tid, status);
        __syncthreads();
        const int len = (p.n + chunks - 1) / chunks, b0 = chunk * len, b1 = min(p.n, b0 + len);
        double s[RA][4] = {};
        float fa[RA][3] = {};
        unsigned hit = 0;
        float top = 0.f;
        for (int b = b0 + tid; b < b1; b += ST_THREADS) {
            if (in.alch[b]) continue;
            const float xb = in.x[3 * (size_t)b], yb = in.x[3 * (size_t)b + 1], zb = in.x[3 * (size_t)b + 2];
            const int gb = in.grp[b];
#pragma unroll
            for (int r = 0; r < RA; ++r) {
                StaticPair o;
                if (r0 + r >= p.n_alch || !static_pair(p, in, tile[r], b, xb, yb, zb, gb, status, o)) continue;
                hit |= 1u << r;
                top = fmaxf(top, o.top);
                fa[r][0] = fmaf(o.fs, o.dx, fa[r][0]);
                fa[r][1] = fmaf(o.fs, o.dy, fa[r][1]);
                fa[r][2] = fmaf(o.fs, o.dz, fa[r][2]);
                s[r][0] += (double)o.dsc;
                s[r][1] += (double)o.rf_u;
                s[r][2] += (double)o.usc;
                s[r][3] += (double)(p.le * o.rf_u);
            }
        }
        bool big = !(top < BIG_PAIR);
        hit = __reduce_or_sync(0xffffffffu, hit);
#pragma unroll
        for (int r = 0; r < RA; ++r) {
            const bool any = (hit >> r) & 1u;  // no pair in the warp: its sums are zero
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const double v = static_sum(s[r][c], any);
                if (lane == 0) wsum[wib][r][c] = v;
            }
            float f[3];
#pragma unroll
            for (int c = 0; c < 3; ++c) f[c] = any ? warp_sumf(fa[r][c]) : 0.f;
            big = big || !(static_top(f[0], f[1], f[2]) < BIG_SHARE);
            if (lane == 0) {
#pragma unroll
                for (int c = 0; c < 3; ++c) wfix[wib][r][c] = f2fix_wrap(f[c]);
            }
        }
        __syncthreads();
        if (tid < 7 * RA && r0 + tid / 7 < p.n_alch) {
            const int r = tid / 7, c = tid % 7;
            unsigned long long *o = part + 7ull * ((size_t)(r0 + r) * chunks + chunk) + c;
            if (c < 4) {
                double v = 0.0;
                for (int q = 0; q < ST_WARPS; ++q) v += wsum[q][r][c];
                *o = (unsigned long long)__double_as_longlong(v);
            } else {
                unsigned long long v = 0ull;
                for (int q = 0; q < ST_WARPS; ++q) v += wfix[q][r][c - 4];
                *o = v;
            }
        }
        // ---- the group's last block adds its chunks (lane = chunk) ----
        unsigned *chunks_done = status + 2;
        __threadfence();
        const unsigned add = __syncthreads_or(big) ? 0x10001u : 1u;
        if (tid == 0) {  // finished chunks, those with a big pair or share from bit 16 on
            const unsigned done = atomicAdd(&chunks_done[r0 / RA], add) + add;
            last = (done & 0xffffu) == (unsigned)chunks ? 1 + (int)(done >> 16) : 0;
        }
        __syncthreads();
        if (!last) return;
        __threadfence();
        unsigned bad = 0;  // atoms of the group out of range
        if (last > 1) {
#pragma unroll 1
            for (int r = 0; r < RA && r0 + r < p.n_alch; ++r)
                if (!alch_force_ok(p, in, tile[r], wforce, status)) bad |= 1u << r;
        }
        for (int r = r0 + wib; r < min(p.n_alch, r0 + RA); r += ST_WARPS) {
            const unsigned long long *o = part + 7ull * ((size_t)r * chunks + lane);
            unsigned long long v[7];
#pragma unroll
            for (int c = 0; c < 7; ++c) v[c] = lane < chunks ? __ldcg(o + c) : 0ull;
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const double t = warp_sum(__longlong_as_double((long long)v[c]));
                if (lane == 0) sums[4 * (size_t)r + c] = t;
            }
#pragma unroll
            for (int c = 4; c < 7; ++c) {
#pragma unroll
                for (int d = 16; d > 0; d >>= 1) v[c] += __shfl_xor_sync(0xffffffffu, v[c], d);
            }
            const int a = in.alch_idx[r];
            if (lane < 3 && (unsigned)a < (unsigned)p.n && in.alch[a])
                forces[3 * (size_t)a + lane] =
                    (bad >> (r - r0)) & 1u ? 0.f : fix_to_float(lane == 0 ? v[4] : (lane == 1 ? v[5] : v[6]));
        }
    }
    // ---- the last group adds the alchemical atoms ----
    __threadfence();
    __syncthreads();
    if (tid == 0) last = atomicAdd(status + 1, 1u) == (gridDim.x - n_env_blocks) / chunks - 1u;
    __syncthreads();
    if (!last) return;
    __threadfence();
    double s[4] = {0.0, 0.0, 0.0, 0.0};
    for (int r = tid; r < p.n_alch; r += ST_THREADS)
#pragma unroll
        for (int c = 0; c < 4; ++c) s[c] += __ldcg(sums + 4 * (size_t)r + c);
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        const double v = warp_sum(s[c]);
        if (lane == 0) wsum[wib][0][c] = v;
    }
    __syncthreads();
    if (tid == 0) {
        for (int c = 0; c < 4; ++c) {
            s[c] = 0.0;
            for (int q = 0; q < ST_WARPS; ++q) s[c] += wsum[q][0][c];
        }
        out[0] = dlv * s[0] + dle * s[1];
        out[1] = s[0];
        out[2] = s[1];
        out[3] = s[2];
        out[4] = s[3];
        // (the environment blocks meet the same pairs: they add no other bits)
        out[5] = (double)*(volatile unsigned *)status;
    }
}

int static_fail(int code, const char *msg) {
    g_static_err = msg;
    return code;
}

// once per device, with that device current: the array's device address
int static_scratch(void **ptr) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return static_fail(LA_ERR_CUDA, cudaGetErrorString(e));
    if (dev < 0 || dev >= MAX_DEVICES) return static_fail(LA_ERR_UNSUPPORTED, "device index out of range");
    std::lock_guard<std::mutex> lock(g_setup_mutex);
    if (!g_scratch_addr[dev]) {
        void *p = nullptr;
        e = cudaGetSymbolAddress(&p, g_static_scratch);
        if (e != cudaSuccess || !p) {
            char buf[256];
            snprintf(buf, sizeof buf, "cudaGetSymbolAddress of the static scratch failed: %s",
                     cudaGetErrorString(e));
            return static_fail(LA_ERR_CUDA, buf);
        }
        g_scratch_addr[dev] = p;
    }
    *ptr = g_scratch_addr[dev];
    return LA_OK;
}

}  // namespace
}  // namespace labf

using namespace labf;

extern "C" int la_alch_pairs_static(int n_atoms, const float *x, const float *q, const float *sigma,
                                    const float *epsilon, const uint8_t *alch, const int32_t *excl_group,
                                    int n_alch, const int32_t *alch_idx, double box, double r_cut,
                                    double eps_rf, double coul, double lam, double b_v, double b_e,
                                    double sc_alpha, int sc_n, int sc_m, float *forces, double *out,
                                    void *stream) {
    if (n_atoms <= 0 || n_alch < 0 || !x || !q || !sigma || !epsilon || !alch || !excl_group || !forces ||
        !out || (n_alch > 0 && !alch_idx))
        return static_fail(LA_ERR_INVALID_ARG, "NULL pointer or non-positive atom count");
    if (n_atoms > LA_STATIC_MAX_ATOMS || n_alch > LA_STATIC_MAX_ALCH) {
        char buf[160];
        snprintf(buf, sizeof buf, "size beyond the static scratch: n_atoms %d (max %d), n_alch %d (max %d)",
                 n_atoms, LA_STATIC_MAX_ATOMS, n_alch, LA_STATIC_MAX_ALCH);
        return static_fail(LA_ERR_INVALID_ARG, buf);
    }
    if (!(box > 0) || !(r_cut > 0) || 2.0 * r_cut > box || !(b_v > 0) || !(b_e < 1))
        return static_fail(LA_ERR_INVALID_ARG, "invalid box, cutoff or alchemical parameters");
    if (sc_n < 1 || sc_m < 1)  // n lambda_v^(n-1) and m (1-lambda_v)^(m-1) at the ends need n, m >= 1
        return static_fail(LA_ERR_INVALID_ARG, "soft-core powers sc_n and sc_m must be >= 1");
    void *base = nullptr;
    int rc = static_scratch(&base);
    if (rc != LA_OK) return rc;
    unsigned long long *part = (unsigned long long *)base;
    double *sums = (double *)(part + LA_STATIC_PART_WORDS);
    unsigned *status = (unsigned *)(sums + LA_STATIC_SUM_WORDS);  // then the counters

    double lv, le, dlv, dle;
    if (lam < b_v) { lv = lam / b_v; dlv = 1.0 / b_v; } else { lv = 1.0; dlv = 0.0; }
    if (lam > b_e) { le = (lam - b_e) / (1.0 - b_e); dle = 1.0 / (1.0 - b_e); } else { le = 0.0; dle = 0.0; }
    StaticParams p;
    p.n = n_atoms;
    p.n_alch = n_alch;
    p.L = (float)box;
    p.Linv = (float)(1.0 / box);
    p.rc2 = (float)(r_cut * r_cut);
    const double krf = eps_rf <= 0.0 ? 1.0 / (2.0 * r_cut * r_cut * r_cut)
                                     : (eps_rf - 1.0) / ((2.0 * eps_rf + 1.0) * r_cut * r_cut * r_cut);
    p.krf = (float)krf;
    p.crf = (float)(1.0 / r_cut + krf * r_cut * r_cut);
    p.sqrt_coul = (float)std::sqrt(coul > 0.0 ? coul : 0.0);
    p.le = (float)le;
    p.lvn = (float)std::pow(lv, (double)sc_n);
    p.dlvn = (float)((double)sc_n * std::pow(lv, (double)(sc_n - 1)));
    p.sa = (float)(sc_alpha * std::pow(1.0 - lv, (double)sc_m));
    p.dsdl = (float)(-(double)sc_m * sc_alpha * std::pow(1.0 - lv, (double)(sc_m - 1)));

    cudaStream_t s = (cudaStream_t)stream;
    const StaticIn in{x, q, sigma, epsilon, alch, excl_group, alch_idx};
    // chunks of at least a block's width; four alchemical atoms per block once
    // single ones would make more blocks than the chip runs in one wave
    const int env = (n_atoms + ST_THREADS - 1) / ST_THREADS;
    const int chunks = env < LA_STATIC_CHUNKS ? env : LA_STATIC_CHUNKS;
    const bool single = n_alch * chunks <= 1024;
    const int groups = n_alch == 0 ? 1 : (single ? n_alch : (n_alch + 3) / 4);
    cudaError_t em = cudaMemsetAsync(status, 0, (2 + groups) * sizeof(unsigned), s);
    if (em != cudaSuccess) return static_fail(LA_ERR_CUDA, cudaGetErrorString(em));
    if (single)
        k_static<1><<<env + groups * chunks, ST_THREADS, 0, s>>>(p, in, env, chunks, part, sums, status, dlv, dle,
                                                                forces, out);
    else
        k_static<4><<<env + groups * chunks, ST_THREADS, 0, s>>>(p, in, env, chunks, part, sums, status, dlv, dle,
                                                                forces, out);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return static_fail(LA_ERR_CUDA, cudaGetErrorString(e));
    return LA_OK;
}

extern "C" const char *la_static_last_error(void) { return g_static_err.c_str(); }
