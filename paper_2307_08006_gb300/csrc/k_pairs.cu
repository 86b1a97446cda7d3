// k_pairs.cu -- the pair pass: LJ + reaction-field forces of normal pairs
// over the cluster-pair list, and, in the same launch, the alchemically
// scaled pairs with the walker's dU/dlambda partials (Sec. 3.1.2, Eq.
// lambda-abf: the engine provides dV/dlambda every step).
//
// Normal pairs: warps take work items (a chunk of one super-cluster's
// j-list) from a global counter.  The super-cluster's 64 slots sit in shared
// memory.  Entries are prepared 32 at a time into shared memory (headers one
// per lane, then eight entries' j-atoms per round with the periodic shift
// applied, lane mask bytes as one contiguous copy); then for each entry lane
// (ia, jb) = (lane >> 2, lane & 3) evaluates the pair (i-atom ia of every
// flagged i-cluster, j-atom jb).  Four neighbouring lanes share an i-atom, so
// the i-cluster's 128-bit shared loads take half the passes they took with
// ia = lane & 7; neighbouring lanes also gather one j-cluster's atoms
// together, and write them without bank conflicts, where each lane fetched a
// whole entry (a gather of 32 rows per load).  The shared-memory pipe was 62%
// busy before, second only to the issue slots (73%).  One j-cluster load and
// one j-force reduction serve up to 8 x 32 pairs, and the eight i-force
// accumulators stay in registers for the whole item.  Forces are summed in
// FP32 and added to the 64-bit fixed-point force array with integer atomics
// (order-free, so results are bit-reproducible).  The i-forces are flushed
// to the fixed-point array after every 32 entries of a super-cluster's list,
// so every kernel variant and work-item size (a multiple of 32 entries)
// produces the same bits.  A lane whose pair is out of the cutoff skips its
// six accumulating instructions by predicate (no select to zero per tile).  An
// evaluation multiplies by zero instead: a distance that is not a number then
// reaches the forces and is reported (an MD step's integrator tests the
// positions themselves).
// All float-to-fixed conversions use integer instructions: the hardware
// conversion to 64-bit integers runs on the FP64 pipe, which is narrow on this
// GPU.  Fused launch before / after the lane map, the staging and the
// predicated sums: 16 x 12 300 atoms 255 / 242 us, 144 x 772 atoms 127 / 117
// us, 2 x 9020 atoms 47 / 43 us, 16 x 96 040 atoms 2600 / 2485 us.
//
// Per in-cutoff pair (force only), 37 FP32 flops (FMA = 2) plus one rsqrt:
//   d = x_i - x_j (3), r2 (5), 1/r2 (1), sigma_ij = s_i + s_j, (sigma/r)^2,
//   (sigma/r)^6 (5), 4 eps_ij (sigma/r)^6 (2), t = 12 (sigma/r)^6 - 6 (2),
//   b = q_i q_j / r + 4eps (sigma/r)^6 t (4), f = b / r2 - 2 k_rf q_i q_j (3),
//   f_i += f d, f_j -= f d (12).
//
// Alchemical pairs: one warp per (walker, alchemical atom); lanes stride over
// its environment list.  Soft-core LJ lambda_v^n 4 eps (s^-2 - s^-1) with
// s = alpha (1 - lambda_v)^m + (r/sigma)^6, RF scaled by lambda_e; per-lane
// FP64 sums of dU/dlambda_v, dU/dlambda_e, energies and theta derivatives,
// reduced with a fixed shuffle tree (deterministic).
#include "labf_dyn.cuh"
#include "labf_internal.cuh"
#include "labf_launch.h"

#include <type_traits>

namespace labf {

constexpr int EPC = 32;  // entries prepared per pass (one per lane)

// x^n for an integer n >= 0 (square and multiply; exact for n <= 1)
__device__ __forceinline__ double ipow(double x, int n) {
    double r = 1.0;
    for (; n > 0; n >>= 1) {
        if (n & 1) r *= x;
        x *= x;
    }
    return r;
}
constexpr unsigned FULL = 0xffffffffu;

template <int WARPS>
struct PairShared {
    float4 sxq[WARPS][SC];      // the item's super-cluster
    float2 slj[WARPS][SC];
    float4 jx[WARPS][EPC][JC];  // prepared j-atoms (shift applied)
    float2 jl[WARPS][EPC][JC];
    unsigned char lb[WARPS][EPC][32];
    int pre[LA_MAX_WALKERS_PER_LAUNCH + 1], first, parts;
};

// Shared memory of the latency form: the super-cluster's i-clusters two by
// two (row (p, ia): atom ia of i-clusters 2p and 2p + 1 as {x x' y y'},
// {z z' q q'}, {s s' e e'}), the prepared j-atoms with every value twice
// (position negated), so that packed operands are loaded as they are, and the
// pairs' forces over distance.
struct PairSharedLat {
    float4 si[3][SC / 2];
    float4 j[EPC][3 * JC];
    unsigned char lb[EPC][32];
    float2 f[EPC][NIC / 2][32];
    unsigned char keep[EPC][NIC / 2];
    int pre[LA_MAX_WALKERS_PER_LAUNCH + 1], first, next, parts;
};
constexpr int LAT_WARPS = NIC / 2;

// counters[4] hands out work items; counters[5] counts warps that found no
// more work; the last one resets both for the next launch
constexpr int CTR_ITEM = 4, CTR_DONE = 5;

// i-forces of one flush, summed over the 4 j-lanes of each i-atom with a
// transposed tree: at the first level (partner jb ^ 1) a lane keeps the
// i-clusters {0, 1, 4, 5} (jb even) or {2, 3, 6, 7} (jb odd) and sends the
// others; at the second (partner jb ^ 2) it keeps the lower or upper pair, so
// lane (ia, jb) ends with i-clusters 2jb and 2jb + 1.  Every i-atom's sum is
// (a0 + a1) + (a2 + a3) over the j-lanes.  The accumulators restart from zero.
__device__ __forceinline__ void flush_i(const Dev &d, int gS, int ia, int jb, unsigned touched,
                                        float (&fi)[NIC][3]) {
    const bool odd = (jb & 1) != 0, upper = (jb & 2) != 0;
    float k1[4][3];
#pragma unroll
    for (int t = 0; t < 4; ++t) {
        const int ke = t < 2 ? t : t + 2;  // 0, 1, 4, 5
        const int ko = ke + 2;             // 2, 3, 6, 7
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const float keep = odd ? fi[ko][c] : fi[ke][c];
            const float send = odd ? fi[ke][c] : fi[ko][c];
            k1[t][c] = keep + __shfl_xor_sync(FULL, send, 1);
        }
    }
#pragma unroll
    for (int t = 0; t < 2; ++t) {
        const int ic = 2 * jb + t;
        unsigned long long *p = d.F + 3 * (size_t)(gS + ic * IC + ia);
        const bool on = (touched >> ic) & 1u;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const float keep = upper ? k1[t + 2][c] : k1[t][c];
            const float send = upper ? k1[t][c] : k1[t + 2][c];
            const float v = keep + __shfl_xor_sync(FULL, send, 2);
            if (on) atomicAdd(p + c, f2fix(v));
        }
    }
#pragma unroll
    for (int ic = 0; ic < NIC; ++ic) fi[ic][0] = fi[ic][1] = fi[ic][2] = 0.f;
}

// j-forces of two entries A and B at once (B absent: pass zeros and
// has_b = false).  Lane (ia, jb) holds j-atom jb's partial sums over its
// i-atoms (a for A, b for B; positive accumulation, the atom receives minus
// the sum).  Transposed tree over the 8 i-lanes: partner ia ^ 4 (lanes
// ia < 4 keep A, the others B), ia ^ 2 (keep x, y or z, 0), ia ^ 1; lane ia
// ends with A's component ia (ia < 3) or B's component ia - 4 (4 <= ia < 7).
// Each sum is ((a0 + a4) + (a2 + a6)) + ((a1 + a5) + (a3 + a7)), whether or
// not B is present.
__device__ __forceinline__ void flush_j2(const Dev &d, int gjA, int gjB, bool has_b, int ia, const float (&a)[3],
                                         const float (&b)[3]) {
    const bool h4 = (ia & 4) != 0, h2 = (ia & 2) != 0, h1 = (ia & 1) != 0;
    float v[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const float keep = h4 ? b[c] : a[c];
        const float send = h4 ? a[c] : b[c];
        v[c] = keep + __shfl_xor_sync(FULL, send, 16);
    }
    // (x, y) kept by h2 = 0, (z, 0) by h2 = 1
    const float k0 = h2 ? v[2] : v[0], k1 = h2 ? 0.f : v[1];
    const float s0 = h2 ? v[0] : v[2], s1 = h2 ? v[1] : 0.f;
    const float w0 = k0 + __shfl_xor_sync(FULL, s0, 8);
    const float w1 = k1 + __shfl_xor_sync(FULL, s1, 8);
    const float kk = h1 ? w1 : w0, ss = h1 ? w0 : w1;
    const float c = kk + __shfl_xor_sync(FULL, ss, 4);
    const int comp = ia & 3;
    if (comp < 3 && (!h4 || has_b)) atomicAdd(d.F + 3 * (size_t)(h4 ? gjB : gjA) + comp, f2fix(-c));
}

// One work item's entries, prepared and evaluated 32 at a time; the
// i-forces are flushed after every 32 entries.  MSHIFT: 8 reads the i-cluster
// mask pruned for the batched step, 16 the listed one (one-task launches,
// which run without pruning).  PRUNE (batched step, walker due for
// re-pruning): the listed mask is evaluated and each entry's pruned mask is
// rewritten with the i-clusters holding a listed pair within r_c + margin (a
// vote per tile, which also skips the force arithmetic of the others), which
// later steps read; every tile that is skipped adds exact zeros, so results do
// not depend on the pruning.  Without the skip a re-pruning launch took 287 us
// against 229 us for a common one (16 x 12 300 atoms, ncu), with it 279 us; the
// passes of hot starts, where two launches in five re-prune, are 1.2-1.8%
// shorter.
template <bool ENERGY, int WARPS, int MSHIFT, bool PRUNE>
__device__ __forceinline__ int item_entries(const Dev &d, PairShared<WARPS> &sh, const SysDev &S, int4 it, int gS,
                                            float &elj, float &erf, int &npair) {
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const int ia = lane >> 2, jb = lane & 3, lbi = jb * IC + ia;
    const float L = S.boxf, rc2 = S.rc2, krf2 = 2.0f * S.krf, krf = S.krf, crf = S.crf;
    const float rp2 = S.rprune2;
    float fi[NIC][3];
#pragma unroll
    for (int ic = 0; ic < NIC; ++ic) fi[ic][0] = fi[ic][1] = fi[ic][2] = 0.f;
    unsigned touched = 0;
    int v_next = 0;
    const size_t ebase = (size_t)it.x * d.ent_cap;
    for (int eb = it.y; eb < it.z; eb += EPC) {
        const int ne = min(EPC, it.z - eb);
        // prepare up to 32 entries, one per lane
        int gj_l = 0, hy_l = 0;
        unsigned im_l = 0, keep_l = 0;
        __syncwarp();
        if (lane < ne) {
            const int2 hdr = d.ent_hdr[ebase + eb + lane];
            gj_l = hdr.x;
            hy_l = hdr.y;
            im_l = ((unsigned)hdr.y >> (PRUNE ? 16 : MSHIFT)) & 0xffu;
            if (!la_in(d, gj_l, d.n_slots - JC + 1)) gj_l = 0, im_l = 0;  // entry skipped
        }
        // lane masks: the entries' bytes are contiguous
        {
            const uint4 *src = reinterpret_cast<const uint4 *>(d.ent_lb + 32 * (ebase + eb));
            uint4 *dst = reinterpret_cast<uint4 *>(&sh.lb[wib][0][0]);
#pragma unroll
            for (int h = 0; h < 2; ++h)
                if (lane + 32 * h < 2 * ne) dst[lane + 32 * h] = src[lane + 32 * h];
        }
        // j-atoms, eight entries per round
#pragma unroll
        for (int r = 0; r < EPC / IC; ++r) {
            const int e = r * IC + (lane >> 2), q = lane & 3;
            const int g = __shfl_sync(FULL, im_l ? gj_l : -1, e);
            const int hy = __shfl_sync(FULL, hy_l, e);
            if (g < 0) continue;  // pruned or absent
            const float sx = (float)((hy & 3) - 1) * L;
            const float sy = (float)(((hy >> 2) & 3) - 1) * L;
            const float sz = (float)(((hy >> 4) & 3) - 1) * L;
            float4 x = d.xq[g + q];
            x.x += sx;
            x.y += sy;
            x.z += sz;
            sh.jx[wib][e][q] = x;
            sh.jl[wib][e][q] = d.lj[g + q];
        }
        // entries whose tiles were all pruned add nothing: skip them
        unsigned emask = __ballot_sync(FULL, im_l != 0u);
        __syncwarp();
        // one entry: every flagged i-cluster against the entry's j-cluster;
        // fjs receives j-atom jb's partial force over this lane's i-atoms.
        // The re-pruning form evaluates every listed tile: the atom whose
        // displacement triggered it may already have moved past the margin
        // the previous pruning allowed for.
        auto entry = [&](int k, float (&fjs)[3]) {
            const unsigned imask = __shfl_sync(FULL, im_l, k);
            const float4 xj = sh.jx[wib][k][jb];
            const float2 lj_j = sh.jl[wib][k][jb];
            const unsigned lb = sh.lb[wib][k][lbi];
            touched |= imask;
            float fj[3] = {0.f, 0.f, 0.f};
            unsigned keep = 0;  // i-clusters with a listed pair within r_c + margin
#pragma unroll
            for (int ic = 0; ic < NIC; ++ic) {
                if (imask & (1u << ic)) {
                    const float4 xi = sh.sxq[wib][ic * IC + ia];
                    const float2 li = sh.slj[wib][ic * IC + ia];
                    const float dx = xi.x - xj.x, dy = xi.y - xj.y, dz = xi.z - xj.z;
                    const float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
                    if (PRUNE) {
                        if (!__any_sync(FULL, (lb & (1u << ic)) && r2 < rp2)) continue;  // adds zeros
                        keep |= 1u << ic;
                    }
                    const bool in = (lb & (1u << ic)) && (r2 < rc2);
                    const float rinv = rsqrtf(r2);
                    const float r2inv = rinv * rinv;
                    const float sg = li.x + lj_j.x;
                    const float sr2 = sg * sg * r2inv;
                    const float sr6 = sr2 * sr2 * sr2;
                    const float e4s6 = li.y * lj_j.y * sr6;
                    const float qq = xi.w * xj.w;
                    const float b = fmaf(qq, rinv, e4s6 * fmaf(12.f, sr6, -6.f));
                    float fs = fmaf(b, r2inv, -qq * krf2);
                    if (ENERGY) fs = in ? fs : 0.f;
                    if (ENERGY || in) {  // predicated
                        fi[ic][0] = fmaf(fs, dx, fi[ic][0]);
                        fi[ic][1] = fmaf(fs, dy, fi[ic][1]);
                        fi[ic][2] = fmaf(fs, dz, fi[ic][2]);
                        fj[0] = fmaf(fs, dx, fj[0]);
                        fj[1] = fmaf(fs, dy, fj[1]);
                        fj[2] = fmaf(fs, dz, fj[2]);
                    }
                    if (ENERGY) {
                        if (in) {
                            elj += e4s6 * (sr6 - 1.f);
                            erf += qq * (rinv + krf * r2 - crf);
                            ++npair;
                        }
                    }
                }
            }
            if (PRUNE) keep_l = lane == k ? keep : keep_l;
            fjs[0] = fj[0];
            fjs[1] = fj[1];
            fjs[2] = fj[2];
        };
        // two entries per iteration (also in the re-pruning form): the
        // compiler interleaves their independent loads and arithmetic (the
        // order of every sum stays), and one transposed reduction serves both
        // j-clusters
        while (emask) {
            const int k0 = __ffs(emask) - 1;
            emask &= emask - 1u;
            float a[3], b[3] = {0.f, 0.f, 0.f};
            const int gA = __shfl_sync(FULL, gj_l, k0) + jb;
            int gB = 0;
            const bool two = emask != 0u;
            if (two) {
                const int k1 = __ffs(emask) - 1;
                emask &= emask - 1u;
                gB = __shfl_sync(FULL, gj_l, k1) + jb;
                entry(k0, a);
                entry(k1, b);
            } else {
                entry(k0, a);
            }
            flush_j2(d, gA, gB, two, ia, a, b);
        }
        // the next item's index, fetched just before the last flush: its round
        // trip is hidden, and no warp holds an item it cannot start yet
        if (eb + EPC >= it.z && lane == 0) v_next = (int)atomicAdd(&d.counters[CTR_ITEM], 1ull);
        flush_i(d, gS, ia, jb, touched, fi);  // every 32 entries (EPC)
        touched = 0;
        if (PRUNE && lane < ne) d.ent_hdr[ebase + eb + lane].y = (hy_l & ~0xff00) | (int)(keep_l << 8);
    }
    return v_next;
}

// the re-pruning form, out of line: the common form's code stays as it is
template <int WARPS>
__device__ __noinline__ int item_entries_prune(const Dev &d, PairShared<WARPS> &sh, const SysDev &S, int4 it, int gS) {
    float elj = 0.f, erf = 0.f;
    int npair = 0;
    return item_entries<false, WARPS, 8, true>(d, sh, S, it, gS, elj, erf, npair);
}

// The same item for launches with few items (at most LAT_ITEMS_PER_SM per SM:
// one or two boxes, small batches), where an item's own latency decides, not
// the issue rate: a block of four warps takes it.
//   1  warp p evaluates i-clusters 2p and 2p + 1 against all entries, both in
//      one packed FP32 instruction and without branches, sums their i-forces
//      and leaves every pair's force over distance in shared memory
//   2  the entries are dealt out to the warps again, which add the j-forces
//      over all i-clusters from those factors
// Every sum keeps the order of the common form (i-forces: one entry after the
// other; j-forces: i-clusters ascending; skipped pairs add exact zeros), so
// the forces are the same bits.  One warp per item took 13 us for its 32
// entries one after the other.
template <int MSHIFT, bool PRUNE>
__device__ __forceinline__ void item_entries_lat(const Dev &d, PairSharedLat &sh, const SysDev &S, int4 it, int gS) {
    const int tid = threadIdx.x, lane = tid & 31, p = tid >> 5;
    const int ia = lane >> 2, jb = lane & 3, lbi = jb * IC + ia;
    const float L = S.boxf, rc2 = S.rc2, rp2 = S.rprune2, krf2 = 2.0f * S.krf;
    const unsigned b0 = 1u << (2 * p), b1 = 2u << (2 * p);
    const size_t ebase = (size_t)it.x * d.ent_cap;
    if (tid < SC) {  // slot tid: atom tid & 7 of i-cluster tid >> 3
        const float4 x = d.xq[gS + tid];
        const float2 l = d.lj[gS + tid];
        float *row = reinterpret_cast<float *>(&sh.si[0][(tid >> 4) * IC + (tid & 7)]) + ((tid >> 3) & 1);
        row[0] = x.x;
        row[2] = x.y;
        row[2 * SC] = x.z;
        row[2 * SC + 2] = x.w;
        row[4 * SC] = l.x;
        row[4 * SC + 2] = l.y;
    }
    for (int eb = it.y; eb < it.z; eb += EPC) {
        const int ne = min(EPC, it.z - eb);
        // headers, by every warp; each prepares eight entries' j-atoms
        int gj_l = 0, hy_l = 0;
        unsigned im_l = 0;
        if (lane < ne) {
            const int2 hdr = d.ent_hdr[ebase + eb + lane];
            gj_l = hdr.x;
            hy_l = hdr.y;
            im_l = ((unsigned)hdr.y >> (PRUNE ? 16 : MSHIFT)) & 0xffu;
            if (!la_in(d, gj_l, d.n_slots - JC + 1)) gj_l = 0, im_l = 0;  // entry skipped
        }
        if (tid < 2 * ne)  // lane masks: the entries' bytes are contiguous
            reinterpret_cast<uint4 *>(&sh.lb[0][0])[tid] = reinterpret_cast<const uint4 *>(d.ent_lb + 32 * (ebase + eb))[tid];
        {
            const int e = p * IC + (lane >> 2), q = lane & 3;
            const int g = __shfl_sync(FULL, im_l ? gj_l : -1, e);
            const int hy = __shfl_sync(FULL, hy_l, e);
            if (g >= 0) {
                const float4 x = d.xq[g + q];
                const float2 l = d.lj[g + q];
                const float nx = -(x.x + (float)((hy & 3) - 1) * L), ny = -(x.y + (float)(((hy >> 2) & 3) - 1) * L),
                            nz = -(x.z + (float)(((hy >> 4) & 3) - 1) * L);
                float4 *row = &sh.j[e][3 * q];
                row[0] = make_float4(nx, nx, ny, ny);
                row[1] = make_float4(nz, nz, x.w, x.w);
                row[2] = make_float4(l.x, l.x, l.y, l.y);
            }
        }
        if (PRUNE) sh.keep[lane][p] = 0;
        __syncthreads();
        // 1: this warp's two i-clusters against the entries that flag one
        f2 fi[3] = {0ull, 0ull, 0ull};
        {
            const ulonglong2 *si = reinterpret_cast<const ulonglong2 *>(&sh.si[0][p * IC + ia]);
            const ulonglong2 i0 = si[0], i1 = si[SC / 2], i2 = si[SC];
            const f2 nkrf2 = pack2(-krf2, -krf2), c12 = pack2(12.f, 12.f), c6 = pack2(-6.f, -6.f);
            auto tile = [&](int k, unsigned lb, f2 &fs, f2 &dx, f2 &dy, f2 &dz) -> unsigned {
                const ulonglong2 *rj = reinterpret_cast<const ulonglong2 *>(&sh.j[k][3 * jb]);
                const ulonglong2 j0 = rj[0], j1 = rj[1], j2 = rj[2];
                dx = add2(i0.x, j0.x);
                dy = add2(i0.y, j0.y);
                dz = add2(i1.x, j1.x);
                float r20, r21, f0, f1;
                unpack2(fma2(dx, dx, fma2(dy, dy, mul2(dz, dz))), r20, r21);
                const bool in0 = (lb & b0) && r20 < rc2, in1 = (lb & b1) && r21 < rc2;
                const f2 rinv = pack2(rsqrtf(r20), rsqrtf(r21));
                const f2 r2inv = mul2(rinv, rinv);
                const f2 sg = add2(i2.x, j2.x);
                const f2 sr2 = mul2(mul2(sg, sg), r2inv);
                const f2 sr6 = mul2(mul2(sr2, sr2), sr2);
                const f2 e4s6 = mul2(mul2(i2.y, j2.y), sr6);
                const f2 qq = mul2(i1.y, j1.y);
                const f2 b = fma2(qq, rinv, mul2(e4s6, fma2(c12, sr6, c6)));
                unpack2(fma2(b, r2inv, mul2(qq, nkrf2)), f0, f1);
                fs = pack2(in0 ? f0 : 0.f, in1 ? f1 : 0.f);
                unsigned kb = 0;  // pairs within r_c + margin
                if (PRUNE) kb = ((lb & b0) && r20 < rp2 ? 1u : 0u) | ((lb & b1) && r21 < rp2 ? 2u : 0u);
                return kb;
            };
            unsigned m = __ballot_sync(FULL, (im_l & (b0 | b1)) != 0u);
            while (m) {  // two entries per round
                const int k0 = __ffs(m) - 1;
                m &= m - 1u;
                const bool two = m != 0u;
                const int k1 = two ? __ffs(m) - 1 : k0;
                m &= m - 1u;
                f2 fa, fb, ax, ay, az, bx, by, bz;
                const unsigned ka = tile(k0, sh.lb[k0][lbi], fa, ax, ay, az);
                const unsigned kb = tile(k1, two ? sh.lb[k1][lbi] : 0u, fb, bx, by, bz);
                fi[0] = fma2(fb, bx, fma2(fa, ax, fi[0]));
                fi[1] = fma2(fb, by, fma2(fa, ay, fi[1]));
                fi[2] = fma2(fb, bz, fma2(fa, az, fi[2]));
                reinterpret_cast<f2 *>(sh.f[k0][p])[lane] = fa;
                if (two) reinterpret_cast<f2 *>(sh.f[k1][p])[lane] = fb;
                if (PRUNE) {
                    const unsigned keep = __reduce_or_sync(FULL, ka | (kb << 2));
                    if (lane == 0) {
                        sh.keep[k0][p] = keep & 3u;
                        if (two) sh.keep[k1][p] = keep >> 2;
                    }
                }
            }
        }
        __syncthreads();
        // 2: the j-forces of every fourth entry with pairs
        const unsigned emask = __ballot_sync(FULL, im_l != 0u);
        unsigned m = __ballot_sync(FULL, im_l != 0u && (__popc(emask & ((1u << lane) - 1u)) & 3) == p);
        if (m) {
            f2 ix[NIC / 2], iy[NIC / 2], iz[NIC / 2];
#pragma unroll
            for (int q = 0; q < NIC / 2; ++q) {
                const ulonglong2 i0 = *reinterpret_cast<const ulonglong2 *>(&sh.si[0][q * IC + ia]);
                ix[q] = i0.x;
                iy[q] = i0.y;
                iz[q] = *reinterpret_cast<const f2 *>(&sh.si[1][q * IC + ia]);
            }
            auto sum_j = [&](int k, float (&fj)[3]) {
                const unsigned imask = __shfl_sync(FULL, im_l, k);
                const ulonglong2 j0 = *reinterpret_cast<const ulonglong2 *>(&sh.j[k][3 * jb]);
                const f2 jz = *reinterpret_cast<const f2 *>(&sh.j[k][3 * jb + 1]);
                fj[0] = fj[1] = fj[2] = 0.f;
#pragma unroll
                for (int q = 0; q < NIC / 2; ++q) {
                    // (factors of pairs of i-clusters that no warp evaluated are not read)
                    const bool on = (imask >> (2 * q)) & 3u;
                    const float2 f = on ? sh.f[k][q][lane] : make_float2(0.f, 0.f);
                    float d0, d1;
                    unpack2(add2(ix[q], j0.x), d0, d1);
                    fj[0] = fmaf(f.y, d1, fmaf(f.x, d0, fj[0]));
                    unpack2(add2(iy[q], j0.y), d0, d1);
                    fj[1] = fmaf(f.y, d1, fmaf(f.x, d0, fj[1]));
                    unpack2(add2(iz[q], jz), d0, d1);
                    fj[2] = fmaf(f.y, d1, fmaf(f.x, d0, fj[2]));
                }
            };
            while (m) {
                const int k0 = __ffs(m) - 1;
                m &= m - 1u;
                const bool two = m != 0u;
                const int k1 = two ? __ffs(m) - 1 : k0;
                m &= m - 1u;
                float a[3], b[3];
                sum_j(k0, a);
                sum_j(k1, b);
                const int gA = __shfl_sync(FULL, gj_l, k0) + jb, gB = __shfl_sync(FULL, gj_l, k1) + jb;
                flush_j2(d, gA, gB, two, ia, a, b);
            }
        }
        // the i-forces: (a0 + a1) + (a2 + a3) over the j-lanes, as flush_i; lane
        // jb ends with i-cluster 2p + (jb & 1)
        {
            const bool odd = (jb & 1) != 0;
            const bool on = (__reduce_or_sync(FULL, im_l) >> (2 * p + (jb & 1))) & 1u;
            unsigned long long *F = d.F + 3 * (size_t)(gS + (2 * p + (jb & 1)) * IC + ia);
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                float e, o;
                unpack2(fi[c], e, o);
                float v = (odd ? o : e) + __shfl_xor_sync(FULL, odd ? e : o, 1);
                v += __shfl_xor_sync(FULL, v, 2);
                if (on && (jb >> 1) == (c == 2)) atomicAdd(F + c, f2fix(v));
            }
        }
        if (PRUNE && p == 0 && lane < ne) {
            unsigned keep = 0;
#pragma unroll
            for (int q = 0; q < NIC / 2; ++q) keep |= (unsigned)sh.keep[lane][q] << (2 * q);
            d.ent_hdr[ebase + eb + lane].y = (hy_l & ~0xff00) | (int)(keep << 8);
        }
        if (eb + EPC < it.z) __syncthreads();  // shared memory free
    }
}

template <bool ENERGY, int WARPS, int MSHIFT>
__device__ __forceinline__ int run_item(const Dev &d, PairShared<WARPS> &sh, const SysDev &S, int w, int4 it, int gS,
                                        float &elj, float &erf, int &npair) {
    if (MSHIFT == 8 && d.prune_now[w] != 0ull) return item_entries_prune<WARPS>(d, sh, S, it, gS);
    return item_entries<ENERGY, WARPS, MSHIFT, false>(d, sh, S, it, gS, elj, erf, npair);
}
// work item v of a launch: its walker, entries and first slot; false when it
// is out of range
__device__ __forceinline__ bool find_item(const Dev &d, const int *pre, int w0, int nw, int v, int &w, int4 &it, int &gS) {
    int lo = 0, hi = nw - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (pre[mid] <= v) lo = mid; else hi = mid - 1;
    }
    w = w0 + lo;
    const WalkerDev &W = d.walk[w];
    it = d.items[W.item_base + (v - pre[lo])];
    gS = W.slot_off + (it.x - W.sc_off) * SC;
    return la_in(d, it.x - W.sc_off, W.sc_cap) && la_in(d, it.z - 1, d.ent_cap) && la_in(d, it.y, it.z);
}

// the last one out of `parts` resets the work counters for the next launch
__device__ __forceinline__ void items_done(const Dev &d, bool arrives, unsigned long long parts) {
    if (!arrives) return;
    __threadfence();
    if (atomicAdd(&d.counters[CTR_DONE], 1ull) == parts - 1ull) {
        d.counters[CTR_ITEM] = 0ull;
        d.counters[CTR_DONE] = 0ull;
        __threadfence();
    }
}

// work items of the normal pairs, handed out by a global counter
template <bool ENERGY, int WARPS, int MSHIFT>
__device__ __forceinline__ void normal_items(const Dev &d, int w0, int w1, PairShared<WARPS> &sh) {
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const int nw = w1 - w0;
    const int total = sh.pre[nw];
    int v_next = sh.first + wib;  // the block's first items came with one atomic
    for (;;) {
        const int v = __shfl_sync(FULL, v_next, 0);
        if (v >= total) break;
        int w, gS;
        int4 it;
        if (!find_item(d, sh.pre, w0, nw, v, w, it, gS)) {  // item skipped
            if (lane == 0) v_next = (int)atomicAdd(&d.counters[CTR_ITEM], 1ull);
            continue;
        }
        const SysDev &S = d.sys[d.walk[w].sys];
        __syncwarp();
        sh.sxq[wib][lane] = d.xq[gS + lane];
        sh.sxq[wib][lane + 32] = d.xq[gS + lane + 32];
        sh.slj[wib][lane] = d.lj[gS + lane];
        sh.slj[wib][lane + 32] = d.lj[gS + lane + 32];
        float elj = 0.f, erf = 0.f;
        int npair = 0;
        v_next = run_item<ENERGY, WARPS, MSHIFT>(d, sh, S, w, it, gS, elj, erf, npair);
        if (ENERGY) {
            const double el = warp_sum((double)elj), er = warp_sum((double)erf);
            int np = npair;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) np += __shfl_xor_sync(FULL, np, o);
            if (lane == 0) {
                atomicAdd((unsigned long long *)&d.eterm[N_ETERMS * w + 0],
                          (unsigned long long)__double2ll_rn(el * E_TO_FIX));
                atomicAdd((unsigned long long *)&d.eterm[N_ETERMS * w + 1],
                          (unsigned long long)__double2ll_rn(er * E_TO_FIX));
                atomicAdd(&d.counters[1], (unsigned long long)np);
            }
        }
    }
    items_done(d, lane == 0 && sh.parts > 0, (unsigned long long)sh.parts * WARPS);
}

// the same with one item per block at a time (latency form)
template <int MSHIFT>
__device__ __forceinline__ void normal_items_lat(const Dev &d, int w0, int w1, PairSharedLat &sh) {
    const int nw = w1 - w0;
    const int total = sh.pre[nw];
    for (int v = sh.first; v < total;) {
        int w, gS;
        int4 it;
        if (find_item(d, sh.pre, w0, nw, v, w, it, gS)) {
            const SysDev &S = d.sys[d.walk[w].sys];
            if (MSHIFT == 8 && d.prune_now[w] != 0ull) item_entries_lat<MSHIFT, true>(d, sh, S, it, gS);
            else item_entries_lat<MSHIFT, false>(d, sh, S, it, gS);
        }
        if (threadIdx.x == 0) sh.next = (int)atomicAdd(&d.counters[CTR_ITEM], 1ull);
        __syncthreads();
        v = sh.next;
        __syncthreads();
    }
    items_done(d, threadIdx.x == 0 && sh.parts > 0, (unsigned long long)sh.parts);
}

// Fused launch: a stage's lambda update (lambda_work) needs the partial sums
// of all its walkers' alchemical items and their restraint terms.  Each
// finished item, plus one restraint item per walker, arrives on the stage's
// counter; the warp that arrives last does the stage's work (a writer's lane
// fences before it arrives; the counter is reset by the last arrival).  No
// warp waits for another.  One hand-off instead of two (walker, then stage)
// and the restraints beside the alchemical items shorten the chain that ends
// a launch of a small system.
__device__ __forceinline__ void arrive_stage(const Dev &d, int w, int lane) {
    const int si = d.walk[w].stage;
    const StageDev &st = d.stage[si];
    const unsigned last = (unsigned)((st.w1 - st.w0) * (d.sys[st.sys].n_alch + 1)) - 1u;
    __syncwarp();
    unsigned old = 0;
    if (lane == 0) {
        __threadfence();
        old = atomicAdd(&d.sdone[si], 1u);
    }
    old = __shfl_sync(FULL, old, 0);
    if (old != last) return;
    if (lane == 0) d.sdone[si] = 0u;
    __threadfence();
    lambda_work<true>(d, si, 0, lane);
}

// walker in [w0, w1) that owns alchemical item it: the last one whose first
// item is not beyond it (32 walkers per load)
__device__ __forceinline__ int walker_of_alch(const Dev &d, int w0, int w1, int it, int lane) {
    int n = 0;
    for (int b = w0; b < w1; b += 32)
        n += __popc(__ballot_sync(FULL, b + lane < w1 && d.walk[min(b + lane, w1 - 1)].alch_base <= it));
    return w0 + n - 1;
}

// What a pair launch does besides the pairs.  STEP (the batched step): bonded
// terms, restraints, and the lambda update by the last arrival; lists pruned.
// EVAL (one energy evaluation): bonded terms and restraints.  PAIRS: nothing.
enum { PAIRS = 0, STEP = 1, EVAL = 2 };

// Alchemical items [a0, a1), one warp each, then (but for PAIRS) one restraint item
// per walker; unit `unit` of `units` takes every units-th item.
template <bool ENERGY, int WARPS, int MODE>
__device__ __forceinline__ void alch_items(const Dev &d, int w0, int w1, int a0, int a1, int unit, int units) {
    const int lane = threadIdx.x & 31;
    const int aend = MODE != PAIRS ? a1 + (w1 - w0) : a1;
    for (int it = a0 + unit; it < aend; it += units) {
        if (MODE != PAIRS && it >= a1) {  // restraint item of walker w0 + (it - a1)
            walker_restraints(d, w0 + (it - a1), lane);
            if (MODE == STEP) arrive_stage(d, w0 + (it - a1), lane);
            continue;
        }
        const int w = walker_of_alch(d, w0, w1, it, lane);
        const WalkerDev &W = d.walk[w];
        const SysDev &S = d.sys[W.sys];
        const bool derivs = ENERGY || S.theta_stats;
        const int r = it - W.alch_base;
        int a = d.alch_atoms[S.alch_off + r];
        bool item_ok = la_in(d, a, S.n_atoms);
        if (!item_ok) a = 0;
        int ga = d.slot_of_atom[W.atom_base + a];
        if (!la_in(d, ga, d.n_slots)) ga = W.slot_off, item_ok = false;  // no pairs, still arrives
        const int cnt = item_ok ? d.alch_cnt[it] : 0;
        const int *lst = d.alch_slot + (size_t)it * d.alch_cap;
        // the list is read two rounds ahead and the environment atoms one round
        // ahead of the arithmetic
        auto slot_at = [&](int k) { return k < cnt ? checked_slot(d, lst[k]) : ga; };
        int gb = slot_at(lane), gb_next = slot_at(lane + 32);
        float4 xb = d.xq[gb];
        float2 lb = d.lj[gb];
        const float4 xa = d.xq[ga];
        const float2 la = d.lj[ga];
        double lvd, led, dlvd, dled;
        lambda_path(d.lam[w], S.b_v, S.b_e, lvd, led, dlvd, dled);
        const float le = (float)led;
        // integer soft-core powers by repeated multiplication: the FP64 pipe
        // is narrow on this GPU, and the warps of a block share one SM's
        const float lvn = (float)ipow(lvd, S.sc_n);
        const float dlvn = (float)((double)S.sc_n * ipow(lvd, S.sc_n - 1));
        const float sa = (float)((double)S.sc_alpha * ipow(1.0 - lvd, S.sc_m));
        const float dsdl = (float)(-(double)S.sc_m * S.sc_alpha * ipow(1.0 - lvd, S.sc_m - 1));
        const float eps_a = 0.25f * la.y * la.y;
        const double inv2eps = derivs ? 0.5 / (double)eps_a : 0.0;  // d e4 / d eps_a = e4 / (2 eps_a)
        const float rc2 = S.rc2, krf = S.krf, crf = S.crf;
        float fax = 0.f, fay = 0.f, faz = 0.f;
        double sv = 0.0, se = 0.0, usc_s = 0.0, urf_s = 0.0;
        double th0 = 0.0, th1 = 0.0, th2 = 0.0, th3 = 0.0, th4 = 0.0, th5 = 0.0;
        int npair = 0;
        for (int k = lane; __any_sync(FULL, k < cnt); k += 32) {
            const float4 xc = xb;
            const float2 lc = lb;
            const int gc = gb;
            gb = gb_next;
            xb = d.xq[gb];
            lb = d.lj[gb];
            gb_next = slot_at(k + 64);
            const float dx = min_image(xa.x - xc.x, S.boxf, S.box_invf);
            const float dy = min_image(xa.y - xc.y, S.boxf, S.box_invf);
            const float dz = min_image(xa.z - xc.z, S.boxf, S.box_invf);
            const float r2 = dx * dx + dy * dy + dz * dz;
            if (k >= cnt || r2 >= rc2) continue;
            ++npair;
            const float rinv = rsqrtf(r2);
            const float r2inv = rinv * rinv;
            const float rf_shape = rinv + krf * r2 - crf;
            const float qq = xa.w * xc.w;
            const float rf_u = qq * rf_shape;
            const float rf_f = qq * (rinv * r2inv - 2.0f * krf);
            const float sg = la.x + lc.x;
            const float e4 = la.y * lc.y;
            float sc_f = 0.f, usc = 0.f, dsc = 0.f, g = 0.f, g1 = 0.f, g2 = 0.f, rho6 = 0.f;
            if (e4 > 0.f) {
                const float q2 = r2 / (sg * sg);
                rho6 = q2 * q2 * q2;
                const float s = sa + rho6;
                const float is = 1.0f / s;
                g = is * is - is;
                g1 = is * is - 2.0f * is * is * is;
                g2 = 6.0f * is * is * is * is - 2.0f * is * is * is;
                usc = lvn * e4 * g;
                sc_f = -lvn * e4 * g1 * 6.0f * rho6 * r2inv;
                dsc = dlvn * e4 * g + lvn * e4 * g1 * dsdl;
            }
            const float fs = sc_f + le * rf_f;
            fax = fmaf(fs, dx, fax);
            fay = fmaf(fs, dy, fay);
            faz = fmaf(fs, dz, faz);
            add_force(d, gc, -fs * dx, -fs * dy, -fs * dz);
            sv += (double)dsc;
            se += (double)rf_u;
            if (ENERGY) {
                usc_s += (double)usc;
                urf_s += (double)(le * rf_u);
            }
            if (derivs) {
                if (e4 > 0.f) {
                    th0 += (double)usc * inv2eps;
                    th3 += (double)dsc * inv2eps;
                    const float ds_dsig = -6.0f * rho6 / sg;
                    th1 += 0.5 * (double)(lvn * e4 * g1 * ds_dsig);
                    th4 += 0.5 * (double)(dlvn * e4 * g1 * ds_dsig + lvn * e4 * g2 * ds_dsig * dsdl);
                }
                // d/dq_a of coul q_a q_b shape = sqrt(coul) * (q_b sqrt(coul)) * shape
                const float qb_c = S.sqrt_coul * xc.w;
                th2 += (double)(le * qb_c * rf_shape);
                th5 += (double)(qb_c * rf_shape);
            }
        }
        fax = warp_sumf(fax);
        fay = warp_sumf(fay);
        faz = warp_sumf(faz);
        sv = warp_sum(sv);
        se = warp_sum(se);
        if (ENERGY) {
            usc_s = warp_sum(usc_s);
            urf_s = warp_sum(urf_s);
        }
        if (derivs) {
            th0 = warp_sum(th0); th1 = warp_sum(th1); th2 = warp_sum(th2);
            th3 = warp_sum(th3); th4 = warp_sum(th4); th5 = warp_sum(th5);
        }
        if (ENERGY) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) npair += __shfl_xor_sync(FULL, npair, o);
        }
        if (lane == 0) {
            double *o = d.alch_out + 4 * (size_t)it;
            o[0] = sv;
            o[1] = se;
            if (ENERGY) {
                o[2] = usc_s;
                o[3] = urf_s;
            }
            if (derivs) {
                double *t = d.alch_th + 6 * (size_t)it;
                t[0] = th0; t[1] = th1; t[2] = th2; t[3] = th3; t[4] = th4; t[5] = th5;
            }
            if (ENERGY) atomicAdd(&d.counters[2], (unsigned long long)npair);
        }
        if (MODE == STEP) arrive_stage(d, w, lane);
        if (lane == 0) add_force(d, ga, fax, fay, faz);
    }
}

// bonded terms in the same launch: blocks [0, nblk) of the bonded range
template <bool ENERGY>
__device__ __forceinline__ void bonded_items(const Dev &d, int w0, int w1, int blk, int nblk) {
    const int b0 = d.walk[w0].bo_off;
    const int b1 = d.walk[w1 - 1].bo_off + d.walk[w1 - 1].n_bo;
    const int nthr = nblk * blockDim.x, lane = threadIdx.x & 31;
    // warps run together (32 terms at a time) for the energy sums
    for (int tw = b0 + blk * blockDim.x + (threadIdx.x & ~31); tw < b1; tw += nthr) {
        long long fix = 0;
        int key = -1;
        if (tw + lane < b1) bonded_term<ENERGY>(d, tw + lane, w0, w1, fix, key);
        if (ENERGY) {
            __syncwarp();
            add_energies(d, fix, key);
        }
    }
}

// Items per SM up to which the latency form is taken, and its blocks per SM
// (42.6 KB of shared memory, 124 registers).  The line lies where the two forms
// take the same time, so that a batch whose lists drift across it does not
// notice.  Fused launch, common / latency form, by items per SM: 3.5 (4 x 2049 LJ
// atoms) 28 / 19 us, 4.8 (8 x 772 atoms) 32 / 26, 9.3 (9020 atoms) 36 / 31, 12.1
// (14 x 2049) 31 / 28, 14.3 (128 x 257) 48 / 48, 14.7 (17 x 2049) 34 / 31, 17.2
// (20 x 2049) 35 / 35, 17.9 (160 x 257) 57 / 58, 18.6 (2 x 9020) 43 / 42, 20.7
// (24 x 2049) 35 / 40, 23.9 (2 x 12 300) 47 / 52, 31 (36 x 2049) 43 / 54, 200 (16
// x 12 300) 242 / 366.
constexpr int LAT_ITEMS_PER_SM = 17;
constexpr int LAT_BLOCKS_PER_SM = 4;

// WARPS x 32 threads per CTA; MINB: resident CTAs per SM the register
// allocation is sized for.  Variants (autotuned): 8 warps / 3 CTAs (80
// registers), 4 warps / 7 CTAs (72), 4 warps / 8 CTAs (64).
template <bool ENERGY, int WARPS, int MINB, int MODE, bool LAT>
__global__ void __launch_bounds__(WARPS * 32, MINB) k_pairs(Dev d, int w0, int w1, int nblk_pairs, int a0, int a1,
                                                          int nblk_bonded, int alch_warps) {
    __shared__ std::conditional_t<LAT, PairSharedLat, PairShared<WARPS>> sh;
    // grid: [alchemical items][bonded terms][normal pairs]; the first two come
    // first so that they run alongside the normal pairs.  (The alchemical
    // blocks return here: when their warps went on to the normal pairs, the
    // compiler treated the pair loop as divergent code, 10% more instructions.)
    const int nblk_alch = gridDim.x - nblk_pairs - nblk_bonded;
    if ((int)blockIdx.x < nblk_alch) {
        if ((int)(threadIdx.x >> 5) < alch_warps)
            alch_items<ENERGY, WARPS, MODE>(d, w0, w1, a0, a1, (threadIdx.x >> 5) * nblk_alch + blockIdx.x,
                                             alch_warps * nblk_alch);
        return;
    }
    if (MODE != PAIRS && (int)blockIdx.x < nblk_alch + nblk_bonded) {
        bonded_items<ENERGY>(d, w0, w1, blockIdx.x - nblk_alch, nblk_bonded);
        return;
    }
    constexpr int PER = LAT ? 1 : WARPS;  // items of a block at a time
    const int blk = blockIdx.x - nblk_alch - nblk_bonded;
    if (threadIdx.x < 32) {  // prefix of the walkers' work items
        int acc = 0;
        for (int b = 0; b < w1 - w0; b += 32) {
            const int k = b + threadIdx.x, n = k < w1 - w0 ? d.n_items[w0 + k] : 0;
            int x = n;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int t = __shfl_up_sync(FULL, x, o);
                if ((int)threadIdx.x >= o) x += t;
            }
            if (k < w1 - w0) sh.pre[k] = acc + x - n;
            acc += __shfl_sync(FULL, x, 31);
        }
        // the blocks that take part: as many as a quarter more items would need;
        // the others find the queue at its end without touching it (idle blocks'
        // atomics cost the others 0.5 us of 17 us for 4 x 257 atoms, 3 us of 35 us
        // for 14 x 2049)
        const int parts = min(nblk_pairs, (acc + acc / 4 + PER - 1) / PER);
        if (threadIdx.x == 0) {
            sh.pre[w1 - w0] = acc;
            sh.parts = blk < parts ? parts : 0;
            sh.first = blk < parts ? (int)atomicAdd(&d.counters[CTR_ITEM], (unsigned long long)PER) : acc;
        }
    }
    __syncthreads();
    if constexpr (LAT) normal_items_lat<MODE == STEP ? 8 : 16>(d, w0, w1, sh);
    else normal_items<ENERGY, WARPS, MODE == STEP ? 8 : 16>(d, w0, w1, sh);
}

template <bool ENERGY, int WARPS, int MINB, int MODE, bool LAT>
static void launch_pairs_v(const Dev &d, const HostView &hv, int w0, int w1, cudaStream_t s) {
    // (pair_blocks counts 8-warp CTAs.)  The grid does not depend on the number of
    // items: the queue serves any number, and the lists may grow while a graph
    // that holds the launch is replayed.
    const int nblk = LAT ? LAT_BLOCKS_PER_SM * hv.n_sm : hv.pair_blocks * 8 / WARPS;
    const int a0 = hv.alch_base[w0], a1 = hv.alch_base[w1 - 1] + hv.n_alch[w1 - 1];
    // alchemical warps per block: one, or as few as keep the blocks at one per
    // SM.  They live on FP64 sums, and an SM's FP64 pipe does 1.9 lanes per
    // clock: eight of them in one block took turns on it (42 instead of 30 us
    // for the fused launch of 8 walkers x 772 atoms with theta statistics).
    const int aitems = a1 - a0 + (MODE != PAIRS ? w1 - w0 : 0);
    int awarps = (aitems + hv.n_sm - 1) / hv.n_sm;
    awarps = awarps < 1 ? 1 : (awarps > WARPS ? WARPS : awarps);
    const int ablk = (aitems + awarps - 1) / awarps;
    int bblk = 0;
    if (MODE != PAIRS) {  // bonded terms: about four per thread
        const int nbo = hv.bo_off[w1 - 1] + hv.n_bo[w1 - 1] - hv.bo_off[w0];
        bblk = (nbo + 4 * WARPS * 32 - 1) / (4 * WARPS * 32);
        bblk = bblk > hv.n_sm ? hv.n_sm : bblk;
    }
    const int grid = ablk + bblk + nblk;
    k_pairs<ENERGY, WARPS, MINB, MODE, LAT><<<grid, WARPS * 32, 0, s>>>(d, w0, w1, nblk, a0, a1, bblk, awarps);
}

// launches whose items leave an SM few enough of them take the latency form.
// The counts are those that the last integrator launch met; both forms take
// any number.
bool pairs_latency(const HostView &hv, int w0, int w1) {
    long long n = 0;
    for (int w = w0; w < w1; ++w) n += hv.items[w];
    return hv.pair_variant == 0 && n <= (long long)LAT_ITEMS_PER_SM * hv.n_sm;
}

template <int MODE>
static void launch_pairs_any(const Dev &d, const HostView &hv, int w0, int w1, bool latency, cudaStream_t s) {
    if (latency) launch_pairs_v<false, LAT_WARPS, LAT_BLOCKS_PER_SM, MODE, true>(d, hv, w0, w1, s);
    else if (hv.pair_variant == 1) launch_pairs_v<false, 4, 7, MODE, false>(d, hv, w0, w1, s);
    else if (hv.pair_variant == 2) launch_pairs_v<false, 4, 8, MODE, false>(d, hv, w0, w1, s);
    else launch_pairs_v<false, 8, 3, MODE, false>(d, hv, w0, w1, s);
}

void launch_pairs_fused(const Dev &d, const HostView &hv, bool latency, cudaStream_t s) {
    launch_pairs_any<STEP>(d, hv, 0, hv.n_walkers, latency, s);
}

void launch_pairs(const Dev &d, const HostView &hv, int w0, int w1, cudaStream_t s) {
    launch_pairs_any<PAIRS>(d, hv, w0, w1, pairs_latency(hv, w0, w1), s);
}

void launch_pairs_energy(const Dev &d, const HostView &hv, int w, cudaStream_t s) {
    launch_pairs_v<true, 8, 3, EVAL, false>(d, hv, w, w + 1, s);
}

}  // namespace labf
