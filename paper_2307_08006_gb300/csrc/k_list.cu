// k_list.cu -- neighbour-list rebuild: integer quantization, spatial sort
// into super-clusters, cluster-pair list with exact atom-pair masks, and the
// alchemical pair list.
//
// The listed pair set is defined on integer coordinates so that it is
// bit-exact and independent of floating-point contraction:
//   u = floor(frac(x L^-1) 2^24) (one rounded FP64 product),
//   d = ((u_i - u_j + 2^23) mod 2^24) - 2^23 per component,
//   listed iff D = |d|^2 < R = floor((r_list L^-1)^2 2^48), i < j, the pair is
//   not excluded, and at most one atom is alchemical.
// Each unordered pair appears in exactly one cluster-pair entry: the entry
// whose periodic shift equals the pair's minimum image, with the half-list
// rule (the j super-cluster less than half-way round the index circle from
// the i super-cluster, or the same one with a positive shift, or the same
// one with shift 0 and slot_i < slot_j).
#include "labf_dyn.cuh"
#include "labf_internal.cuh"
#include "labf_launch.h"

namespace labf {

// -------------------------------------------------------------------------
// R1: quantize every real slot and drop it into its xy column's bucket
// -------------------------------------------------------------------------
__global__ void k_quantize(Dev d, int g0, int g1) {
    const int nthr = gridDim.x * blockDim.x;
    for (int g = g0 + blockIdx.x * blockDim.x + threadIdx.x; g < g1; g += nthr) {
        const int w = d.slot_walker[g];
        if (!la_in(d, w, d.n_walkers) || !d.rebuild[w]) continue;
        const int a = d.atom_of_slot[g];
        if (a < 0) continue;
        const WalkerDev &W = d.walk[w];
        const SysDev &S = d.sys[W.sys];
        if (!la_in(d, a, S.n_atoms)) continue;
        const float4 x = d.xq[g];
        const uint32_t ux = quantize(x.x, S.box_inv), uy = quantize(x.y, S.box_inv),
                       uz = quantize(x.z, S.box_inv);
        const int cx = (int)(((unsigned long long)ux * (unsigned)S.ncx) >> 24);
        const int cy = (int)(((unsigned long long)uy * (unsigned)S.ncx) >> 24);
        const int c = cx + S.ncx * cy;
        if (!la_in(d, c, W.n_cols)) continue;
        d.t_uq[g] = make_int4((int)ux, (int)uy, (int)uz, a);
        // one atomic per (walker, column) group of the warp's active lanes
        // (slots of a warp are spatially sorted, so most lanes share one)
        const int key = W.col_off + c;
        const unsigned grp = __match_any_sync(__activemask(), key);
        const int leader = __ffs(grp) - 1;
        const int lane = threadIdx.x & 31;
        int base = 0;
        if (lane == leader) base = atomicAdd(&d.col_count[key], __popc(grp));
        base = __shfl_sync(grp, base, leader);
        const int p = base + __popc(grp & ((1u << lane) - 1u));
        if (p < MAX_COL) d.bucket[(size_t)key * MAX_COL + p] = g;
    }
}

// -------------------------------------------------------------------------
// R2-R6, one block per column: its place among the super-clusters (sizes of
// the columns before it), the column sorted by (u_z, atom id) in shared
// memory and cut into super-clusters of 64; then one warp per super-cluster:
// four k-d splits (longest axis first, ranks by (coordinate, atom id), larger
// half first) give 16 leaves of <= 4 atoms, leaf k in slots 4k..4k+3, and the
// bounding boxes and the state in the new slot order are written.
//
// Latency decides these steps (a rebuild of one system has few columns), so
// they are one launch, and both sorts are bitonic networks of 64-bit keys
// (coordinate, atom id, index within the column): log^2 steps where rank
// counting took one per atom of the column or super-cluster.  The five
// kernels before (scan, scatter, column sort, k-d split, gather) took 57 us
// for one walker of 12 300 atoms and 88 us for 16; this one takes 24 and 35 us.
// -------------------------------------------------------------------------
constexpr int CK_THREADS = 256, CK_WARPS = CK_THREADS / 32;
constexpr int IDX_BITS = 11;  // index within a column
static_assert((1 << IDX_BITS) == MAX_COL, "index bits");
constexpr unsigned long long NO_KEY = ~0ull;

struct ColumnShared {
    unsigned long long key[MAX_COL];
    int x[MAX_COL], y[MAX_COL], z[MAX_COL];
    int part[CK_WARPS];
};

// coordinate (24 bits), atom id (29 bits), index (11 bits)
__device__ __forceinline__ unsigned long long sort_key(int coord, int atom, int idx) {
    return ((unsigned long long)(unsigned)coord << 40) | ((unsigned long long)(unsigned)atom << IDX_BITS) | (unsigned)idx;
}

// ascending bitonic sort of every aligned block of B positions; lane l holds
// positions 2l and 2l + 1
template <int B>
__device__ __forceinline__ void warp_sort(unsigned long long (&k)[2], int lane) {
#pragma unroll
    for (int size = 2; size <= B; size <<= 1) {
#pragma unroll
        for (int t = size >> 1; t > 0; t >>= 1) {
            const bool up = size == B || ((2 * lane) & size) == 0;
            if (t == 1) {
                const bool swap = (k[0] > k[1]) == up;
                const unsigned long long a = swap ? k[1] : k[0], b = swap ? k[0] : k[1];
                k[0] = a;
                k[1] = b;
            } else {
                const bool low = (((2 * lane) & t) == 0) == up;  // keeps the smaller of the two
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const unsigned long long o = __shfl_xor_sync(0xffffffffu, k[h], t >> 1);
                    k[h] = (o < k[h]) == low ? o : k[h];
                }
            }
        }
    }
}

struct Extent {
    int lo[3], hi[3], n;
};
__device__ __forceinline__ Extent extent_of(const int (&u)[2][3], const bool (&real)[2]) {
    Extent e;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        e.lo[c] = min(real[0] ? u[0][c] : 1 << 30, real[1] ? u[1][c] : 1 << 30);
        e.hi[c] = max(real[0] ? u[0][c] : -(1 << 30), real[1] ? u[1][c] : -(1 << 30));
    }
    e.n = (int)real[0] + (int)real[1];
    return e;
}
// joins the extents of the lanes at distance o
__device__ __forceinline__ void join(Extent &e, int o) {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        e.lo[c] = min(e.lo[c], __shfl_xor_sync(0xffffffffu, e.lo[c], o));
        e.hi[c] = max(e.hi[c], __shfl_xor_sync(0xffffffffu, e.hi[c], o));
    }
    e.n += __shfl_xor_sync(0xffffffffu, e.n, o);
}
__device__ __forceinline__ void store_box(int4 *dst, const Extent &e) {
    dst[0] = make_int4(e.lo[0], e.lo[1], e.lo[2], e.n);
    dst[1] = make_int4(e.hi[0], e.hi[1], e.hi[2], 0);
}

// one k-d level: every aligned block of B positions (its atoms first) is
// sorted along its longest axis and its upper half moved to the block's second
// half
template <int B>
__device__ __forceinline__ void kd_level(const ColumnShared &sh, unsigned long long (&k)[2], int (&u)[2][3],
                                         bool (&real)[2], int lane, bool full) {
    Extent e = extent_of(u, real);
#pragma unroll
    for (int o = 1; o < B / 2; o <<= 1) join(e, o);
    // longest axis, the first of equal ones
    int ax = 0, eb = e.hi[0] - e.lo[0];
    if (e.hi[1] - e.lo[1] > eb) {
        ax = 1;
        eb = e.hi[1] - e.lo[1];
    }
    if (e.hi[2] - e.lo[2] > eb) ax = 2;
    constexpr unsigned long long LOW = (1ull << 40) - 1ull;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int c = ax == 0 ? u[h][0] : (ax == 1 ? u[h][1] : u[h][2]);
        k[h] = real[h] ? ((unsigned long long)(unsigned)c << 40) | (k[h] & LOW) : NO_KEY;
    }
    warp_sort<B>(k, lane);
    if (!full) {
        const int half = (e.n + 1) / 2, base = (2 * lane) & ~(B - 1);
        unsigned long long m[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int p = 2 * lane + h - base;  // position in the block; its source rank
            const int r = p < B / 2 ? p : half + p - B / 2;
            const bool on = p < B / 2 ? p < half : r < e.n;
            const int src = on ? base + r : 0;
            const unsigned long long a = __shfl_sync(0xffffffffu, k[0], src >> 1), b = __shfl_sync(0xffffffffu, k[1], src >> 1);
            m[h] = !on ? NO_KEY : (src & 1) ? b : a;
        }
        k[0] = m[0];
        k[1] = m[1];
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        real[h] = k[h] != NO_KEY;
        const int i = (int)(k[h] & (MAX_COL - 1));
        u[h][0] = sh.x[i];
        u[h][1] = sh.y[i];
        u[h][2] = sh.z[i];
    }
}

__global__ void __launch_bounds__(CK_THREADS) k_columns(Dev d, int w0) {
    const int w = w0 + blockIdx.y;
    if (!d.rebuild[w]) return;
    __shared__ ColumnShared sh;
    const WalkerDev &W = d.walk[w];
    const int tid = threadIdx.x, lane = tid & 31, wib = tid >> 5;
    for (int c = blockIdx.x; c < W.n_cols; c += gridDim.x) {
        // super-clusters of the columns before this one
        int before = 0;
        for (int k = tid; k < c; k += CK_THREADS) before += (min(d.col_count[W.col_off + k], MAX_COL) + SC - 1) / SC;
        before = __reduce_add_sync(0xffffffffu, before);
        __syncthreads();  // shared memory free
        if (lane == 0) sh.part[wib] = before;
        const int cnt0 = d.col_count[W.col_off + c];
        const int cnt = min(cnt0, MAX_COL);
        const int *bucket = d.bucket + (size_t)(W.col_off + c) * MAX_COL;
        int size = SC;
        while (size < cnt) size <<= 1;
        for (int k = tid; k < size; k += CK_THREADS) {
            unsigned long long key = NO_KEY;
            if (k < cnt) {
                const int g = bucket[k];
                if (la_in(d, g, d.n_slots)) {  // (an entry out of range becomes padding)
                    const int4 u = d.t_uq[g];
                    sh.x[k] = u.x;
                    sh.y[k] = u.y;
                    sh.z[k] = u.z;
                    key = sort_key(u.z, u.w, k);
                }
            }
            sh.key[k] = key;
        }
        __syncthreads();
        int sc0 = 0;
#pragma unroll
        for (int q = 0; q < CK_WARPS; ++q) sc0 += sh.part[q];
        const int nsc = (cnt + SC - 1) / SC;
        if (tid == 0) {
            if (cnt0 > MAX_COL) set_status(d, LA_STATUS_COLUMN_OVERFLOW);
            d.col_sc[W.col_off + c] = sc0;
            d.col_nsc[W.col_off + c] = nsc;
            if (c == W.n_cols - 1) {
                if (sc0 + nsc > W.sc_cap) set_status(d, LA_STATUS_LIST_OVERFLOW);
                d.n_sc[w] = min(sc0 + nsc, W.sc_cap);
            }
        }
        // bitonic sort; steps of stride <= 32 stay within a warp's own 64 keys
        for (int s = 2; s <= size; s <<= 1) {
            for (int t = s >> 1; t > 0; t >>= 1) {
                if (t > 32 || (t == 32 && s > SC)) __syncthreads(); else __syncwarp();
                for (int i = tid; i < size / 2; i += CK_THREADS) {
                    const int a = 2 * i - (i & (t - 1)), b = a + t;
                    const unsigned long long ka = sh.key[a], kb = sh.key[b];
                    if ((ka > kb) == ((a & s) == 0)) {
                        sh.key[a] = kb;
                        sh.key[b] = ka;
                    }
                }
            }
        }
        __syncthreads();
        for (int q = wib; q < nsc; q += CK_WARPS) {
            const int s_local = sc0 + q, n = min(SC, cnt - q * SC);
            if (s_local >= W.sc_cap) break;
            const int s = W.sc_off + s_local;
            unsigned long long k[2];
            int u[2][3];
            bool real[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int p = 2 * lane + h;
                k[h] = p < n ? sh.key[q * SC + p] : NO_KEY;
                real[h] = k[h] != NO_KEY;
                const int i = (int)(k[h] & (MAX_COL - 1));
                u[h][0] = sh.x[i];
                u[h][1] = sh.y[i];
                u[h][2] = sh.z[i];
            }
            const int first = (int)(__shfl_sync(0xffffffffu, k[0], 0) & (MAX_COL - 1));
            const bool full = n == SC;
            kd_level<64>(sh, k, u, real, lane, full);
            kd_level<32>(sh, k, u, real, lane, full);
            kd_level<16>(sh, k, u, real, lane, full);
            kd_level<8>(sh, k, u, real, lane, full);
            // inside a leaf: by atom id
#pragma unroll
            for (int h = 0; h < 2; ++h)
                if (real[h]) k[h] &= (1ull << 40) - 1ull;
            warp_sort<4>(k, lane);
            const float4 park = d.xq[bucket[first]];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int g = W.slot_off + s_local * SC + 2 * lane + h;
                real[h] = k[h] != NO_KEY;
                const int i = (int)(k[h] & (MAX_COL - 1));
                u[h][0] = sh.x[i];
                u[h][1] = sh.y[i];
                u[h][2] = sh.z[i];
                if (real[h]) {
                    const int old = bucket[i];
                    d.t_xq[g] = d.xq[old];
                    d.t_vv[g] = d.vv[old];
                    d.uq[g] = make_int4(u[h][0], u[h][1], u[h][2], (int)(k[h] >> IDX_BITS));
                } else {
                    // padding: parked on a real atom of the same super-cluster
                    // (finite, never listed)
                    d.t_xq[g] = make_float4(park.x, park.y, park.z, 0.f);
                    d.t_vv[g] = make_float4(0.f, 0.f, 0.f, 0.f);
                    d.uq[g] = make_int4(0, 0, 0, -1);
                }
            }
            // bounding boxes (integer, real atoms only): j-clusters are two lanes,
            // i-clusters four
            Extent e = extent_of(u, real);
            join(e, 1);
            if ((lane & 1) == 0) store_box(d.bb_jc + 2 * ((size_t)s * NJC + (lane >> 1)), e);
            join(e, 2);
            if ((lane & 3) == 0) store_box(d.bb_ic + 2 * ((size_t)s * NIC + (lane >> 2)), e);
            join(e, 4);
            join(e, 8);
            join(e, 16);
            if (lane == 0) store_box(d.bb_sc + 2 * (size_t)s, e);
        }
    }
}

constexpr int LB_WARPS = 8, LB_THREADS = LB_WARPS * 32;
constexpr int LB_COLS = 32;   // columns per round of A (four per warp)
constexpr int LB_VCAP = 512;  // visits per round (a column has at most 3 x 32)
constexpr int LB_CCAP = 512;  // candidates per pass of C and D (a visit has at most 16)
static_assert(LB_COLS == 4 * LB_WARPS && LB_VCAP == 2 * LB_THREADS && 3 * (MAX_COL / SC) <= LB_VCAP, "round sizes");
// counters[8] hands out work items, counters[9] counts blocks that found no
// more; the last one resets both for the next launch
constexpr int CTR_LB_ITEM = 8, CTR_LB_DONE = 9;

// Staged codes: exclusion group (bits 0-29, ids below MAX_GROUPS; "no group"
// differs on the two sides, so one compare decides the group test) |
// EXTRA_FLAG when the slot has extra excluded partners.  Slots without normal pairs (padding,
// alchemical) sit at FAR on the i side and -FAR on the j side, out of every
// list radius.
constexpr int GROUP_MASK = 0x3fffffff, EXTRA_FLAG = 0x40000000;
constexpr int NO_GROUP_I = 0x3fffffff, NO_GROUP_J = 0x3ffffffe;
static_assert(MAX_GROUPS == NO_GROUP_J && NO_GROUP_I == GROUP_MASK, "group ids and codes");
constexpr float FAR = 536870912.0f;  // 2^29

// exclusive scan over the block (v per thread); every thread gets the total
__device__ __forceinline__ int block_scan(int v, int *wtot, int &total) {
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    int x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += t;
    }
    __syncthreads();  // wtot free
    if (lane == 31) wtot[wib] = x;
    __syncthreads();
    int base = 0, tot = 0;
#pragma unroll
    for (int q = 0; q < LB_WARPS; ++q) {
        const int t = wtot[q];
        base += q < wib ? t : 0;
        tot += t;
    }
    total = tot;
    return base + x - v;
}

// R8 plan, by one block before the list kernel: the walkers that rebuild and
// the prefixes of their alchemical atoms and super-clusters
__device__ __forceinline__ void list_plan(const Dev &d, int w0, int w1) {
    __shared__ int wtot[3][LB_WARPS];
    const int w = w0 + threadIdx.x;
    const bool on = w < w1 && d.rebuild[w] != 0;
    const int ns = on ? d.n_sc[w] : 0, na = on ? d.sys[d.walk[w].sys].n_alch : 0;
    int nt, st, at;
    const int r = block_scan(on ? 1 : 0, wtot[0], nt);
    const int sp = block_scan(ns, wtot[1], st);
    const int ap = block_scan(na, wtot[2], at);
    if (on) {
        d.lb_w[r] = w;
        d.lb_spre[r] = sp;
        d.lb_apre[r] = ap;
        d.lb_done[w] = 0;
    }
    if (threadIdx.x == 0) {
        d.lb_tot[0] = nt;
        d.lb_tot[1] = at;
        d.lb_tot[2] = st;
    }
}

// R7: write the new layout back and refresh per-slot parameters (slots of
// unused super-clusters go to the origin), and clear the column counts for the
// next rebuild; the first block also plans the list kernel's work
__global__ void __launch_bounds__(256) k_permute_scatter(Dev d, int g0, int g1, int w0, int w1) {
    if (blockIdx.x == 0) list_plan(d, w0, w1);
    const int nthr = gridDim.x * blockDim.x;
    // (the counts of walkers that do not rebuild are zero already)
    const int c0 = d.walk[w0].col_off, c1 = d.walk[w1 - 1].col_off + d.walk[w1 - 1].n_cols;
    for (int c = c0 + blockIdx.x * blockDim.x + threadIdx.x; c < c1; c += nthr) d.col_count[c] = 0;
    for (int g = g0 + blockIdx.x * blockDim.x + threadIdx.x; g < g1; g += nthr) {
        const int w = d.slot_walker[g];
        if (!d.rebuild[w]) continue;
        const WalkerDev &W = d.walk[w];
        const SysDev &S = d.sys[W.sys];
        const bool used = (g - W.slot_off) / SC < d.n_sc[w];
        int a = used ? d.uq[g].w : -1;
        if (a >= 0 && !la_in(d, a, S.n_atoms)) a = -1;
        float4 x = used ? d.t_xq[g] : make_float4(0.f, 0.f, 0.f, 0.f);
        if (!used) d.uq[g] = make_int4(0, 0, 0, -1);
        // wrap into [0, L) (the list built from this layout assumes it)
        x.x -= S.boxf * floorf(x.x * S.box_invf);
        x.y -= S.boxf * floorf(x.y * S.box_invf);
        x.z -= S.boxf * floorf(x.z * S.box_invf);
        d.vv[g] = used ? d.t_vv[g] : make_float4(0.f, 0.f, 0.f, 0.f);
        d.atom_of_slot[g] = a;
        if (a >= 0) {
            const float4 ap = d.aparam_mut[S.atom_off + a];
            x.w = ap.x;
            d.lj[g] = make_float2(ap.y, ap.z);
            d.im[g] = make_float2(ap.w, d.anoise[S.atom_off + a]);
            d.slot_of_atom[W.atom_base + a] = g;
            const int grp = d.agroup[S.atom_off + a], alch = (int)d.aalch[S.atom_off + a];
            const int4 ex = d.aexcl[S.atom_off + a];
            d.smeta[g] = make_int2(grp, alch);
            d.sexcl[g] = ex;
            d.lcode[g] = alch ? -1 : ((grp >= 0 ? grp : GROUP_MASK) | ((ex.x & ex.y & ex.z & ex.w) != -1 ? EXTRA_FLAG : 0));
        } else {
            d.lj[g] = make_float2(0.f, 0.f);
            d.im[g] = make_float2(0.f, 0.f);
            d.smeta[g] = make_int2(-1, 1);
            d.sexcl[g] = make_int4(-1, -1, -1, -1);
            d.lcode[g] = -1;
        }
        d.xq[g] = x;
        d.xref[g] = x;
    }
}

// -------------------------------------------------------------------------
// R8: cluster-pair list, alchemical list and pair-kernel work items.
//
// One block of eight warps per super-cluster S (work items handed out by a
// global counter, alchemical atoms first):
//   A  the candidate columns, four per warp: lane l tests the column's l-th
//      super-cluster T (cyclic half rule, box distance for the three z
//      images); the visits (T, image) go to shared memory in column, T,
//      image order
//   B  per visit the 16 j-clusters of T against S's box, 16 lanes each, and
//      the candidates compacted in order
//   C  per warp 8 candidates = 32 j-atoms, one per lane: every i-atom of S is
//      broadcast from shared memory and tested, two i-atoms per packed FP32
//      instruction; the lane collects its 64 result bits
//   D  the candidates with a listed pair are appended to S's list in order
// The lists need no per-column sub-lists, no compaction pass and no separate
// launches for the alchemical lists and the work items: the last block of a
// walker cuts its lists into work items.
//
// Bound by instruction issue (68% of the slots; the ALU pipe is active in 49%
// of the cycles, the FMA pipe in 43%).  One j-atom per lane keeps every lane on a candidate
// j-cluster and puts the distances on the FMA pipe; per two i-atoms a lane
// spends 8 packed FP32 and 7 ALU instructions, against about 55 for the two
// half tiles with 64-bit integer arithmetic.  A rebuild of 16 walkers x 12 300
// atoms (r_list 1.15 nm): 196 us, against 468 us for the four kernels before
// (one warp per candidate column, compaction, alchemical lists, items); of one
// such walker: 35 us against 156 us (ncu durations).
//
// The decision D < R is exact although it is made in FP32: coordinates are
// taken relative to S's box, where they are integers below 2^24 (exact in
// FP32), so D is off by less than tol; a lane that meets |D - R| <= tol
// (about one pair in 10^5) repeats its 64 tests in integers.
// -------------------------------------------------------------------------
__device__ __forceinline__ long long bb_dist2(const int4 &alo, const int4 &ahi, const int4 &blo,
                                              const int4 &bhi, int sx, int sy, int sz) {
    long long dx = max(0, max(blo.x + sx - ahi.x, alo.x - (bhi.x + sx)));
    long long dy = max(0, max(blo.y + sy - ahi.y, alo.y - (bhi.y + sy)));
    long long dz = max(0, max(blo.z + sz - ahi.z, alo.z - (bhi.z + sz)));
    return dx * dx + dy * dy + dz * dz;
}

__device__ __forceinline__ int floordiv(int a, int b) { return a >= 0 ? a / b : -((-a + b - 1) / b); }

// nonbonded exclusion of two real atoms (group, then extra partner lists)
__device__ __forceinline__ bool excluded_meta(int a, int2 ma, int4 ea, int b, int2 mb, int4 eb) {
    if (ma.x >= 0 && ma.x == mb.x) return true;
    if (ea.x == b || ea.y == b || ea.z == b || ea.w == b) return true;
    return eb.x == a || eb.y == a || eb.z == a || eb.w == a;
}

struct ListShared {
    float4 row[SC / 2][2];  // i-atoms ia of i-clusters 2p, 2p + 1 at row 8p + ia: {x x' y y'}, {z z' code code'}
    float4 ibox[NIC / 2][2];
    int4 iex[SC];           // extra excluded partners and atom ids of S
    int iatom[SC];
    int colcnt[LB_COLS];
    unsigned visit[LB_VCAP];  // T << 6 | shift bits
    unsigned vmask[LB_VCAP];  // j-clusters of the visit in reach of S's box
    int vpre[LB_VCAP + 1];
    unsigned cand[LB_CCAP];   // visit << 4 | j-cluster
    int cim[LB_CCAP], cpos[LB_CCAP];
    unsigned long long mask[LB_CCAP][JC];
    int wtot[LB_WARPS];
};
struct AlchShared {
    unsigned long long okm[LB_THREADS];
    int near_sc[LB_THREADS], off[LB_THREADS], wtot[LB_WARPS];
};
struct ItemShared {
    int wtot[LB_WARPS];
};

// extra excluded partners: atoms a (list ea) and b (list eb)
__device__ __forceinline__ bool in_extra(int a, const int4 &ea, int b, const int4 &eb) {
    return ea.x == b || ea.y == b || ea.z == b || ea.w == b || eb.x == a || eb.y == a || eb.z == a || eb.w == a;
}

// one lane's 64 tests in integers (coordinates relative to S's box; the
// staged i side holds them exactly); bit ia * 8 + ic
__device__ __noinline__ unsigned long long exact_bits(const ListShared &sh, int jx, int jy, int jz, int jcode,
                                                      long long R) {
    unsigned long long m = 0;
    for (int i = 0; i < SC; ++i) {
        const int ic = i >> 3, ia = i & 7;
        const float *r = reinterpret_cast<const float *>(&sh.row[(ic >> 1) * IC + ia][0]) + (ic & 1);
        const long long dx = jx - (int)r[0], dy = jy - (int)r[2], dz = jz - (int)r[4];
        if (dx * dx + dy * dy + dz * dz < R && ((__float_as_int(r[6]) ^ jcode) & GROUP_MASK) != 0)
            m |= 1ull << (ia * 8 + ic);
    }
    return m;
}

// word |= BIT when e < 0 and the exclusion groups of the two codes differ
template <unsigned BIT>
__device__ __forceinline__ void listed_bit(unsigned &word, float e, int ci, int cj) {
    asm("{\n\t"
        ".reg .pred q, p;\n\t"
        ".reg .b32 t;\n\t"
        "setp.lt.f32 q, %1, 0f00000000;\n\t"
        "lop3.and.b32 t|p, %2, %3, %4, 0x28, q;\n\t"  // ((ci ^ cj) & GROUP_MASK) != 0 && q
        "@p or.b32 %0, %0, %5;\n\t"
        "}"
        : "+r"(word)
        : "f"(e), "r"(ci), "r"(cj), "r"(GROUP_MASK), "n"(BIT));
}

// C: the lane's 64 bits of one j-atom (rel. coordinates jx..jz) against S
__device__ __forceinline__ unsigned long long test_atom(const ListShared &sh, float jx, float jy, float jz, int jcode,
                                                        float Rf, float tol, bool &amb) {
    const f2 nx = pack2(-jx, -jx), ny = pack2(-jy, -jy), nz = pack2(-jz, -jz), nR = pack2(-Rf, -Rf);
    const float reach = Rf + tol;
    unsigned half0 = 0u, half1 = 0u;
    float emin = 3e38f;  // smallest |D - R| met
#pragma unroll 1
    for (int p = 0; p < NIC / 2; ++p) {
        const float4 lo = sh.ibox[p][0], hi = sh.ibox[p][1];
        const float gx = fmaxf(0.f, fmaxf(lo.x - jx, jx - hi.x)), gy = fmaxf(0.f, fmaxf(lo.y - jy, jy - hi.y)),
                    gz = fmaxf(0.f, fmaxf(lo.z - jz, jz - hi.z));
        // no lane within reach of the two i-clusters' box: nothing to test
        if (!__any_sync(0xffffffffu, fmaf(gx, gx, fmaf(gy, gy, gz * gz)) <= reach)) continue;
        unsigned h0 = 0u, h1 = 0u;
#define LABF_ROW(IA)                                                                                     \
    {                                                                                                    \
        const ulonglong2 a = *reinterpret_cast<const ulonglong2 *>(&sh.row[p * IC + IA][0]);              \
        const ulonglong2 b = *reinterpret_cast<const ulonglong2 *>(&sh.row[p * IC + IA][1]);              \
        const f2 dx = add2(a.x, nx), dy = add2(a.y, ny), dz = add2(b.x, nz);                              \
        float e0, e1;                                                                                    \
        unpack2(add2(fma2(dx, dx, fma2(dy, dy, mul2(dz, dz))), nR), e0, e1);                              \
        emin = fminf(fminf(emin, fabsf(e0)), fabsf(e1));                                                 \
        listed_bit<(1u << ((IA & 3) * 8))>(IA < 4 ? h0 : h1, e0, (int)b.y, jcode);                        \
        listed_bit<(2u << ((IA & 3) * 8))>(IA < 4 ? h0 : h1, e1, (int)(b.y >> 32), jcode);                \
    }
        LABF_ROW(0) LABF_ROW(1) LABF_ROW(2) LABF_ROW(3) LABF_ROW(4) LABF_ROW(5) LABF_ROW(6) LABF_ROW(7)
#undef LABF_ROW
        half0 |= h0 << (2 * p);
        half1 |= h1 << (2 * p);
    }
    amb = emin <= tol;
    return ((unsigned long long)half1 << 32) | half0;
}

__device__ __forceinline__ void list_item(const Dev &d, ListShared &sh, int w, int S_loc) {
    const int tid = threadIdx.x, lane = tid & 31, wib = tid >> 5;
    const WalkerDev &W = d.walk[w];
    const SysDev &S = d.sys[W.sys];
    const int s = W.sc_off + S_loc, gS = W.slot_off + S_loc * SC;
    const int nsc = d.n_sc[w], ncx = S.ncx, cspan = S.cspan;
    const int U = 1 << 24;
    const long long R = S.R;
    const float Rf = (float)R;
    // conversion of coordinates beyond 2^24 (at most 1 each, so 2 sqrt(3 D) in
    // D) and the roundings of D, twice over
    const float tol = fmaf(Rf, 9.5367431640625e-07f, 16.0f * (float)S.Rq);
    const int4 slo = d.bb_sc[2 * (size_t)s], shi = d.bb_sc[2 * (size_t)s + 1];
    // ---- stage S ----
    bool extra = false;
    if (tid < SC) {
        const int4 u = d.uq[gS + tid];
        const int code = d.lcode[gS + tid];
        const int ic = tid >> 3, ia = tid & 7;
        float *r = reinterpret_cast<float *>(&sh.row[(ic >> 1) * IC + ia][0]) + (ic & 1);
        r[0] = code < 0 ? FAR : (float)(u.x - slo.x);
        r[2] = code < 0 ? FAR : (float)(u.y - slo.y);
        r[4] = code < 0 ? FAR : (float)(u.z - slo.z);
        const int g = code & GROUP_MASK;
        r[6] = __int_as_float((g == GROUP_MASK ? NO_GROUP_I : g) | (code & EXTRA_FLAG));
        sh.iatom[tid] = u.w;
        sh.iex[tid] = d.sexcl[gS + tid];
        extra = code >= 0 && (code & EXTRA_FLAG);
    } else if (tid < SC + NIC / 2) {
        const int p = tid - SC;
        float4 lo = make_float4(4e9f, 4e9f, 4e9f, 0.f), hi = make_float4(-4e9f, -4e9f, -4e9f, 0.f);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int4 a = d.bb_ic[2 * ((size_t)s * NIC + 2 * p + h)], b = d.bb_ic[2 * ((size_t)s * NIC + 2 * p + h) + 1];
            if (a.w <= 0) continue;
            lo = make_float4(fminf(lo.x, (float)(a.x - slo.x)), fminf(lo.y, (float)(a.y - slo.y)),
                             fminf(lo.z, (float)(a.z - slo.z)), 0.f);
            hi = make_float4(fmaxf(hi.x, (float)(b.x - slo.x)), fmaxf(hi.y, (float)(b.y - slo.y)),
                             fmaxf(hi.z, (float)(b.z - slo.z)), 0.f);
        }
        sh.ibox[p][0] = lo;
        sh.ibox[p][1] = hi;
    }
    const bool s_extra = __syncthreads_or(extra) != 0;
    const int cx0 = (int)(((long long)(slo.x - S.Rq) * ncx) >> 24);
    const int cx1 = (int)(((long long)(shi.x + S.Rq) * ncx) >> 24);
    const int cy0 = (int)(((long long)(slo.y - S.Rq) * ncx) >> 24);
    const int cy1 = (int)(((long long)(shi.y + S.Rq) * ncx) >> 24);
    if (tid == 0 && (cx1 - cx0 >= cspan || cy1 - cy0 >= cspan))
        set_status(d, LA_STATUS_LIST_OVERFLOW);  // cannot happen for boxes inside a column
    const size_t ebase = (size_t)s * d.ent_cap;
    int nent = 0;
    const int ncol = cspan * cspan;
    for (int c0 = 0; c0 < ncol;) {
        // ---- A: visits of up to 32 columns, four per warp ----
        unsigned zp = 0;  // z images in range of this lane's T, 3 bits per own column
        int t_of[4], bits_of[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int k = c0 + 4 * wib + q;
            const int cx = cx0 + k % cspan, cy = cy0 + k / cspan;
            unsigned z = 0;
            t_of[q] = bits_of[q] = 0;
            if (k < ncol && cx <= cx1 && cy <= cy1) {
                const int ty = floordiv(cy, ncx), tx = floordiv(cx, ncx);
                const int col = cx - tx * ncx + ncx * (cy - ty * ncx);
                bits_of[q] = (tx + 1) | ((ty + 1) << 2);
                if (la_in(d, col, W.n_cols)) {
                    const int T_loc = d.col_sc[W.col_off + col] + lane;
                    t_of[q] = T_loc;
                    bool partner = lane < min(d.col_nsc[W.col_off + col], MAX_COL / SC) && T_loc < nsc;
                    // cyclic half list over super-clusters: T is S's partner when it
                    // lies less than half-way round the index circle
                    if (partner && T_loc != S_loc) {
                        const int del = T_loc > S_loc ? T_loc - S_loc : T_loc - S_loc + nsc;
                        partner = !(2 * del > nsc || (2 * del == nsc && T_loc < S_loc));
                    }
                    if (partner) {
                        const int t = W.sc_off + T_loc;
                        const int4 tlo = d.bb_sc[2 * (size_t)t], thi = d.bb_sc[2 * (size_t)t + 1];
                        if (tlo.w != 0)
                            for (int tz = -1; tz <= 1; ++tz) {
                                if (T_loc == S_loc && (tx < 0 || (tx == 0 && (ty < 0 || (ty == 0 && tz < 0))))) continue;
                                if (bb_dist2(slo, shi, tlo, thi, tx * U, ty * U, tz * U) < R) z |= 1u << (tz + 1);
                            }
                    }
                }
            }
            zp |= z << (3 * q);
            const int cnt = __reduce_add_sync(0xffffffffu, __popc(z));
            if (lane == 0) sh.colcnt[4 * wib + q] = cnt;
        }
        __syncthreads();
        // the leading columns whose visits fit the buffer (all of them, but for
        // very crowded boxes)
        const int cc = sh.colcnt[lane];
        int incl = cc;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += t;
        }
        const int ncols = __popc(__ballot_sync(0xffffffffu, incl <= LB_VCAP));
        const int nvis = __shfl_sync(0xffffffffu, incl, ncols - 1);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int col = 4 * wib + q;
            int pos = __shfl_sync(0xffffffffu, incl - cc, col);
            const unsigned z = (zp >> (3 * q)) & 7u;
            const int n = __popc(z);
            int x = n;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int t = __shfl_up_sync(0xffffffffu, x, o);
                if (lane >= o) x += t;
            }
            if (col < ncols) {
                pos += x - n;
                for (unsigned m = z; m; m &= m - 1u)
                    sh.visit[pos++] = ((unsigned)t_of[q] << 6) | bits_of[q] | ((unsigned)(__ffs(m) - 1) << 4);
            }
        }
        __syncthreads();
        c0 += ncols;
        // ---- B: the visits' j-clusters against S's box ----
        for (int vb = 2 * wib; vb < nvis; vb += 2 * LB_WARPS) {
            const int v = vb + (lane >> 4);
            bool ok = false;
            if (v < nvis) {
                const unsigned vis = sh.visit[v];
                const size_t b = 2 * ((size_t)(W.sc_off + (int)(vis >> 6)) * NJC + (lane & 15));
                const int4 jlo = d.bb_jc[b], jhi = d.bb_jc[b + 1];
                ok = jlo.w > 0 && bb_dist2(slo, shi, jlo, jhi, ((int)(vis & 3) - 1) * U, ((int)((vis >> 2) & 3) - 1) * U,
                                           ((int)((vis >> 4) & 3) - 1) * U) < R;
            }
            const unsigned m = __ballot_sync(0xffffffffu, ok);
            if ((lane & 15) == 0 && v < nvis) sh.vmask[v] = (m >> (lane & 16)) & 0xffffu;
        }
        __syncthreads();
        {
            const int n0 = 2 * tid < nvis ? __popc(sh.vmask[2 * tid]) : 0;
            const int n1 = 2 * tid + 1 < nvis ? __popc(sh.vmask[2 * tid + 1]) : 0;
            int tot;
            const int pre = block_scan(n0 + n1, sh.wtot, tot);
            sh.vpre[2 * tid] = pre;
            sh.vpre[2 * tid + 1] = pre + n0;
            if (tid == 0) sh.vpre[LB_VCAP] = tot;
        }
        __syncthreads();
        for (int v0 = 0; v0 < nvis;) {
            // the visits [v0, v1) whose candidates fit a pass
            const int base = sh.vpre[v0];
            int v1 = nvis;
            if (sh.vpre[LB_VCAP] - base > LB_CCAP) {
                int lo = v0 + 1, hi = nvis;  // largest v1 with vpre[v1] - base <= LB_CCAP
                while (lo < hi) {
                    const int mid = (lo + hi + 1) >> 1;
                    if (sh.vpre[mid] - base <= LB_CCAP) lo = mid; else hi = mid - 1;
                }
                v1 = lo;
            }
            const int nc = (v1 < LB_VCAP ? sh.vpre[v1] : sh.vpre[LB_VCAP]) - base;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int v = 2 * tid + h;
                if (v < v0 || v >= v1) continue;
                int pos = sh.vpre[v] - base;
                for (unsigned m = sh.vmask[v]; m; m &= m - 1u) sh.cand[pos++] = ((unsigned)v << 4) | (__ffs(m) - 1);
            }
            __syncthreads();
            // ---- C: atom tests, eight candidates per warp ----
            for (int g = wib; 8 * g < nc; g += LB_WARPS) {
                const int c = 8 * g + (lane >> 2), q = lane & 3;
                int rx = 0, ry = 0, rz = 0, jcode = NO_GROUP_J, gj = 0;
                bool real = false, self0 = false;
                if (c < nc) {
                    const unsigned cd = sh.cand[c], vis = sh.visit[cd >> 4];
                    const int T_loc = (int)(vis >> 6), sj = (int)(cd & 15u) * JC + q;
                    gj = W.slot_off + T_loc * SC + sj;
                    const int4 u = d.uq[gj];
                    const int code = d.lcode[gj];
                    real = code >= 0;
                    rx = u.x + ((int)(vis & 3) - 1) * U - slo.x;
                    ry = u.y + ((int)((vis >> 2) & 3) - 1) * U - slo.y;
                    rz = u.z + ((int)((vis >> 4) & 3) - 1) * U - slo.z;
                    const int gr = code & GROUP_MASK;
                    jcode = (gr == GROUP_MASK ? NO_GROUP_J : gr) | (code & EXTRA_FLAG);
                    self0 = T_loc == S_loc && (vis & 63u) == 21u;  // no shift
                }
                bool amb;
                unsigned long long m = test_atom(sh, real ? (float)rx : -FAR, real ? (float)ry : -FAR,
                                                 real ? (float)rz : -FAR, jcode, Rf, tol, amb);
                if (amb) m = exact_bits(sh, rx, ry, rz, jcode, R);
                if (self0) {  // the same super-cluster: only slot_i < slot_j
                    const int sj = gj - gS, a = sj >> 3, b = sj & 7;
                    const unsigned long long ones = 0x0101010101010101ull;
                    m &= ((1ull << a) - 1ull) * ones | (ones & ((1ull << (8 * b)) - 1ull)) << a;
                }
                if (__any_sync(0xffffffffu, m != 0ull && (s_extra || (jcode & EXTRA_FLAG))) && m != 0ull) {
                    const int b = d.uq[gj].w;
                    const int4 eb = d.sexcl[gj];
                    for (unsigned long long k = m; k; k &= k - 1ull) {
                        const int bit = __ffsll((long long)k) - 1, i = (bit & 7) * IC + (bit >> 3);
                        if (in_extra(sh.iatom[i], sh.iex[i], b, eb)) m &= ~(1ull << bit);
                    }
                }
                unsigned f = (unsigned)m | (unsigned)(m >> 32);
                f |= f >> 16;
                f = (f | (f >> 8)) & 0xffu;
                f |= __shfl_xor_sync(0xffffffffu, f, 1);
                f |= __shfl_xor_sync(0xffffffffu, f, 2);
                if (c < nc) {
                    sh.mask[c][q] = m;
                    if (q == 0) sh.cim[c] = (int)f;
                }
            }
            __syncthreads();
            // ---- D: append the candidates with a listed pair ----
            for (int b = 0; b < nc; b += LB_THREADS) {
                const int c = b + tid;
                const unsigned im = c < nc ? (unsigned)sh.cim[c] : 0u;
                int tot;
                const int e = nent + block_scan(im ? 1 : 0, sh.wtot, tot);
                nent += tot;
                if (c < nc) {
                    sh.cpos[c] = im && e < d.ent_cap ? e : -1;
                    if (im && e < d.ent_cap) {
                        // i-cluster mask twice: bits 8-15 are pruned by the batched
                        // step, bits 16-23 keep the listed set
                        const unsigned cd = sh.cand[c], vis = sh.visit[cd >> 4];
                        d.ent_hdr[ebase + e] = make_int2(W.slot_off + (int)(vis >> 6) * SC + (int)(cd & 15u) * JC,
                                                         (int)((vis & 63u) | (im << 8) | (im << 16)));
                    }
                }
            }
            __syncthreads();
            for (int k = tid; k < nc * JC; k += LB_THREADS) {
                const int e = sh.cpos[k >> 2];
                if (e >= 0)
                    *reinterpret_cast<unsigned long long *>(d.ent_lb + 32 * (ebase + e) + 8 * (k & 3)) = sh.mask[k >> 2][k & 3];
            }
            __syncthreads();
            v0 = v1;
        }
    }
    if (tid == 0) {
        if (nent > d.ent_cap) set_status(d, LA_STATUS_LIST_OVERFLOW);
        d.sc_nent[s] = min(nent, d.ent_cap);
    }
}

// alchemical list of one (walker, alchemical atom): super-cluster boxes are
// tested one per thread, the near ones compacted in ascending order and
// tested slot by slot by the block's warps in turn; the hits are written in
// (super-cluster, slot) order
__device__ __forceinline__ void alch_item(const Dev &d, AlchShared &sh, int w, int r) {
    const int tid = threadIdx.x, lane = tid & 31, wib = tid >> 5;
    const WalkerDev &W = d.walk[w];
    const SysDev &S = d.sys[W.sys];
    const int it = W.alch_base + r;
    const int a = d.alch_atoms[S.alch_off + r];
    if (!la_in(d, a, S.n_atoms)) return;
    const int ga = d.slot_of_atom[W.atom_base + a];
    if (!la_in(d, ga, d.n_slots)) return;
    const int4 ua = d.uq[ga];
    const int2 ma = d.smeta[ga];
    const int4 ea = d.sexcl[ga];
    const int U = 1 << 24;
    int cnt = 0;
    const int nsc = d.n_sc[w];
    int *out = d.alch_slot + (size_t)it * d.alch_cap;
    for (int b0 = 0; b0 < nsc; b0 += LB_THREADS) {
        // super-cluster box within the list radius of the atom (any image)
        bool near = false;
        if (b0 + tid < nsc) {
            const size_t t = (size_t)(W.sc_off + b0 + tid);
            const int4 tlo = d.bb_sc[2 * t], thi = d.bb_sc[2 * t + 1];
            if (tlo.w > 0) {
                long long D = 0;
                const int uc[3] = {ua.x, ua.y, ua.z};
                const int lc[3] = {tlo.x, tlo.y, tlo.z}, hc[3] = {thi.x, thi.y, thi.z};
                for (int c = 0; c < 3; ++c) {
                    long long best = -1;
                    for (int sh3 = -1; sh3 <= 1; ++sh3) {
                        const long long gap = max(0, max(lc[c] + sh3 * U - uc[c], uc[c] - (hc[c] + sh3 * U)));
                        if (best < 0 || gap < best) best = gap;
                    }
                    D += best * best;
                }
                near = D < S.R;
            }
        }
        int nn;
        const int pos = block_scan(near ? 1 : 0, sh.wtot, nn);
        if (near) sh.near_sc[pos] = b0 + tid;
        __syncthreads();
        for (int kk = wib; kk < nn; kk += LB_WARPS) {
            const int gbase = W.slot_off + sh.near_sc[kk] * SC;
            unsigned bits[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int g = gbase + lane + 32 * h;
                const int4 ub = d.uq[g];
                const int2 mb = d.smeta[g];
                const int4 eb = d.sexcl[g];
                bool ok = false;
                if (ub.w >= 0 && !mb.y) {
                    const long long dx = torus_delta(ub.x, ua.x), dy = torus_delta(ub.y, ua.y),
                                    dz = torus_delta(ub.z, ua.z);
                    ok = dx * dx + dy * dy + dz * dz < S.R && !excluded_meta(a, ma, ea, ub.w, mb, eb);
                }
                bits[h] = __ballot_sync(0xffffffffu, ok);
            }
            if (lane == 0) sh.okm[kk] = ((unsigned long long)bits[1] << 32) | bits[0];
        }
        __syncthreads();
        int tot;
        const int off = block_scan(tid < nn ? __popcll(sh.okm[tid]) : 0, sh.wtot, tot);
        sh.off[tid] = cnt + off;
        __syncthreads();
        for (int kk = wib; kk < nn; kk += LB_WARPS) {
            const int gbase = W.slot_off + sh.near_sc[kk] * SC;
            const unsigned long long om = sh.okm[kk];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int b = lane + 32 * h;
                const int pos2 = sh.off[kk] + __popcll(om & ((1ull << b) - 1ull));
                if (((om >> b) & 1ull) && pos2 < d.alch_cap) out[pos2] = gbase + b;
            }
        }
        cnt += tot;
        __syncthreads();
    }
    if (tid == 0) {
        if (cnt > d.alch_cap) set_status(d, LA_STATUS_ALCH_OVERFLOW);
        d.alch_cnt[it] = min(cnt, d.alch_cap);
    }
}

// pair-kernel work items of a walker (chunks of `chunk` entries of one
// super-cluster); clears the rebuild flag.  In the batched step (prune_fresh)
// a walker with pruning on has its fresh list pruned by this step's pair pass.
// Entry counts may come from other blocks of the launch: read past L1.
__device__ __forceinline__ void make_items(const Dev &d, ItemShared &sh, int w, int prune_fresh) {
    const WalkerDev &W = d.walk[w];
    const int nsc = d.n_sc[w];
    int done = 0;
    for (int base = 0; base < nsc; base += LB_THREADS) {
        const int sl = base + threadIdx.x;
        const int ne = sl < nsc ? __ldcg(d.sc_nent + W.sc_off + sl) : 0;
        const int nch = (ne + d.chunk - 1) / d.chunk;
        int tot;
        const int first = done + block_scan(nch, sh.wtot, tot);
        done += tot;
        for (int c = 0; c < nch; ++c)
            if (first + c < W.item_cap)
                d.items[W.item_base + first + c] = make_int4(W.sc_off + sl, c * d.chunk, min(ne, (c + 1) * d.chunk), w);
    }
    if (threadIdx.x == 0) {
        if (done > W.item_cap) set_status(d, LA_STATUS_LIST_OVERFLOW);
        d.n_items[w] = min(done, W.item_cap);
        d.rebuild[w] = 0;
        d.near[w] = 0;
        if (prune_fresh && d.sys[W.sys].prune_disp2 > 0.f) d.prune_now[w] = d.step[w] + 1ull;
        atomicAdd(&d.counters[0], 1ull);
    }
}

// work items alone (the autotuner's other chunk sizes)
__global__ void __launch_bounds__(LB_THREADS) k_items(Dev d, int w0) {
    __shared__ ItemShared sh;
    const int w = w0 + blockIdx.x;
    if (d.rebuild[w]) make_items(d, sh, w, 0);
}

__global__ void __launch_bounds__(LB_THREADS, 4) k_listbuild(Dev d, int prune_fresh) {
    __shared__ union {
        ListShared list;
        AlchShared alch;
        ItemShared item;
    } sh;
    __shared__ int s_w[LA_MAX_WALKERS_PER_LAUNCH], s_pre[2][LA_MAX_WALKERS_PER_LAUNCH];
    __shared__ int s_idx, s_last;
    const int tid = threadIdx.x;
    const int nw = d.lb_tot[0], n_alch = d.lb_tot[1], total = n_alch + d.lb_tot[2];
    if (tid < nw) {
        s_w[tid] = d.lb_w[tid];
        s_pre[0][tid] = d.lb_apre[tid];
        s_pre[1][tid] = d.lb_spre[tid];
    }
    // the next item's index is fetched one item ahead
    int next = 0;
    if (tid == 0) next = (int)atomicAdd(&d.counters[CTR_LB_ITEM], 1ull);
    for (;;) {
        if (tid == 0) s_idx = next;
        __syncthreads();
        const int idx = s_idx;
        if (idx >= total) break;
        if (tid == 0) next = (int)atomicAdd(&d.counters[CTR_LB_ITEM], 1ull);
        const bool alch = idx < n_alch;
        const int v = alch ? idx : idx - n_alch;
        const int *pre = s_pre[alch ? 0 : 1];
        int lo = 0, hi = nw - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (pre[mid] <= v) lo = mid; else hi = mid - 1;
        }
        const int w = s_w[lo];
        if (alch) {
            alch_item(d, sh.alch, w, v - pre[lo]);
            __syncthreads();
            continue;
        }
        list_item(d, sh.list, w, v - pre[lo]);
        if (tid == 0) {
            __threadfence();
            s_last = atomicAdd(&d.lb_done[w], 1u) == (unsigned)d.n_sc[w] - 1u;
        }
        __syncthreads();
        if (s_last) {  // the walker's last super-cluster: cut its lists into work items
            __threadfence();
            make_items(d, sh.item, w, prune_fresh);
        }
        __syncthreads();
    }
    // the last block out resets the work counters for the next launch
    if (tid == 0) {
        __threadfence();
        const unsigned long long done = atomicAdd(&d.counters[CTR_LB_DONE], 1ull);
        if (done == (unsigned long long)gridDim.x - 1ull) {
            d.counters[CTR_LB_ITEM] = 0ull;
            d.counters[CTR_LB_DONE] = 0ull;
            __threadfence();
        }
    }
}

__global__ void k_gate(Dev d, int w0, int w1, cudaGraphConditionalHandle handle, int conditional) {
    gate_work(d, w0, w1, handle, conditional);
}

void launch_gate(const Dev &d, int w0, int w1, cudaGraphConditionalHandle handle, bool conditional,
                 cudaStream_t s) {
    k_gate<<<1, 256, 0, s>>>(d, w0, w1, handle, conditional ? 1 : 0);
}

// the one-walker-per-launch form's coalescing (no pruning there)
__global__ void k_coalesce(Dev d, int w0, int w1) {
    __shared__ int any;
    if (threadIdx.x == 0) any = 0;
    __syncthreads();
    for (int w = w0 + threadIdx.x; w < w1; w += blockDim.x)
        if (d.rebuild[w]) any = 1;
    __syncthreads();
    coalesce_rebuilds(d, w0, w1, any);
}

void launch_coalesce(const Dev &d, int w0, int w1, cudaStream_t s) { k_coalesce<<<1, 256, 0, s>>>(d, w0, w1); }

// -------------------------------------------------------------------------
// host launcher of the whole rebuild chain (every kernel exits early for
// walkers whose rebuild flag is clear)
// -------------------------------------------------------------------------
void launch_rebuild(const Dev &d, const HostView &hv, int w0, int w1, cudaStream_t s, bool batched) {
    const int g0 = hv.slot_off[w0], g1 = hv.slot_off[w1 - 1] + hv.slot_cap[w1 - 1];
    int sb = (g1 - g0 + 255) / 256;
    sb = sb < 1 ? 1 : (sb > hv.n_sm * 8 ? hv.n_sm * 8 : sb);
    const int nw = w1 - w0;
    int max_cols = 1;
    for (int w = w0; w < w1; ++w) max_cols = hv.n_cols[w] > max_cols ? hv.n_cols[w] : max_cols;
    int nsc = 0;
    for (int w = w0; w < w1; ++w) nsc += hv.sc_cap[w];
    const int a0 = hv.alch_base[w0], a1 = hv.alch_base[w1 - 1] + hv.n_alch[w1 - 1];
    k_quantize<<<sb, 256, 0, s>>>(d, g0, g1);
    k_columns<<<dim3(max_cols < 1024 ? max_cols : 1024, nw), CK_THREADS, 0, s>>>(d, w0);
    k_permute_scatter<<<sb, LB_THREADS, 0, s>>>(d, g0, g1, w0, w1);
    const int lb = nsc + a1 - a0 < hv.n_sm * 4 ? nsc + a1 - a0 : hv.n_sm * 4;  // resident grid
    k_listbuild<<<lb < 1 ? 1 : lb, LB_THREADS, 0, s>>>(d, batched ? 1 : 0);
}

void launch_items(const Dev &d, const HostView &, int w0, int w1, cudaStream_t s) {
    k_items<<<w1 - w0, LB_THREADS, 0, s>>>(d, w0);
}

int rebuild_kernel_count(const HostView &, int, int) { return 4; }

}  // namespace labf
