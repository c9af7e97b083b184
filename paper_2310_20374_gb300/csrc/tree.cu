// tree.cu -- octree build from sorted Hilbert keys (Sect. 3.4.1, 3.4.6) and
// the two tree climbs of Sect. 3.4.2 (collision search: Eqs. center, rmax,
// rcrit; gravity: Eqs. expansion_center, rmax_2, rcrit_2 with the corner cap,
// the opening angle theta(M) of Dehnen 2002 Eq. 13) with P2M
// (Eq. multipole_moment) at the leaves and M2M (App. C) at the parents.
//
// Cells are stored level-major, in Hilbert order within a level, children of a
// cell contiguous; every cell owns a contiguous range of the key-sorted
// moonlets.  All geometry that decides the walk (centres, r_max, r_crit) is
// computed with exactly rounded FP64 operations in the same order as a plain
// sequential evaluation (moonlets in key order, children in cell order), so
// it is reproducible bit for bit.
#include "ctx.h"

namespace ncorp {

// exponents (a, b, c) of every packed symmetric index up to order 7
struct ExpTable {
    unsigned char e[off(MAXP + 2)][3];
};
constexpr ExpTable make_exp_table() {
    ExpTable t{};
    for (int n = 0; n <= MAXP + 1; n++)
        for (int k = 0; k <= n; k++)
            for (int c = 0; c <= k; c++) {
                int idx = off(n) + tri(k) + c;
                t.e[idx][0] = static_cast<unsigned char>(n - k);
                t.e[idx][1] = static_cast<unsigned char>(k - c);
                t.e[idx][2] = static_cast<unsigned char>(c);
            }
    return t;
}
__constant__ ExpTable c_exp = make_exp_table();

// ---------------------------------------------------------------------------
// Build: every cell is found from the sorted keys by the moonlet it starts
// with, all levels at once, in one cooperative launch with one grid barrier.
//
// Let lcp(a, b) be the number of leading octal digits two keys share (the depth
// of the deepest cell that could hold both), and a moonlet i with
// l = lcp(key[i - 1], key[i]) (-1 at a disk's first moonlet).  A cell of level L
// starts at i iff l < L and its parent, the cell of level L - 1 that holds i, is
// split (more than s moonlets, level below MAX_LEVEL):
//   - a parent that starts at i is split iff lcp(key[i], key[i + s]) >= L - 1;
//   - the parent of the first of them (level l + 1) starts at some p < i, found
//     by a binary search among the s keys before i (if it starts earlier still it
//     holds more than s), and is split iff lcp(key[p], key[p + s]) >= l.
// So the cells starting at i have the levels L0 = l + 1 .. Lmax, the deepest is a
// leaf and the others are not.  The index of a cell (level-major, Hilbert order
// within a level) is its level's first index plus the number of cells of that
// level starting before i: per-block counts of every level, one grid barrier,
// prefix sums over blocks, then ballots.  A cell's end is known to the moonlet j
// that starts the next cell: j ends the cells of levels L0(j) .. the leaf level of
// j - 1.  Counts (end - start) and children are added with atomics into zeroed
// fields.
//
// Latency-bound: a level-by-level build (a grid barrier, the placement and
// dependent octant searches per level) took 46 / 90 / 268 us at N = 1e3 / 1e5 /
// 1e6 with its two helper launches; this takes 12 / 22 / 76 us.
// ---------------------------------------------------------------------------
struct BuildArgs {
    const uint64_t *key;
    const uint32_t *qx, *qy, *qz;
    int n, s, cap, chunk;   // chunk: moonlets per block, a multiple of BUILD_T
    int *level, *first, *count, *child0, *nchild, *parent, *arrive_m;
    uint32_t *cx, *cy, *cz;
    int *wcnt, *woff;       // the walk's per-cell counts [cap + 1], zeroed for it
    int *leaves, *leaf_of;  // leaf_of[i] first holds moonlet i's levels, (L0 << 8 | Lmax) or -1
    int *bcount;            // [gridDim.x][BUILD_ROW]: cells of each level the block starts, its leaves, and the leaf
                            // level of its last start (-1: none)
    Ctrl *ctl;
    const int *gate;        // nothing to do while *gate is 0 (null: always build)
};

constexpr int BUILD_T = 256, BUILD_W = BUILD_T / 32;
constexpr int BUILD_LEVELS = MAX_LEVEL + 1;   // levels 0 .. MAX_LEVEL
constexpr int BUILD_COUNTS = BUILD_LEVELS + 1;   // and the leaves (every moonlet that starts cells starts one leaf)
constexpr int BUILD_ROW = BUILD_COUNTS + 1;
static_assert(BUILD_COUNTS <= 32, "a lane per count");

__device__ __forceinline__ int common_levels(uint64_t a, uint64_t b) {
    const uint64_t x = a ^ b;
    return x ? (__clzll(static_cast<long long>(x)) - 1) / 3 : MAX_LEVEL;
}

// The levels (L0, Lmax) of the cells starting at moonlet i of the disk [d0, d1); false: none.
__device__ __forceinline__ bool cells_starting(const BuildArgs &A, int i, int d0, int d1, int &L0, int &Lmax) {
    const uint64_t k = __ldg(&A.key[i]);
    const int s = A.s;
    int l = -1;
    if (i > d0) {
        l = common_levels(__ldg(&A.key[i - 1]), k);
        if (l >= MAX_LEVEL) return false;
        const int shift = 63 - 3 * l;
        const uint64_t lo_key = l > 0 ? (k >> shift) << shift : 0;   // first key of the level-l cell that holds i
        if (i - d0 < s || __ldg(&A.key[i - s]) < lo_key) {           // the cell starts less than s before i
            int p = max(d0, i - s), e = i - 1;
            while (p < e) {
                const int mid = (p + e) >> 1;
                if (__ldg(&A.key[mid]) < lo_key) p = mid + 1;
                else e = mid;
            }
            if (d1 - p <= s || common_levels(__ldg(&A.key[p + s]), k) < l) return false;
        }
    }
    L0 = l + 1;
    Lmax = L0;
    if (d1 - i > s) Lmax = max(L0, min(MAX_LEVEL, common_levels(k, __ldg(&A.key[i + s])) + 1));
    return true;
}

__global__ void __launch_bounds__(BUILD_T) k_build(BuildArgs A) {
    __shared__ int s_cnt[BUILD_COUNTS];                   // phase 1: the block's cells per level, its leaves
    __shared__ int s_base[BUILD_COUNTS];                  // next index of each level, next leaf
    __shared__ unsigned s_bal[BUILD_W][BUILD_COUNTS];        // starts of each level among the warp's moonlets
    __shared__ int s_pre[BUILD_W][BUILD_COUNTS];          // index of the first of them
    __shared__ int s_tot[BUILD_COUNTS], s_low[BUILD_COUNTS];
    __shared__ int s_last[BUILD_W];                       // leaf level of the last start in each warp's moonlets
    __shared__ int s_prev;
    if ((A.gate && *A.gate == 0) || aborted(A.ctl)) return;   // every block, before the barrier
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5, b = blockIdx.x, G = gridDim.x;
    const int c0 = min(A.n, b * A.chunk), c1 = min(A.n, c0 + A.chunk);
    const unsigned le = 0xffffffffu >> (31 - lane);       // lanes up to this one
    const int *doff = A.ctl->doff;
    // ---- 1. the cells each moonlet starts, and the block's counts
    for (int i = b * BUILD_T + tid; i <= A.cap; i += G * BUILD_T) {
        if (i < A.cap) A.count[i] = A.nchild[i] = 0;
        A.wcnt[i] = A.woff[i] = 0;
    }
    if (tid < BUILD_COUNTS) s_cnt[tid] = 0;
    if (tid == 0) s_prev = -1;
    __syncthreads();
    for (int i = c0 + tid; i < c1; i += BUILD_T) {
        int d0 = 0, d1 = A.n;
        if (doff) {
            const int d = A.ctl->disk_of[i];
            d0 = __ldg(&doff[d]);
            d1 = __ldg(&doff[d + 1]);
        }
        int L0 = 0, Lmax = 0, code = -1;
        if (cells_starting(A, i, d0, d1, L0, Lmax)) {
            code = L0 << 8 | Lmax;
            for (int L = L0; L <= Lmax; L++) atomicAdd(&s_cnt[L], 1);
            atomicAdd(&s_cnt[BUILD_LEVELS], 1);
            atomicMax(&s_prev, (i - c0) << 5 | Lmax);
        }
        A.leaf_of[i] = code;
    }
    __syncthreads();
    if (tid < BUILD_COUNTS) A.bcount[b * BUILD_ROW + tid] = s_cnt[tid];
    if (tid == BUILD_COUNTS) A.bcount[b * BUILD_ROW + BUILD_COUNTS] = s_prev < 0 ? -1 : s_prev & 31;
    unsigned bar = 0;
    if (!grid_sync_on(&A.ctl->bar_build, A.ctl, bar)) return;
    // ---- 2. totals of every level, and what the blocks before this one hold (a warp per level)
    for (int L = w; L < BUILD_COUNTS; L += BUILD_W) {
        int tot = 0, low = 0;
        for (int q = lane; q < G; q += 32) {
            const int v = __ldcg(&A.bcount[q * BUILD_ROW + L]);
            tot += v;
            if (q < b) low += v;
        }
        tot = warp_sum(tot);
        low = warp_sum(low);
        if (lane == 0) {
            s_tot[L] = tot;
            s_low[L] = low;
        }
    }
    if (w == BUILD_W - 1) {   // the leaf level of the last start before this block
        int m = -1;
        for (int q = lane; q < b; q += 32) {
            const int v = __ldcg(&A.bcount[q * BUILD_ROW + BUILD_COUNTS]);
            if (v >= 0) m = max(m, q << 5 | v);
        }
        m = __reduce_max_sync(0xffffffffu, m);
        if (lane == 0) s_prev = m < 0 ? -1 : m & 31;
    }
    __syncthreads();
    if (w == 0) {
        const int t = lane < BUILD_LEVELS ? s_tot[lane] : 0;
        int incl = t;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int u = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += u;
        }
        if (lane < BUILD_COUNTS) s_base[lane] = (lane < BUILD_LEVELS ? incl - t : 0) + s_low[lane];
        if (b == 0) {   // the tree's description
            const unsigned used = __ballot_sync(0xffffffffu, t > 0);
            if (lane <= BUILD_LEVELS) A.ctl->level_start[lane] = incl - t;   // (levels past the deepest are empty)
            if (lane == 31) {
                A.ctl->n_cells = incl;
                A.ctl->n_leaves = s_tot[BUILD_LEVELS];
                A.ctl->max_level = 31 - __clz(static_cast<int>(used));
                A.ctl->col_stale = 1;   // a new tree: no collision pairs listed for it yet
                A.ctl->bar_count = 0;   // for the cooperative kernel that follows
                if (incl > A.cap) atomicOr(&A.ctl->err, ERR_CELLS);
            }
        }
    }
    __syncthreads();
    // ---- 3. the cells, BUILD_T moonlets at a time
    int level_base = lane < BUILD_COUNTS ? s_base[lane] : 0;   // warp 0: running index of level `lane`, of the leaves
    int prev = s_prev;                                         // leaf level of the last start before the tile
    for (int t0 = c0; t0 < c1; t0 += BUILD_T) {
        const int i = t0 + tid;
        const int code = i < c1 ? A.leaf_of[i] : -1;
        const bool starts = code >= 0;
        const int L0 = starts ? code >> 8 : 32, Lmax = starts ? code & 255 : -1;
        const int lv_lo = __reduce_min_sync(0xffffffffu, L0), lv_hi = __reduce_max_sync(0xffffffffu, Lmax);
        unsigned mine = 0;
        for (int L = lv_lo; L <= lv_hi; L++) {
            const unsigned bal = __ballot_sync(0xffffffffu, L0 <= L && L <= Lmax);
            if (lane == L) mine = bal;
        }
        const unsigned any = __ballot_sync(0xffffffffu, starts);
        if (lane == BUILD_LEVELS) mine = any;
        const int last = __shfl_sync(0xffffffffu, Lmax, any ? 31 - __clz(static_cast<int>(any)) : 0);
        __syncthreads();   // the last tile's reads of the shared arrays are over
        if (lane < BUILD_COUNTS) s_bal[w][lane] = mine;
        if (lane == 0) s_last[w] = any ? last : -1;
        __syncthreads();
        if (w == 0 && lane < BUILD_COUNTS) {
#pragma unroll
            for (int q = 0; q < BUILD_W; q++) {
                s_pre[q][lane] = level_base;
                level_base += __popc(s_bal[q][lane]);
            }
        }
        __syncthreads();
        // leaf level of the last start before the warp, then before and up to the lane
        int before = prev;
        for (int q = 0; q < BUILD_W; q++) {
            const int v = s_last[q];
            if (v >= 0) {
                if (q < w) before = v;
                prev = v;
            }
        }
        const unsigned lt = any & (le >> 1);
        const int src = lt ? 31 - __clz(static_cast<int>(lt)) : 0;
        const int from = __shfl_sync(0xffffffffu, Lmax, src);
        const int leaf_before = lt ? from : before;            // leaf level of moonlet i - 1
        const int leaf_here = starts ? Lmax : leaf_before;     // and of moonlet i
        // index of the cell of level L that holds moonlet i (its last start at or before i), or i - 1
        auto upto = [&](int L) { return s_pre[w][L] + __popc(s_bal[w][L] & le) - 1; };
        auto below = [&](int L) { return s_pre[w][L] + __popc(s_bal[w][L] & (le >> 1)) - 1; };
        if (i < c1) A.leaf_of[i] = upto(leaf_here);
        if (starts) {
            const int slot = upto(BUILD_LEVELS);
            if (slot < A.cap) A.leaves[slot] = upto(Lmax);
            const uint32_t qx = A.qx[i], qy = A.qy[i], qz = A.qz[i];
            int par = L0 > 0 ? below(L0 - 1) : -1;
            for (int L = L0; L <= Lmax; L++) {
                const int c = upto(L);
                if (c < A.cap) {
                    A.level[c] = L;
                    A.first[c] = i;
                    A.child0[c] = L < Lmax ? upto(L + 1) : -1;
                    A.parent[c] = par;
                    A.arrive_m[c] = 0;   // arrival counters of the multipoles, zeroed as cells are made
                    A.cx[c] = qx >> (KEY_BITS - L);
                    A.cy[c] = qy >> (KEY_BITS - L);
                    A.cz[c] = qz >> (KEY_BITS - L);
                    atomicAdd(&A.count[c], -i);
                    if (par >= 0) atomicAdd(&A.nchild[par], 1);
                }
                par = c;
            }
            for (int L = L0; L <= leaf_before; L++) {   // the cells that end where this one starts
                const int c = below(L);
                if (c < A.cap) atomicAdd(&A.count[c], i);
            }
        }
        if (i == A.n - 1)   // and those that end with the last moonlet
            for (int L = 0; L <= leaf_here; L++) {
                const int c = upto(L);
                if (c < A.cap) atomicAdd(&A.count[c], A.n);
            }
    }
}

static int coop_grid(ncorp_ctx *c, const void *kernel, int block, size_t smem) {
    int per_sm = 0;
    NCORP_CUDA_CHECK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, block, smem));
    if (per_sm < 1) per_sm = 1;
    if (per_sm > 2) per_sm = 2;
    return coop_blocks(c, per_sm);
}

void launch_build(ncorp_ctx *c, const ParticleSet &P, int n, int s, const int *gate) {
    Cells &C = c->cells;
    BuildArgs A;
    A.gate = gate;
    A.key = P.key;
    A.qx = P.qx; A.qy = P.qy; A.qz = P.qz;
    A.n = n; A.s = s; A.cap = C.cap;
    A.level = C.level; A.first = C.first; A.count = C.count; A.child0 = C.child0; A.nchild = C.nchild;
    A.parent = C.parent; A.cx = C.cx; A.cy = C.cy; A.cz = C.cz;
    A.arrive_m = C.arrive_m;
    A.leaves = C.leaves; A.leaf_of = C.leaf_of;
    A.wcnt = c->wl.cnt; A.woff = c->wl.p2p_off;
    A.bcount = C.blocksum; A.ctl = c->ctl;
    // ctl->bar_build was zeroed by k_keys
    const int most = std::min(coop_grid(c, reinterpret_cast<const void *>(k_build), BUILD_T, 0),
                              BLOCKSUM_INTS / BUILD_ROW);
    const int tiles = (n + BUILD_T - 1) / BUILD_T, per = (tiles + most - 1) / most;
    A.chunk = per * BUILD_T;
    const int grid = (tiles + per - 1) / per;
    void *args[] = {&A};
    NCORP_CUDA_CHECK(cudaLaunchCooperativeKernel(reinterpret_cast<const void *>(k_build), dim3(grid), dim3(BUILD_T),
                                                 args, 0, c->stream));
    c->launches++;
}

// ---------------------------------------------------------------------------
// Corner cap (Sect. 3.4.2): distance from s to the farthest corner of the
// cell's cube, the cube widened by L 2^-48 on each side.
// ---------------------------------------------------------------------------
// One FP64 warp instruction takes 64 cycles of its SM sub-partition, a divide
// 550, a square root 584, a compare and select 111, a conversion 84.  So what
// only looks at an FP64 value's bits is done in integers: maxima and compares
// of values that are not negative, scalings by powers of two.

// v 2^e for a power of two v (or 0): exact, as ldexp
__device__ __forceinline__ double scale_pow2(double v, int e) {
    const long long u = __double_as_longlong(v);
    const int ex = static_cast<int>(u >> 52) & 0x7ff;
    if (ex + e > 0 && ex + e < 0x7ff && ex > 0) return __longlong_as_double(u + (static_cast<long long>(e) << 52));
    return ldexp(v, e);
}

// the larger of a >= 0 and b, b taken as 0 when it is NaN or negative (fmax of a >= 0 and b)
__device__ __forceinline__ double max_nn(double a, double b) {
    const long long x = __double_as_longlong(a), y = __double_as_longlong(b);
    return (y > x && y <= 0x7ff0000000000000ll) ? b : a;
}

// a < b for values that are not negative (false when b is NaN or a is)
__device__ __forceinline__ bool less_nn(double a, double b) {
    const long long x = __double_as_longlong(a), y = __double_as_longlong(b);
    return x < y && y <= 0x7ff0000000000000ll;
}

// root: the cube of the cell's disk (x_lo, y_lo, z_lo, L)
__device__ __forceinline__ double cell_side(const double *root, int lev) { return scale_pow2(root[3], -lev); }

// the root cube of cell c's disk
__device__ __forceinline__ const double *cell_root(const Ctrl *ctl, const int *first, int c) {
    return disk_root(ctl, disk_of(ctl, first[c]));
}

__device__ __forceinline__ double corner_axis(const double *root, int k, double h, uint32_t c, double s) {
    const double eps = scale_pow2(root[3], -48);
    const double lo = dadd(root[k], dmul(__dsub_rn(__hiloint2double(0x43300000, static_cast<int>(c)), 0x1p52), h));
    const double a = dsub(s, dsub(lo, eps));
    const double b = dsub(dadd(dadd(lo, h), eps), s);
    // (a + b = h + 2 eps > 0: at most one is negative, so the integer order is the values')
    return __double_as_longlong(a) > __double_as_longlong(b) ? a : b;
}

// Power-of-two scale of a cell's expansions: the smallest >= r_max (so |x - s|/rho <= 1)
// and >= side/256, so that the scale ratios met in M2M, M2L and L2L stay
// below 2^(level difference + 8) even for one-moonlet cells (r_max ~ 0).
__device__ __forceinline__ double cell_scale(const double *root, int lev, double rmax) {
    const double v = max_nn(rmax, scale_pow2(cell_side(root, lev), -8));
    const long long u = __double_as_longlong(v);
    const int ex = static_cast<int>(u >> 52) & 0x7ff;
    if (ex == 0 || ex >= 0x7fe) return pow2_ceil(v);
    return __longlong_as_double((u & 0xfffffffffffffll) ? static_cast<long long>(ex + 1) << 52 : u);
}

// FP32 double-float copy of a coordinate: hi = fl32(v), lo = fl32(v - hi)
__device__ __forceinline__ void split1(double v, float &hi, float &lo) {
    hi = static_cast<float>(v);
    lo = static_cast<float>(v - static_cast<double>(hi));
}

// The three coordinates of a centre, one on each of lanes base + first .. + 2, as FP32 pairs on every lane
__device__ __forceinline__ void gather_split(float h, float l, int from, float4 &hi, float4 &lo) {
    hi.x = __shfl_sync(0xffffffffu, h, from);
    hi.y = __shfl_sync(0xffffffffu, h, from + 1);
    hi.z = __shfl_sync(0xffffffffu, h, from + 2);
    lo.x = __shfl_sync(0xffffffffu, l, from);
    lo.y = __shfl_sync(0xffffffffu, l, from + 1);
    lo.z = __shfl_sync(0xffffffffu, l, from + 2);
    hi.w = lo.w = 0.f;
}

// ---------------------------------------------------------------------------
// Climbs.  GB300 executes an FP64 warp instruction in the same time whatever
// the number of active lanes, so the sequential, order-fixed FP64 sums that
// make the geometry reproducible bit for bit are spread one cell per thread
// (leaves) or one sum per lane (parents), never run on a single lane.
// r_max of a leaf is sqrt(max_i |x_i - s|^2): a correctly rounded square root
// is non-decreasing, so this equals max_i sqrt(|x_i - s|^2) exactly.
// ---------------------------------------------------------------------------
struct ClimbArgs {
    const double *x, *y, *z, *m;
    const float4 *hi4, *lo4;
    const double *vx, *vy, *vz, *R;
    int *first, *count, *child0, *nchild, *parent, *level;
    uint32_t *cx, *cy, *cz;
    double *M, *sx, *sy, *sz, *rmax, *rcrit, *rho;
    float4 *gh, *gl;
    void *Mh;
    float4 *cv4;
    const int *leaves;
    Ctrl *ctl;
    double G, dt, theta;
    double K3;                // (theta_min^5 / (1 - theta_min)^2)^3
    int cap;
    WalkStart ws;             // the walk that follows
    const double *rc_given;   // collision climb (nullable): each moonlet's R + dt |v| given (tree order)
    const int *gate;          // collision climb (nullable): nothing to do while *gate is 0
};

constexpr int CLIMB_WARPS_COOP = 8;

// ---- leaves: eight leaves per warp, four lanes per leaf.  The centre's
// sums run in the oracle's order, one sum per lane (q = 0: the weights,
// q = 1..3: the weighted coordinates), so a warp instruction advances 32
// independent sums; the maxima over the moonlets are exact in any order and
// are split over the four lanes.
constexpr int LEAF_GROUP = 8;

struct LeafSlot {
    int sub, q, base, t, c, f, cnt;
    bool valid;
};

__device__ __forceinline__ LeafSlot leaf_slot(const ClimbArgs &A, int gw, int lane, int n_leaves) {
    LeafSlot L;
    L.sub = lane >> 2;
    L.q = lane & 3;
    L.base = lane & ~3;
    L.t = gw * LEAF_GROUP + L.sub;
    L.valid = L.t < n_leaves;
    L.c = L.valid ? A.leaves[L.t] : 0;
    L.f = L.valid ? A.first[L.c] : 0;
    L.cnt = L.valid ? A.count[L.c] : 0;
    return L;
}

__device__ __forceinline__ double quad_max(double v) {   // (of values that are not negative)
    v = max_nn(v, __shfl_xor_sync(0xffffffffu, v, 1));
    return max_nn(v, __shfl_xor_sync(0xffffffffu, v, 2));
}

// The largest of a leaf's values, found in FP32: every lane keeps the largest
// and second largest FP32 estimate of its quarter and where the largest is.
// After the quad's maximum is known, only the moonlets whose estimate reaches
// it within the estimates' error (2^-18 of it, four times the bound) need the
// exact FP64 value: one a leaf as a rule, evaluated once for the whole warp.
// A leaf whose estimates may not show it (a second candidate on one lane, values
// that are not finite or too small to carry their relative error) is left to
// the exact loop over its moonlets: settle() is false on its four lanes.
struct LeafMax {
    float best = -1.f, second = -1.f;
    int at = -1;
    bool odd = false;      // an estimate that says nothing
    __device__ __forceinline__ void add(float v, int k) {
        if (!(v >= 0.f && v < 3e38f)) odd = true;
        if (v > best) {
            second = best;
            best = v;
            at = k;
        } else if (v > second) {
            second = v;
        }
    }
    // floor_: values at or below it say nothing.  On true, `at` is the lane's candidate (-1: none).
    __device__ __forceinline__ bool settle(float floor_, int base) {
        float m = fmaxf(best, __shfl_xor_sync(0xffffffffu, best, 1));
        m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 2));
        const float thr = m * (1.0f - 0x1p-18f);
        const bool ok = !odd && m > floor_ && !(second >= thr);
        if (!(best >= thr)) at = -1;
        return ((__ballot_sync(0xffffffffu, ok) >> base) & 0xfu) == 0xfu;
    }
};

// Corner cap of the leaf (lanes q = 0..2 take one axis each), returned on every lane of the quad.
__device__ __forceinline__ double quad_corner(const ClimbArgs &A, const LeafSlot &L, double sx, double sy, double sz) {
    double d = 0.0;
    if (L.valid && L.q < 3) {   // (lanes of the other quads run with it)
        const int lev = A.level[L.c];
        const double *rt = disk_root(A.ctl, disk_of(A.ctl, L.f));
        const double h = cell_side(rt, lev);
        d = corner_axis(rt, L.q, h, L.q == 0 ? A.cx[L.c] : (L.q == 1 ? A.cy[L.c] : A.cz[L.c]),
                        L.q == 0 ? sx : (L.q == 1 ? sy : sz));
    }
    const double d0 = __shfl_sync(0xffffffffu, d, L.base), d1 = __shfl_sync(0xffffffffu, d, L.base + 1),
                 d2 = __shfl_sync(0xffffffffu, d, L.base + 2);
    return dnorm3(d0, d1, d2);
}

// FP32 estimate of |x_k - s|^2 of moonlet k, s given as FP32 pairs
__device__ __forceinline__ float dist2_f32(const float4 &h, const float4 &l, const float4 &sh, const float4 &sl) {
    const float dx = (h.x - sh.x) + (l.x - sl.x), dy = (h.y - sh.y) + (l.y - sl.y), dz = (h.z - sh.z) + (l.z - sl.z);
    return dx * dx + dy * dy + dz * dz;
}

// max_k |x_k - s|^2 of the quad's leaf, exact, on every lane of the quad; sh, sl: the centre in FP32 pairs
// (which carry an absolute error of 2^-47 |s|: distances below 2^-20 |s| are left to the exact loop)
__device__ __forceinline__ double leaf_dist2(const ClimbArgs &A, const LeafSlot &L, double sx, double sy, double sz,
                                             const float4 &sh, const float4 &sl) {
    LeafMax M;
    for (int k = L.f + L.q; k < L.f + L.cnt; k += 4) M.add(dist2_f32(A.hi4[k], A.lo4[k], sh, sl), k);
    const float fl = (fabsf(sh.x) + fabsf(sh.y) + fabsf(sh.z)) * 0x1p-20f;
    double d2 = 0.0;
    if (M.settle(fl * fl + 1e-30f, L.base)) {
        const int k = M.at;
        if (k >= 0) d2 = dsq3(dsub(A.x[k], sx), dsub(A.y[k], sy), dsub(A.z[k], sz));
    } else {
        for (int k = L.f + L.q; k < L.f + L.cnt; k += 4)
            d2 = max_nn(d2, dsq3(dsub(A.x[k], sx), dsub(A.y[k], sy), dsub(A.z[k], sz)));
    }
    __syncwarp();
    return quad_max(max_nn(0.0, d2));
}

// ---- gravity leaves (Eqs. expansion_center, rmax_2, corner cap): the
// group of LEAF_GROUP leaves of warp-group gw.
__device__ __forceinline__ void leaf_gravity_group(const ClimbArgs &A, int gw, int lane, int n_leaves) {
    const LeafSlot L = leaf_slot(A, gw, lane, n_leaves);
    const double *coord = L.q == 1 ? A.x : (L.q == 2 ? A.y : A.z);
    double acc = 0.0;
#pragma unroll 4
    for (int k = L.f; k < L.f + L.cnt; k++) {
        const double m = A.m[k], c = coord[k];
        acc = dadd(acc, L.q == 0 ? m : dmul(m, c));
    }
    const double M = __shfl_sync(0xffffffffu, acc, L.base);
    const double sq = L.q == 0 ? M : ddiv(acc, M);
    const double sx = __shfl_sync(0xffffffffu, sq, L.base + 1), sy = __shfl_sync(0xffffffffu, sq, L.base + 2),
                 sz = __shfl_sync(0xffffffffu, sq, L.base + 3);
    float h1, l1;
    split1(sq, h1, l1);
    float4 hi, lo;
    gather_split(h1, l1, L.base + 1, hi, lo);
    double rmax = dsqrt(leaf_dist2(A, L, sx, sy, sz, hi, lo));
    const double cap = quad_corner(A, L, sx, sy, sz);
    if (less_nn(cap, rmax)) rmax = cap;
    if (L.valid && L.q == 0) {
        const int c = L.c;
        const double rho = cell_scale(cell_root(A.ctl, A.first, c), A.level[c], rmax);
        A.M[c] = M;
        A.sx[c] = sx;
        A.sy[c] = sy;
        A.sz[c] = sz;
        A.rmax[c] = rmax;
        A.rho[c] = rho;
        lo.w = static_cast<float>(rho);
        A.gh[c] = hi;
        A.gl[c] = lo;
    }
}

// acc[midx(beta)] += mu d^beta for orders 0 and 2..P-1
template <int P, typename real>
__device__ __forceinline__ void p2m_add(real dx, real dy, real dz, real mu, real *acc) {
    real px[P], py[P], pz[P];
    px[0] = py[0] = pz[0] = real(1);
#pragma unroll
    for (int k = 1; k < P; k++) {
        px[k] = px[k - 1] * dx;
        py[k] = py[k - 1] * dy;
        pz[k] = pz[k - 1] * dz;
    }
    acc[0] += mu;
#pragma unroll
    for (int n = 2; n < P; n++)
#pragma unroll
        for (int k = 0; k <= n; k++)
#pragma unroll
            for (int c = 0; c <= k; c++) acc[midx(n - k, k - c, c)] += mu * px[n - k] * py[k - c] * pz[c];
}

// ---- gravity geometry of parents from their children (Eqs. expansion_center,
// rmax_2, corner cap), four parents per warp, eight lanes each (a parent has
// at most eight children), so that one FP64 warp instruction advances four
// parents.  Lane j of a group holds child j; lanes
// j = 0..3 form the centre's sums over the children in child order (lane 0
// the mass, as w * 1 = w exactly, lanes 1..3 the weighted coordinates).  c is
// the group's parent, -1 for none; every lane of the warp calls this.
constexpr int PARENT_GROUP = 4;

// Sums over a parent's children in child order: lane 0 of its eight the
// weights w, lanes 1..3 the weighted coordinates; lane j < nch gives child j's.
// Each lane forms its own child's products, so a child costs the sums one FP64
// addition.
__device__ __forceinline__ double children_sum(double w, double x, double y, double z, int nch, int j, int base) {
    const double wx = dmul(w, x), wy = dmul(w, y), wz = dmul(w, z);
    const int most = __reduce_max_sync(0xffffffffu, nch);
    double acc = 0.0;
    for (int ch = 0; ch < most; ch++) {
        const double a = __shfl_sync(0xffffffffu, w, base + ch), bx = __shfl_sync(0xffffffffu, wx, base + ch),
                     by = __shfl_sync(0xffffffffu, wy, base + ch), bz = __shfl_sync(0xffffffffu, wz, base + ch);
        if (ch < nch) acc = dadd(acc, j == 1 ? bx : (j == 2 ? by : (j == 3 ? bz : a)));
    }
    return acc;
}

__device__ __forceinline__ void parent_gravity_group(const ClimbArgs &A, int c, int lane) {
    const int j = lane & 7, base = lane & ~7;
    const bool valid = c >= 0;
    const int c0 = valid ? A.child0[c] : 0, nch = valid ? A.nchild[c] : 0;
    double cm = 0.0, csx = 0.0, csy = 0.0, csz = 0.0, crm = 0.0;
    if (j < nch) {
        cm = __ldcg(&A.M[c0 + j]);
        csx = __ldcg(&A.sx[c0 + j]);
        csy = __ldcg(&A.sy[c0 + j]);
        csz = __ldcg(&A.sz[c0 + j]);
        crm = __ldcg(&A.rmax[c0 + j]);
    }
    const double acc = children_sum(cm, csx, csy, csz, nch, j, base);
    const double M = __shfl_sync(0xffffffffu, acc, base);
    const double q = ddiv(acc, M);
    const double px = __shfl_sync(0xffffffffu, q, base + 1), py = __shfl_sync(0xffffffffu, q, base + 2),
                 pz = __shfl_sync(0xffffffffu, q, base + 3);
    double rm = 0.0;
    if (j < nch) rm = dadd(crm, dnorm3(dsub(csx, px), dsub(csy, py), dsub(csz, pz)));
    rm = max_nn(0.0, rm);
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) rm = max_nn(rm, __shfl_xor_sync(0xffffffffu, rm, o));
    float h1, l1;
    split1(q, h1, l1);
    float4 hi, lo;
    gather_split(h1, l1, base + 1, hi, lo);
    const int plev = valid ? A.level[c] : 0;
    double d = 0.0;
    if (valid && j < 3) {
        const double *rt = cell_root(A.ctl, A.first, c);
        const double h = cell_side(rt, plev);
        d = corner_axis(rt, j, h, j == 0 ? A.cx[c] : (j == 1 ? A.cy[c] : A.cz[c]), j == 0 ? px : (j == 1 ? py : pz));
    }
    const double d0 = __shfl_sync(0xffffffffu, d, base), d1 = __shfl_sync(0xffffffffu, d, base + 1),
                 d2 = __shfl_sync(0xffffffffu, d, base + 2);
    const double pcap = dnorm3(d0, d1, d2);
    if (less_nn(pcap, rm)) rm = pcap;
    if (valid && j == 0) {
        const double prho = cell_scale(cell_root(A.ctl, A.first, c), plev, rm);
        A.M[c] = M;
        A.sx[c] = px;
        A.sy[c] = py;
        A.sz[c] = pz;
        A.rmax[c] = rm;
        A.rho[c] = prho;
        lo.w = static_cast<float>(prho);
        A.gh[c] = hi;
        A.gl[c] = lo;
    }
}

// ---- multipoles (Eq. multipole_moment, scaled: M-hat_beta = sum mu (d/rho)^beta / beta!,
// orders 0 and 2..p-1; the dipole vanishes about the centre of mass).
// Leaves take the sum over their moonlets (one warp per leaf, lanes over the
// moonlets, a butterfly sum per coefficient).  A parent takes its children's
// moments translated to its own centre (the M2M shift of App. C), which in
// scaled form reads, with delta = (s_c - s_P)/rho_P and r = rho_c/rho_P,
//   M-hat_P(beta) = sum_children sum_{gamma <= beta, |gamma| != 1}
//                   M-hat_c(gamma) r^|gamma| delta^(beta - gamma) / (beta - gamma)!
// (the multinomial expansion of (d_c + delta)^beta / beta!, axis by axis).
// The children are added in child order.
struct P2MArgs {
    const double *x, *y, *z, *m;
    const float4 *hi4, *lo4;
    const int *first, *count, *child0, *nchild, *parent, *leaves;
    int *arrive;       // per cell: children whose moments are done (zeroed by the build)
    const double *sx, *sy, *sz, *rho;
    const float4 *gh, *gl;
    void *Mh;
    double G;
    Ctrl *ctl;
};

constexpr int P2M_WARPS = 4;

template <int P, typename real>
struct M2MShared {
    real a[P2M_WARPS][8][off(P) < 1 ? 1 : off(P)];   // per child: full storage, orders 0..P-1
    real b[P2M_WARPS][8][off(P) < 1 ? 1 : off(P)];
};

// (n, b + c, c) of slot j of the full storage (orders 0..P-1): order n starts
// at n(n+1)(n+2)/6, and within it k = b + c runs 0..n with c = 0..k
template <int P>
__device__ __forceinline__ void full_exps(int j, int &n, int &kk, int &c) {
    n = 0;
    while (n + 1 < P && off(n + 1) <= j) n++;
    const int rem = j - off(n);
    kk = 0;
    while (kk < n && tri(kk + 1) <= rem) kk++;
    c = rem - tri(kk);
}

// One-dimensional shift of full-storage moments along AXIS: out(a,b,c) = sum_{k <= exponent} in(... - k e_axis) w_k
template <int P, int AXIS, typename real>
__device__ __forceinline__ real m_shift(const real *in, const real (&w)[P], int n, int kk, int c) {
    const int ax = AXIS == 0 ? n - kk : (AXIS == 1 ? kk - c : c);   // the exponent along the axis
    real s = real(0);
#pragma unroll
    for (int k = 0; k < P; k++) {
        if (k > ax) break;
        const int m = n - k, t = AXIS == 0 ? kk : kk - k, cc = AXIS == 2 ? c - k : c;
        s += in[m * (m + 1) * (m + 2) / 6 + t * (t + 1) / 2 + cc] * w[k];
    }
    return s;
}

// Eight leaves per warp, four lanes per leaf: each lane sums a quarter of its
// leaf's moonlets, then the four partial sums are added by two butterfly
// steps and each lane stores a quarter of the coefficients.  Every lane of
// the warp calls this (valid: the lane's group has a leaf).
template <int P, typename real>
__device__ __forceinline__ void leaf_moments(const P2MArgs &A, int c, bool valid, int q, real *Mh) {
    constexpr int NM = num_m(P);
    real acc[NM];
#pragma unroll
    for (int j = 0; j < NM; j++) acc[j] = real(0);
    if (valid) {
        const int f = A.first[c], e = f + A.count[c];
        if constexpr (sizeof(real) == 4) {   // double-float difference, no FP64 work
            const float4 gh = A.gh[c], gl = A.gl[c];
            const float ir = 1.0f / gl.w;   // exact: rho is a power of two
            for (int k = f + q; k < e; k += 4) {
                const float4 h = A.hi4[k], l = A.lo4[k];
                p2m_add<P, real>(((h.x - gh.x) + (l.x - gl.x)) * ir, ((h.y - gh.y) + (l.y - gl.y)) * ir,
                                 ((h.z - gh.z) + (l.z - gl.z)) * ir, h.w, acc);
            }
        } else {
            const double irho = 1.0 / A.rho[c], sx = A.sx[c], sy = A.sy[c], sz = A.sz[c];
            for (int k = f + q; k < e; k += 4)
                p2m_add<P, real>((A.x[k] - sx) * irho, (A.y[k] - sy) * irho, (A.z[k] - sz) * irho, A.G * A.m[k], acc);
        }
    }
#pragma unroll
    for (int n = 0; n < P; n++) {
        if (n == 1) continue;
#pragma unroll
        for (int k = 0; k <= n; k++)
#pragma unroll
            for (int cc = 0; cc <= k; cc++) {
                const int j = midx(n - k, k - cc, cc);
                real v = acc[j] * static_cast<real>(inv_mfact(n - k, k - cc, cc));
                v += __shfl_xor_sync(0xffffffffu, v, 1);
                v += __shfl_xor_sync(0xffffffffu, v, 2);
                if (valid && (j & 3) == q) Mh[(size_t)c * NM + j] = v;
            }
    }
}

// M2M of a parent from its children, as three one-dimensional shifts per
// child (the expansion of (d_c + delta)^beta / beta! factorises over the
// axes): the child's moments scaled by r^|gamma| go into full storage with
// zero dipole slots, are shifted along x, y and z by delta, and the slots of
// orders 0 and 2..P-1 are summed over the children in child order (the
// parent's dipole about its own centre of mass vanishes).  The children are
// shifted side by side: four lanes per child (a parent has at most eight),
// each lane a quarter of the child's slots.
template <int P, typename real>
__device__ __forceinline__ void parent_moments(const P2MArgs &A, M2MShared<P, real> &S, int wl, int pc, int lane,
                                               real *Mh) {
    constexpr int NM = num_m(P), NF = off(P);
    constexpr int PER4 = (NF + 3) / 4;   // slots per lane of a child's quad
    const int ch = lane >> 2, sub = lane & 3;
    const int c0 = A.child0[pc], nch = A.nchild[pc];
    const bool act = ch < nch;
    const int c = act ? c0 + ch : c0;
    real ipr, dx, dy, dz, rr;
    if constexpr (sizeof(real) == 4) {
        const float4 ch_h = A.gh[c], ch_l = A.gl[c], p_h = A.gh[pc], p_l = A.gl[pc];
        ipr = 1.0f / p_l.w;   // exact: rho is a power of two
        dx = ((ch_h.x - p_h.x) + (ch_l.x - p_l.x)) * ipr;
        dy = ((ch_h.y - p_h.y) + (ch_l.y - p_l.y)) * ipr;
        dz = ((ch_h.z - p_h.z) + (ch_l.z - p_l.z)) * ipr;
        rr = ch_l.w * ipr;
    } else {
        ipr = 1.0 / A.rho[pc];
        dx = (A.sx[c] - A.sx[pc]) * ipr;
        dy = (A.sy[c] - A.sy[pc]) * ipr;
        dz = (A.sz[c] - A.sz[pc]) * ipr;
        rr = A.rho[c] * ipr;
    }
    real wx[P], wy[P], wz[P];
    wx[0] = wy[0] = wz[0] = real(1);
#pragma unroll
    for (int k = 1; k < P; k++) {
        wx[k] = wx[k - 1] * dx;
        wy[k] = wy[k - 1] * dy;
        wz[k] = wz[k - 1] * dz;
    }
#pragma unroll
    for (int k = 2; k < P; k++) {
        const real f = static_cast<real>(ifact(k));
        wx[k] *= f; wy[k] *= f; wz[k] *= f;
    }
    int en[PER4], ek[PER4], ec[PER4];
#pragma unroll
    for (int q = 0; q < PER4; q++) full_exps<P>(sub + 4 * q, en[q], ek[q], ec[q]);
    real *sa = S.a[wl][ch], *sb = S.b[wl][ch];
    __syncwarp();
    if (act) {
#pragma unroll
        for (int q = 0; q < PER4; q++) {   // the child's moments, scaled by r^n, dipole slots zero
            const int j = sub + 4 * q;
            if (j >= NF) continue;
            real v = real(0);
            if (en[q] != 1) {
                v = __ldcg(&Mh[(size_t)c * NM + (en[q] == 0 ? 0 : j - 3)]);
                for (int t = 0; t < en[q]; t++) v *= rr;
            }
            sa[j] = v;
        }
    }
    __syncwarp();
    if (act) {
#pragma unroll
        for (int q = 0; q < PER4; q++)
            if (sub + 4 * q < NF) sb[sub + 4 * q] = m_shift<P, 0>(sa, wx, en[q], ek[q], ec[q]);
    }
    __syncwarp();
    if (act) {
#pragma unroll
        for (int q = 0; q < PER4; q++)
            if (sub + 4 * q < NF) sa[sub + 4 * q] = m_shift<P, 1>(sb, wy, en[q], ek[q], ec[q]);
    }
    __syncwarp();
    if (act) {
#pragma unroll
        for (int q = 0; q < PER4; q++)
            if (sub + 4 * q < NF) sb[sub + 4 * q] = m_shift<P, 2>(sa, wz, en[q], ek[q], ec[q]);
    }
    __syncwarp();
    // sums over the children in child order; lane j takes slots j, j + 32
    for (int j = lane; j < NF; j += 32) {
        int n, kk, cc;
        full_exps<P>(j, n, kk, cc);
        if (n == 1) continue;
        real acc = real(0);
        for (int k = 0; k < nch; k++) acc += S.b[wl][k][j];
        Mh[(size_t)pc * NM + (n == 0 ? 0 : j - 3)] = acc;
    }
}

// One launch, no waiting: the leaves' moments from their moonlets (eight
// leaves per warp), then the parents up the tree.  A warp that has finished a
// cell adds its arrival to the parent's counter (release); the warp that
// arrives last (acquire) computes the parent, whose children are then all
// done, and goes on up.  The children are added in child order, so the
// result does not depend on which warp arrives last.
template <int P, typename real>
__device__ __forceinline__ int arrive_last(const P2MArgs &A, int c) {
    const int pc = A.parent[c];
    if (pc < 0) return -1;
    fence_acq_rel_gpu();   // release: the cell's moments before the arrival
    if (atomicAdd(&A.arrive[pc], 1) != A.nchild[pc] - 1) return -1;
    fence_acq_rel_gpu();   // acquire: the other children's moments
    return pc;
}

template <int P, typename real>
__global__ void __launch_bounds__(32 * P2M_WARPS) k_multipoles(P2MArgs A) {
    __shared__ M2MShared<P, real> S;
    if (aborted(A.ctl)) return;
    const int lane = threadIdx.x & 31, wl = threadIdx.x >> 5;
    const int gw0 = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, nwarps = (gridDim.x * blockDim.x) >> 5;
    const int nl = A.ctl->n_leaves;
    real *Mh = static_cast<real *>(A.Mh);
    for (int base = gw0 * 8; base < nl; base += nwarps * 8) {   // eight leaves per warp, four lanes each
        const int li = base + (lane >> 2);
        const bool valid = li < nl;
        const int c = valid ? A.leaves[li] : 0;
        leaf_moments<P, real>(A, c, valid, lane & 3, Mh);
        __syncwarp();
        int up = -1;   // the parent this quad's leaf completed, if any
        if (valid && (lane & 3) == 0) up = arrive_last<P, real>(A, c);
        unsigned todo = __ballot_sync(0xffffffffu, up >= 0);
        while (todo) {
            const int src = __ffs(todo) - 1;
            todo &= todo - 1;
            int pc = __shfl_sync(0xffffffffu, up, src);
            __syncwarp();   // orders the quad leader's acquire before every lane's reads
            while (true) {
                parent_moments<P, real>(A, S, wl, pc, lane, Mh);
                __syncwarp();
                int next = -1;
                if (lane == 0) next = arrive_last<P, real>(A, pc);
                next = __shfl_sync(0xffffffffu, next, 0);
                if (next < 0) break;
                __syncwarp();
                pc = next;
            }
        }
    }
}

template <int P, typename real>
static void p2m_t(ncorp_ctx *c, const P2MArgs &B) {
    k_multipoles<P, real><<<4 * c->num_sms, 32 * P2M_WARPS, 0, c->stream>>>(B); c->launches++;
}

// theta(M) of Dehnen (2002) Eq. 13: theta^5/(1-theta)^2 = K (M/M_tot)^(-1/3),
// K = theta_min^5/(1-theta_min)^2, i.e. the root in [theta_min, 1) of the
// increasing f(theta) = theta^15 M - K^3 M_tot (1-theta)^6: 12 bisection
// steps, then 4 Newton steps kept inside the final bracket (+ - x / only).
// K3 = K^3, rhs = K^3 M_tot in FP64; tmin > 0.
// A bisection step only needs the sign of f, so it is taken from FP32 values
// of the two terms when they differ by more than their error (theta and its
// complement cut to FP32: 2^-23 each, 15 and 6 powers, the roundings of the
// products: below 2^-18 + 2^-20 / (1 - theta) together), else from FP64: one
// FP64 instruction a step in place of fourteen.
__device__ double theta_of(double M, double rhs, double tmin) {
    double lo = tmin, hi = 1.0;
    const float Mf = static_cast<float>(M), rf = static_cast<float>(rhs);
    const bool small = !(Mf > 1e-15f && Mf < 1e15f && rf > 1e-15f && rf < 1e15f);   // (products may leave the FP32 range)
#pragma unroll 1
    for (int it = 0; it < 12; it++) {
        const double sum = dadd(lo, hi);   // in (0, 2): halved exactly by its exponent
        const double mid = __longlong_as_double(__double_as_longlong(sum) - (1ll << 52));
        // mid in FP32 (cut): 0 < mid < 1
        const unsigned mh = static_cast<unsigned>(__double2hiint(mid)), ml = static_cast<unsigned>(__double2loint(mid));
        const float t = (mh >> 20) > 900u ? __uint_as_float(((mh - (896u << 20)) << 3) | (ml >> 29)) : 0.f;
        const float w = 1.0f - t;
        const float t2 = t * t, t3 = t2 * t, t6 = t3 * t3, t12 = t6 * t6, w2 = w * w, w4 = w2 * w2;
        const float a = t12 * t3 * Mf, c = w4 * w2 * rf;
        const float margin = (0x1p-17f + 0x1p-19f / w) * fmaxf(a, c);
        bool up;   // f > 0
        if (small || !(t12 > 1e-15f && w4 > 1e-12f) || !(fabsf(a - c) > margin)) {
            const double m2 = dmul(mid, mid), m3 = dmul(m2, mid), m6 = dmul(m3, m3), m12 = dmul(m6, m6),
                         m15 = dmul(m12, m3);
            const double v = dsub(1.0, mid), v2 = dmul(v, v), v3 = dmul(v2, v), v6 = dmul(v3, v3);
            up = dsub(dmul(m15, M), dmul(rhs, v6)) > 0.0;
        } else {
            up = a > c;
        }
        if (up) hi = mid;
        else lo = mid;
    }
    double th = dmul(dadd(lo, hi), 0.5);
    const double rhs6 = dmul(6.0, rhs);
    for (int it = 0; it < 4; it++) {
        const double w = dsub(1.0, th);
        const double q2 = dmul(th, th), q3 = dmul(q2, th), q6 = dmul(q3, q3), q12 = dmul(q6, q6),
                     q14 = dmul(q12, q2), q15 = dmul(q14, th);
        const double w2 = dmul(w, w), w3 = dmul(w2, w), w5 = dmul(w3, w2), w6 = dmul(w3, w3);
        const double f = dsub(dmul(q15, M), dmul(rhs, w6));
        const double fp = dadd(dmul(dmul(15.0, q14), M), dmul(rhs6, w5));
        double nt = dsub(th, ddiv(f, fp));
        if (__double_as_longlong(nt) < __double_as_longlong(lo)) nt = lo;   // (lo > 0: a negative nt too)
        if (less_nn(hi, nt)) nt = hi;
        th = nt;
    }
    return th;
}

// ---- gravity geometry in one cooperative launch: the leaves, then the
// parents level by level from the deepest (each needs its children's), then
// theta(M) and r_crit = r_max / theta (which need the root's mass).  One FP64
// warp instruction costs the same whatever the number of active lanes, so the
// leaves go eight to a warp with four lanes each, theta(M) 32 cells to a
// warp, and the parents four to a warp with eight lanes each.
__global__ void __launch_bounds__(32 * CLIMB_WARPS_COOP) k_geometry(ClimbArgs A) {
    if (aborted(A.ctl)) return;
    const int lane = threadIdx.x & 31;
    // warps numbered across the blocks first, so that consecutive work items land on different SMs
    const int gw0 = (threadIdx.x >> 5) * gridDim.x + blockIdx.x, nwarps = (gridDim.x * blockDim.x) >> 5;
    unsigned bar = 0;
    if (blockIdx.x == 0) walk_start(A.ws, A.ctl);
    const int n_leaves = A.ctl->n_leaves;
    for (int gw = gw0; gw * LEAF_GROUP < n_leaves; gw += nwarps) leaf_gravity_group(A, gw, lane, n_leaves);
    if (!grid_sync(A.ctl, bar)) return;
    const int maxl = A.ctl->max_level;
    for (int lev = maxl - 1; lev >= 0; lev--) {
        const int ls = A.ctl->level_start[lev], le = A.ctl->level_start[lev + 1];
        for (int g = gw0; ls + g * PARENT_GROUP < le; g += nwarps) {
            const int cc = ls + g * PARENT_GROUP + (lane >> 3);
            const int c = (cc < le && A.nchild[cc] > 0) ? cc : -1;
            if (__any_sync(0xffffffffu, c >= 0)) parent_gravity_group(A, c, lane);
        }
        if (!grid_sync(A.ctl, bar)) return;
    }
    const int nc = min(A.ctl->n_cells, A.cap);
    // theta(M): every lane one cell; the dependent FP64 chain of a warp bounds this phase, so fewer,
    // fuller warps (at most one per sub-partition) finish first.  M_tot is the mass of the cell's disk
    // (its root: cell d of disk d).
    {
        for (int i = gw0 * 32 + lane; i < nc; i += nwarps * 32) {
            const double Mtot = __ldcg(&A.M[disk_of(A.ctl, A.first[i])]);
            const double rc = ddiv(__ldcg(&A.rmax[i]), theta_of(__ldcg(&A.M[i]), dmul(A.K3, Mtot), A.theta));
            A.rcrit[i] = rc;
            A.gh[i].w = static_cast<float>(rc);
        }
    }
}


void launch_climb_geometry(ncorp_ctx *c, const ParticleSet &P, double G, double theta, int walk) {
    Cells &C = c->cells;
    ClimbArgs A{};
    A.x = P.x; A.y = P.y; A.z = P.z; A.m = P.m; A.hi4 = P.hi4; A.lo4 = P.lo4;
    A.first = C.first; A.count = C.count; A.child0 = C.child0; A.nchild = C.nchild; A.parent = C.parent;
    A.level = C.level; A.cx = C.cx; A.cy = C.cy; A.cz = C.cz;
    A.M = C.M; A.sx = C.sx; A.sy = C.sy; A.sz = C.sz; A.rmax = C.rmax; A.rcrit = C.rcrit; A.rho = C.rho;
    A.gh = C.gh; A.gl = C.gl;
    A.Mh = C.Mh; A.leaves = C.leaves; A.ctl = c->ctl; A.G = G; A.theta = theta; A.cap = C.cap;
    if (walk) {
        A.ws.fcount = c->wl.front_count;
        A.ws.work = c->work_counter;
        A.ws.gravity = 1;
        A.ws.collisions = walk == 2;
    }
    {   // K^3, each operation rounded once as on the device (no contraction: products and quotients only)
        const double t2 = theta * theta, t4 = t2 * t2, t5 = t4 * theta, u = 1.0 - theta, u2 = u * u, K = t5 / u2;
        const double K2 = K * K;
        A.K3 = K2 * K;
    }
    const int block = 32 * CLIMB_WARPS_COOP;
    // every SM: the FP64 work of the leaves and of theta(M) is bound by the FP64 units of the
    // sub-partitions, so it is spread over all of them
    const int grid = coop_grid(c, reinterpret_cast<const void *>(k_geometry), block, 0);
    void *args[] = {&A};   // ctl->bar_count was zeroed by k_build
    NCORP_CUDA_CHECK(cudaLaunchCooperativeKernel(reinterpret_cast<const void *>(k_geometry), dim3(grid), dim3(block),
                                                 args, 0, c->stream));
    c->launches++;
}

void launch_multipoles(ncorp_ctx *c, const ParticleSet &P, int p, bool mixed, double G) {
    Cells &C = c->cells;
    P2MArgs B;
    B.x = P.x; B.y = P.y; B.z = P.z; B.m = P.m; B.hi4 = P.hi4; B.lo4 = P.lo4;
    B.first = C.first; B.count = C.count; B.child0 = C.child0; B.nchild = C.nchild; B.parent = C.parent;
    B.leaves = C.leaves; B.arrive = C.arrive_m;
    B.sx = C.sx; B.sy = C.sy; B.sz = C.sz; B.rho = C.rho; B.gh = C.gh; B.gl = C.gl;
    B.Mh = C.Mh;
    B.G = G; B.ctl = c->ctl;
#define NCORP_P2M_CASE(PP)                     \
    case PP:                                   \
        if (mixed) p2m_t<PP, float>(c, B);     \
        else p2m_t<PP, double>(c, B);          \
        break;
    switch (p) {
        NCORP_P2M_CASE(1)
        NCORP_P2M_CASE(2)
        NCORP_P2M_CASE(3)
        NCORP_P2M_CASE(4)
        NCORP_P2M_CASE(5)
        NCORP_P2M_CASE(6)
        default: break;
    }
#undef NCORP_P2M_CASE
    NCORP_CUDA_CHECK(cudaGetLastError());
}

// FP64 value cut to FP32 in integers (relative error below 2^-23; beyond the FP32 range: 0, infinity; NaN stays NaN)
__device__ __forceinline__ float cut_f32(double v) {
    const unsigned h = static_cast<unsigned>(__double2hiint(v)), l = static_cast<unsigned>(__double2loint(v));
    const int ex = static_cast<int>((h >> 20) & 0x7ff) - 896;
    const unsigned sign = h & 0x80000000u;
    if (ex <= 0) return __uint_as_float(sign);
    if (ex >= 255) return (ex == 0x7ff - 896 && ((h & 0xfffffu) | l)) ? __uint_as_float(0x7fffffffu) : __uint_as_float(sign | 0x7f800000u);
    return __uint_as_float(sign | (static_cast<unsigned>(ex) << 23) | ((h & 0xfffffu) << 3) | (l >> 29));
}

// ---------------------------------------------------------------------------
// Collision climb (Eqs. center, rmax, rcrit): s-bar is the mean moonlet
// position (children weighted by their moonlet counts); r_crit = r_max + max
// over children of (r_crit - r_max), a moonlet's being R + dt |v| (stored,
// as an FP32 upper bound, with the velocity in FP32, for the pair
// prefilter).
// ---------------------------------------------------------------------------
// One block per SM, two of which leave the main stream's key sort its room: it
// needs a block on every SM at once (blocks of 64 threads, up to sixteen on an
// SM that other kernels had left free, held it back 19 us at N = 1e5).
constexpr int LEAF_COL_T = 384;
__global__ void __launch_bounds__(LEAF_COL_T) k_leaf_collision(ClimbArgs A) {
    if (A.gate && *A.gate == 0) return;
    // the grid barrier counter of the parents' cooperative climb that follows on this stream
    if (blockIdx.x == 0 && threadIdx.x == 0) A.ctl->bar_count2 = 0;
    if (aborted(A.ctl)) return;
    if (blockIdx.x == 0) walk_start(A.ws, A.ctl);
    const int lane = threadIdx.x & 31;
    const int n_leaves = A.ctl->n_leaves;
    const int nwarps = (gridDim.x * blockDim.x) >> 5;
    const float dtf = static_cast<float>(A.dt);
    for (int gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; gw * LEAF_GROUP < n_leaves; gw += nwarps) {
        const LeafSlot L = leaf_slot(A, gw, lane, n_leaves);
        const double *coord = L.q == 0 ? A.x : (L.q == 1 ? A.y : A.z);
        double acc = 0.0;
#pragma unroll 4
        for (int k = L.f; k < L.f + L.cnt; k++) acc = dadd(acc, coord[k]);
        const double sq = ddiv(acc, static_cast<double>(L.valid ? L.cnt : 1));
        const double sx = __shfl_sync(0xffffffffu, sq, L.base), sy = __shfl_sync(0xffffffffu, sq, L.base + 1),
                     sz = __shfl_sync(0xffffffffu, sq, L.base + 2);
        float h1, l1;
        split1(sq, h1, l1);
        float4 hi, lo;
        gather_split(h1, l1, L.base, hi, lo);
        const double d2 = leaf_dist2(A, L, sx, sy, sz, hi, lo);
        // the largest R + dt |v|: estimated in FP32 like the distances; the estimate's upper bound goes to the
        // pair test, which needs R + dt |v| from above
        double ex = 0.0;
        if (A.rc_given) {   // bounds given: the pair test's per-moonlet values come later
            for (int k = L.f + L.q; k < L.f + L.cnt; k += 4) ex = max_nn(ex, A.rc_given[k]);
        } else {
            LeafMax E;
            for (int k = L.f + L.q; k < L.f + L.cnt; k += 4) {
                const float vx = cut_f32(A.vx[k]), vy = cut_f32(A.vy[k]), vz = cut_f32(A.vz[k]), r = cut_f32(A.R[k]);
                const float v2 = vx * vx + vy * vy + vz * vz;
                float e, up;
                if (r >= 0.f && v2 > 1e-30f && v2 < 1e30f) {
                    e = r + dtf * sqrtf(v2);
                    up = e * (1.0f + 0x1p-19f);
                } else {   // at rest, a negative radius, or speeds whose squares leave the FP32 range
                    const double x = dadd(A.R[k], dmul(A.dt, dnorm3(A.vx[k], A.vy[k], A.vz[k])));
                    e = static_cast<float>(x);
                    up = __double2float_ru(x);
                }
                E.add(e, k);
                A.cv4[k] = make_float4(vx, vy, vz, up);
            }
            if (E.settle(1e-35f, L.base)) {
                const int k = E.at;
                if (k >= 0) ex = dadd(A.R[k], dmul(A.dt, dnorm3(A.vx[k], A.vy[k], A.vz[k])));
            } else {
                for (int k = L.f + L.q; k < L.f + L.cnt; k += 4)
                    ex = max_nn(ex, dadd(A.R[k], dmul(A.dt, dnorm3(A.vx[k], A.vy[k], A.vz[k]))));
            }
            __syncwarp();
        }
        ex = quad_max(max_nn(0.0, ex));
        double rmax = dsqrt(d2);
        const double cap = quad_corner(A, L, sx, sy, sz);
        if (less_nn(cap, rmax)) rmax = cap;
        if (L.valid && L.q == 0) {
            const int c = L.c;
            const double rc = dadd(rmax, ex);
            A.sx[c] = sx;
            A.sy[c] = sy;
            A.sz[c] = sz;
            A.rmax[c] = rmax;
            A.rcrit[c] = rc;
            hi.w = static_cast<float>(rc);
            A.gh[c] = hi;
            A.gl[c] = lo;
        }
    }
}

// ---- collision geometry of parents from their children (Eqs. center, rmax,
// rcrit, corner cap), four parents per warp, eight lanes each, as for gravity
// (parent_gravity_group) with the children's moonlet counts as weights and
// the parent's count as divisor; r_crit = r_max + the largest (r_crit - r_max)
// of the children.  c is the group's parent, -1 for none; every lane of the
// warp calls this.
__device__ __forceinline__ void parent_collision_group(const ClimbArgs &A, int c, int lane) {
    const int j = lane & 7, base = lane & ~7;
    const bool valid = c >= 0;
    const int c0 = valid ? A.child0[c] : 0, nch = valid ? A.nchild[c] : 0;
    double cw = 0.0, csx = 0.0, csy = 0.0, csz = 0.0, crm = 0.0, cex = 0.0;
    if (j < nch) {
        cw = static_cast<double>(A.count[c0 + j]);
        csx = __ldcg(&A.sx[c0 + j]);
        csy = __ldcg(&A.sy[c0 + j]);
        csz = __ldcg(&A.sz[c0 + j]);
        crm = __ldcg(&A.rmax[c0 + j]);
        cex = dsub(__ldcg(&A.rcrit[c0 + j]), crm);
    }
    const double acc = children_sum(cw, csx, csy, csz, nch, j, base);
    const double q = ddiv(acc, valid ? static_cast<double>(A.count[c]) : 1.0);
    const double px = __shfl_sync(0xffffffffu, q, base + 1), py = __shfl_sync(0xffffffffu, q, base + 2),
                 pz = __shfl_sync(0xffffffffu, q, base + 3);
    double rm = 0.0;
    if (j < nch) rm = dadd(crm, dnorm3(dsub(csx, px), dsub(csy, py), dsub(csz, pz)));
    rm = max_nn(0.0, rm);
    cex = max_nn(0.0, cex);
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) {
        rm = max_nn(rm, __shfl_xor_sync(0xffffffffu, rm, o));
        cex = max_nn(cex, __shfl_xor_sync(0xffffffffu, cex, o));
    }
    float h1, l1;
    split1(q, h1, l1);
    float4 hi, lo;
    gather_split(h1, l1, base + 1, hi, lo);
    double d = 0.0;
    if (valid && j < 3) {
        const double *rt = cell_root(A.ctl, A.first, c);
        const double h = cell_side(rt, A.level[c]);
        d = corner_axis(rt, j, h, j == 0 ? A.cx[c] : (j == 1 ? A.cy[c] : A.cz[c]), j == 0 ? px : (j == 1 ? py : pz));
    }
    const double d0 = __shfl_sync(0xffffffffu, d, base), d1 = __shfl_sync(0xffffffffu, d, base + 1),
                 d2 = __shfl_sync(0xffffffffu, d, base + 2);
    const double pcap = dnorm3(d0, d1, d2);
    if (less_nn(pcap, rm)) rm = pcap;
    if (valid && j == 0) {
        const double rc = dadd(rm, cex);
        A.sx[c] = px;
        A.sy[c] = py;
        A.sz[c] = pz;
        A.rmax[c] = rm;
        A.rcrit[c] = rc;
        hi.w = static_cast<float>(rc);
        A.gh[c] = hi;
        A.gl[c] = lo;
    }
}

// The parents, level by level from the deepest, in one cooperative launch
// (the leaves were done by k_leaf_collision, which also zeroed the barrier
// counter).  Four parents per warp, so that one FP64 warp instruction
// advances four parents.
__global__ void __launch_bounds__(32 * CLIMB_WARPS_COOP) k_climb_collision(ClimbArgs A) {
    if ((A.gate && *A.gate == 0) || aborted(A.ctl)) return;
    const int lane = threadIdx.x & 31;
    // warps numbered across the blocks first, so that consecutive work items land on different SMs
    const int gw0 = (threadIdx.x >> 5) * gridDim.x + blockIdx.x, nwarps = (gridDim.x * blockDim.x) >> 5;
    unsigned bar = 0;
    const int maxl = A.ctl->max_level;
    for (int lev = maxl - 1; lev >= 0; lev--) {
        const int ls = A.ctl->level_start[lev], le = A.ctl->level_start[lev + 1];
        for (int g = gw0; ls + g * PARENT_GROUP < le; g += nwarps) {
            const int cc = ls + g * PARENT_GROUP + (lane >> 3);
            const int c = (cc < le && A.nchild[cc] > 0) ? cc : -1;
            if (__any_sync(0xffffffffu, c >= 0)) parent_collision_group(A, c, lane);
        }
        if (lev > 0 && !grid_sync_on(&A.ctl->bar_count2, A.ctl, bar)) return;
    }
}

void launch_climb_collision(ncorp_ctx *c, const ParticleSet &P, const double *vx, const double *vy,
                            const double *vz, double dt, bool walk, const double *rc_given, const int *gate) {
    Cells &C = c->cells;
    ClimbArgs A{};
    A.x = P.x; A.y = P.y; A.z = P.z; A.R = P.R; A.vx = vx; A.vy = vy; A.vz = vz;
    A.hi4 = P.hi4; A.lo4 = P.lo4;
    A.first = C.first; A.count = C.count; A.child0 = C.child0; A.nchild = C.nchild; A.parent = C.parent;
    A.level = C.level; A.cx = C.cx; A.cy = C.cy; A.cz = C.cz;
    A.sx = C.bx; A.sy = C.by; A.sz = C.bz; A.rmax = C.bmax; A.rcrit = C.bcrit;
    A.gh = C.bh; A.gl = C.bl;
    A.leaves = C.leaves; A.ctl = c->ctl; A.dt = dt; A.cv4 = c->cv4;
    if (walk) {
        A.ws.fcount = c->wl.front_count;
        A.ws.collisions = 1;
    }
    A.rc_given = rc_given;
    A.gate = gate;
    k_leaf_collision<<<c->num_sms, LEAF_COL_T, 0, c->stream>>>(A); c->launches++;
    NCORP_CUDA_CHECK(cudaGetLastError());
    const int block = 32 * CLIMB_WARPS_COOP;
    const int grid = coop_grid(c, reinterpret_cast<const void *>(k_climb_collision), block, 0);
    void *args[] = {&A};   // ctl->bar_count2 was zeroed by k_leaf_collision
    NCORP_CUDA_CHECK(cudaLaunchCooperativeKernel(reinterpret_cast<const void *>(k_climb_collision), dim3(grid),
                                                 dim3(block), args, 0, c->stream));
    c->launches++;
}

}  // namespace ncorp
