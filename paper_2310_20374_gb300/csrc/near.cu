// near.cu -- near field: the direct ("brute force") gravity of each leaf's
// direct list.  Every moonlet gets
//   sum_j mu_j (x_j - x)/|x_j - x|^3 over the moonlets of its leaf's direct list
// (mu_j = G m_j; coincident pairs, the moonlet itself included, are skipped),
// left in (nx, ny, nz) for the evaluation kernel (eval.cu), which adds the far
// field and the external forces.  The lists are all it needs, so it runs while
// M2L and the descent produce the local expansions.
//
// Mixed precision: positions are read as FP32 pairs (hi, lo) with x = hi + lo;
// (hi_j - hi_i) + (lo_j - lo_i) gives the separation to ~1e-7 relative at any
// distance, so no FP64 work is done per pair.
#include <algorithm>

#include "ctx.h"
#include "fields.cuh"

namespace ncorp {

struct NearArgs {
    const int4 *items;        // (first moonlet of the leaf, its moonlets, first and end of the item's direct entries)
    const int2 *p2p_src;      // per directed entry: the source leaf's (first, count)
    int item_cap;
    const double *x, *y, *z, *m;
    const float4 *hi4, *lo4;
    double G;
    double *nx, *ny, *nz;     // near-field sums per moonlet (tree order), zeroed by the gather
    int *work;                // items handed out so far (zeroed by the geometry climb)
    const Ctrl *ctl;
};

constexpr int NEAR_THREADS = 128, NEAR_WARPS = NEAR_THREADS / 32;

// The direct list of a leaf as one sequence of source moonlets, taken in
// windows of 32 entries (source leaves), each warp holding the whole window:
// lane l its entry's first moonlet and the number of moonlets before it, so
// that every warp maps a place in the window to a moonlet with shuffles alone.
struct NearWindow {
    int first, before;   // this lane's entry
    int total;           // moonlets of the window
    __device__ __forceinline__ void load(const int2 *src, int at, int end, int lane) {
        set(at + lane < end ? __ldg(&src[at + lane]) : make_int2(0, 0), lane);
    }
    __device__ __forceinline__ void set(int2 e, int lane) {
        int incl = e.y;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += v;
        }
        first = e.x;
        before = incl - e.y;
        total = __shfl_sync(0xffffffffu, incl, 31);
    }
    // moonlet at place pos + lane of the window, -1 past its end (every lane of the warp calls this): the
    // entries that begin among the 32 places are marked in a word, and a place's entry is found by counting
    __device__ __forceinline__ int moonlet(int pos, int lane) const {
        const int d = before - pos;
        const unsigned starts = __reduce_or_sync(0xffffffffu, d >= 0 && d < 32 ? 1u << d : 0u);
        const int earlier = __popc(__ballot_sync(0xffffffffu, d < 0));
        const int q = earlier + __popc(starts & (0xffffffffu >> (31 - lane))) - 1;
        const int f = __shfl_sync(0xffffffffu, first, q), s = __shfl_sync(0xffffffffu, before, q);
        return pos + lane < total ? f + pos + lane - s : -1;
    }
};

// An item of the list the walk made: a leaf's moonlets and a share of its
// direct entries.  A leaf whose list is one item (count > 0) gets its sums
// stored; the shares of a split list (count < 0) add up with FP64 atomics in
// sums that the gather zeroed.
struct NearItem {
    int first, count, s0, s1;
    bool whole;
    __device__ __forceinline__ explicit NearItem(int4 v)
        : first(v.x), count(abs(v.y)), s0(v.z), s1(v.w), whole(v.y > 0) {}
};

__device__ __forceinline__ void near_store(const NearArgs &A, int i, bool whole, double x, double y, double z) {
    if (whole) {
        A.nx[i] = x;
        A.ny[i] = y;
        A.nz[i] = z;
    } else {
        atomicAdd(&A.nx[i], x);
        atomicAdd(&A.ny[i], y);
        atomicAdd(&A.nz[i], z);
    }
}

// ---------------------------------------------------------------------------
// Mixed precision.  The items (a leaf and a share of its direct list, of about
// equal cost: near_targets and near_shares in ctx.h) are handed out to the warps one by one.  A
// warp works alone: it stages sources into its own part of shared memory, and
// no block barrier separates the chunks (with a block of 128 threads per leaf,
// two barriers a chunk and five a leaf cost a quarter of the warps' time).  The
// item's m targets (at most 64) are taken two per lane by
// G = floor(32 / ceil(m / 2)) groups of ceil(m / 2) lanes: lane (g, t) sums for
// its targets every G-th quad of the staged sources.
//
// Bound by the FP32 pipe.  The pair takes 21 FP32 operations (9 for the
// double-float separation, 3 for r^2, 6 for mu r^-3 with the corrected
// reciprocal square root, 3 to add), one MUFU and one maximum.  As scalar code
// it issued 41 instructions a pair (operations, two 16-byte loads, loop) and
// the issue slots were the limit (69 % busy at 24 warps per SM).  Here the
// sources are staged by component, so that one 16-byte load brings four
// sources' values of a component, and the arithmetic is done on two sources at
// a time with Blackwell's packed FP32 instructions (fma.rn.f32x2: two
// operations per issue slot, the same rounding as the scalar ones): 15 issue
// slots a pair, below the pipe's 21 cycles.  The next chunk's positions are
// loaded into registers before the current chunk is summed.  Measured alone:
// 207 -> 161 us at N = 1e5, p = 6 (as captured, caches cold: 163 us, 60 % of the
// issue slots and 59 % of the FP32 pipe busy, 28.5 lanes an instruction, four
// blocks per SM), 740 us at N = 1e6, p = 4.
//
// Every lane adds its FP32 partial sums (two running sums, one per half of
// the packed registers, of at most 32 terms each) to double-float totals
// (two-sum), and the halves' and the groups' totals are added in a fixed
// order, so that the rounding of a long FP32 running sum (dominated by the
// nearest pull) does not grow with the direct list.
// ---------------------------------------------------------------------------
using f32x2 = unsigned long long;   // two FP32 values in a register pair

__device__ __forceinline__ f32x2 pack2(float a, float b) {
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void unpack2(f32x2 v, float &a, float &b) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
    f32x2 r;
    asm("add.rn.ftz.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
    f32x2 r;
    asm("mul.rn.ftz.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
    f32x2 r;
    asm("fma.rn.ftz.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

// p2p_f32 (fields.cuh) for two sources and one target, whose negated position
// is given in both halves
struct Target2 {
    f32x2 hx, hy, hz, lx, ly, lz;
};
__device__ __forceinline__ void p2p_f32x2(f32x2 hx, f32x2 hy, f32x2 hz, f32x2 mu, f32x2 lx, f32x2 ly, f32x2 lz,
                                          const Target2 &T, f32x2 &ax, f32x2 &ay, f32x2 &az) {
    const f32x2 dx = add2(add2(hx, T.hx), add2(lx, T.lx));
    const f32x2 dy = add2(add2(hy, T.hy), add2(ly, T.ly));
    const f32x2 dz = add2(add2(hz, T.hz), add2(lz, T.lz));
    float ra, rb;
    unpack2(fma2(dz, dz, fma2(dx, dx, mul2(dy, dy))), ra, rb);
    ra = fmaxf(ra, 1e-20f);   // (see p2p_f32)
    rb = fmaxf(rb, 1e-20f);
    const f32x2 r2 = pack2(ra, rb), y = pack2(rsqrtf(ra), rsqrtf(rb));
    const f32x2 y2 = mul2(y, y);
    const f32x2 e = fma2(r2, y2, pack2(-1.0f, -1.0f));          // -(1 - r^2 y^2)
    const f32x2 f = mul2(mu, mul2(y2, y));
    const f32x2 f3 = fma2(f, mul2(e, pack2(-1.5f, -1.5f)), f);
    ax = fma2(dx, f3, ax);
    ay = fma2(dy, f3, ay);
    az = fma2(dz, f3, az);
}

constexpr int NEAR_CHUNK = 64;   // sources a warp stages at a time

__global__ void __launch_bounds__(NEAR_THREADS, 4) k_near_f32(NearArgs A) {
    // hi x, y, z, mu, lo x, y, z of the warp's staged sources
    __shared__ __align__(16) float s_src[NEAR_WARPS][7][NEAR_CHUNK];
    if (aborted(A.ctl)) return;
    const int lane = threadIdx.x & 31;
    float(*S)[NEAR_CHUNK] = s_src[threadIdx.x >> 5];
    const int n_items = min(A.ctl->n_near, A.item_cap);
    int li = lane == 0 ? atomicAdd(A.work, 1) : 0;
    li = __shfl_sync(0xffffffffu, li, 0);
    int4 item = li < n_items ? __ldg(&A.items[li]) : make_int4(0, 0, 0, 0);
    while (li < n_items) {
        const NearItem I(item);
        // the next item: its number and description arrive while this one is summed
        int next = lane == 0 ? atomicAdd(A.work, 1) : 0;
        bool asked = false;
        const int m = I.count, L = (m + 1) >> 1;   // at most 64 targets
        const int G = 32 / L, g = lane / L, tt = lane - g * L;
        const bool act = g < G;   // the last 32 - G L lanes only help with staging
        const int i0 = I.first + (act ? 2 * tt : 0), i1 = min(i0 + 1, I.first + m - 1);
        const float4 th0 = A.hi4[i0], tl0 = A.lo4[i0], th1 = A.hi4[i1], tl1 = A.lo4[i1];
        const Target2 T0 = {pack2(-th0.x, -th0.x), pack2(-th0.y, -th0.y), pack2(-th0.z, -th0.z),
                            pack2(-tl0.x, -tl0.x), pack2(-tl0.y, -tl0.y), pack2(-tl0.z, -tl0.z)};
        const Target2 T1 = {pack2(-th1.x, -th1.x), pack2(-th1.y, -th1.y), pack2(-th1.z, -th1.z),
                            pack2(-tl1.x, -tl1.x), pack2(-tl1.y, -tl1.y), pack2(-tl1.z, -tl1.z)};
        f32x2 a0[3] = {0, 0, 0}, a1[3] = {0, 0, 0};
        float h0[3] = {0.f, 0.f, 0.f}, l0[3] = {0.f, 0.f, 0.f}, h1[3] = {0.f, 0.f, 0.f}, l1[3] = {0.f, 0.f, 0.f};
        const int rounds = (NEAR_CHUNK / 4 + G - 1) / G;   // most quads of a chunk per lane
        int since = 0;                                     // quads since the running sums were folded
        auto fold = [&]() {
#pragma unroll
            for (int d = 0; d < 3; d++) {
                float p, q;
                unpack2(a0[d], p, q);
                df_add(h0[d], l0[d], p);
                df_add(h0[d], l0[d], q);
                unpack2(a1[d], p, q);
                df_add(h1[d], l1[d], p);
                df_add(h1[d], l1[d], q);
                a0[d] = a1[d] = 0;
            }
            since = 0;
        };
        NearWindow W;
        int at = I.s0, pos = 0;
        float4 ph[2], pl[2];                        // the next chunk's sources of this lane
        auto fetch = [&]() {
#pragma unroll
            for (int r = 0; r < 2; r++) {
                const int j = W.moonlet(pos + 32 * r, lane);
                // (a place past the window, which a last chunk's padding to quads sums: a massless source at the
                // item's first moonlet, so that its separations are as finite as the leaf's)
                ph[r] = A.hi4[j >= 0 ? j : I.first];
                pl[r] = A.lo4[j >= 0 ? j : I.first];
                if (j < 0) ph[r].w = 0.f;
            }
        };
        if (at < I.s1) {
            W.load(A.p2p_src, at, I.s1, lane);
            fetch();
        }
        while (at < I.s1) {
            const int quads = (min(NEAR_CHUNK, W.total - pos) + 3) >> 2;
            __syncwarp();   // the last chunk has been summed
#pragma unroll
            for (int r = 0; r < 2; r++) {
                const int t = lane + 32 * r;
                S[0][t] = ph[r].x;
                S[1][t] = ph[r].y;
                S[2][t] = ph[r].z;
                S[3][t] = ph[r].w;
                S[4][t] = pl[r].x;
                S[5][t] = pl[r].y;
                S[6][t] = pl[r].z;
            }
            __syncwarp();
            pos += NEAR_CHUNK;   // the next chunk, or the next window's first
            if (pos >= W.total) {
                at += 32;
                pos = 0;
                if (at < I.s1) W.load(A.p2p_src, at, I.s1, lane);
            }
            if (at < I.s1) fetch();
            if (act) {
                for (int k = g; k < quads; k += G) {
                    const ulonglong2 hx = *reinterpret_cast<const ulonglong2 *>(&S[0][4 * k]);
                    const ulonglong2 hy = *reinterpret_cast<const ulonglong2 *>(&S[1][4 * k]);
                    const ulonglong2 hz = *reinterpret_cast<const ulonglong2 *>(&S[2][4 * k]);
                    const ulonglong2 mu = *reinterpret_cast<const ulonglong2 *>(&S[3][4 * k]);
                    const ulonglong2 lx = *reinterpret_cast<const ulonglong2 *>(&S[4][4 * k]);
                    const ulonglong2 ly = *reinterpret_cast<const ulonglong2 *>(&S[5][4 * k]);
                    const ulonglong2 lz = *reinterpret_cast<const ulonglong2 *>(&S[6][4 * k]);
                    p2p_f32x2(hx.x, hy.x, hz.x, mu.x, lx.x, ly.x, lz.x, T0, a0[0], a0[1], a0[2]);
                    p2p_f32x2(hx.x, hy.x, hz.x, mu.x, lx.x, ly.x, lz.x, T1, a1[0], a1[1], a1[2]);
                    p2p_f32x2(hx.y, hy.y, hz.y, mu.y, lx.y, ly.y, lz.y, T0, a0[0], a0[1], a0[2]);
                    p2p_f32x2(hx.y, hy.y, hz.y, mu.y, lx.y, ly.y, lz.y, T1, a1[0], a1[1], a1[2]);
                }
            }
            since += rounds;
            if (since + rounds > 16) fold();   // a half's running sum takes two terms a quad: at most 32
            if (!asked) {
                asked = true;
                li = __shfl_sync(0xffffffffu, next, 0);
                if (li < n_items) item = __ldg(&A.items[li]);
            }
        }
        if (since) fold();
        // the groups' totals in group order
        const float f0[6] = {h0[0], h0[1], h0[2], l0[0], l0[1], l0[2]};
        const float f1[6] = {h1[0], h1[1], h1[2], l1[0], l1[1], l1[2]};
        for (int q = 1; q < G; q++) {
            const int from = min(31, q * L + lane);   // (lanes past the first group add values of no use)
#pragma unroll
            for (int d = 0; d < 3; d++) {
                const float p = __shfl_sync(0xffffffffu, f0[d], from), pl_ = __shfl_sync(0xffffffffu, f0[3 + d], from);
                df_add(h0[d], l0[d], p);
                l0[d] += pl_;
                const float q1 = __shfl_sync(0xffffffffu, f1[d], from), ql = __shfl_sync(0xffffffffu, f1[3 + d], from);
                df_add(h1[d], l1[d], q1);
                l1[d] += ql;
            }
        }
        if (g == 0) {
            near_store(A, i0, I.whole, static_cast<double>(h0[0]) + static_cast<double>(l0[0]),
                       static_cast<double>(h0[1]) + static_cast<double>(l0[1]),
                       static_cast<double>(h0[2]) + static_cast<double>(l0[2]));
            if (2 * tt + 1 < m)
                near_store(A, i0 + 1, I.whole, static_cast<double>(h1[0]) + static_cast<double>(l1[0]),
                           static_cast<double>(h1[1]) + static_cast<double>(l1[1]),
                           static_cast<double>(h1[2]) + static_cast<double>(l1[2]));
        }
        if (!asked) {
            li = __shfl_sync(0xffffffffu, next, 0);
            if (li < n_items) item = __ldg(&A.items[li]);
        }
    }
}

// FP64: bound by the FP64 pipe (one warp instruction per 64 cycles per SM
// sub-partition), so a pair of leaves is summed once for both: the separation
// and r^-3 serve the pull on either moonlet, 20 FP64 instructions for what
// takes 32 as two pulls.  Of an item's entries those with a later leaf count
// (and the leaf itself, one way).  A block takes an item, each warp a quarter
// of its targets (a pair of leaves keeps one warp's share of the pipe busy for
// half a millisecond) and all its sources, 32 at a time, one per lane, so that
// all lanes work whatever the leaves' sizes.  A warp goes through its m targets
// with lane l starting at target l mod m: the lanes' pulls on the targets go to
// distinct places of the warp's sums in shared memory (lanes that would meet
// have copies of the sums), those on the lane's source stay in registers.  Both
// are added to the moonlets' sums in memory with FP64 atomics, so a sum's last
// bits depend on the order of the blocks and of the targets (the far kernel
// gives coincident moonlets one result).  With few targets to a leaf some of
// the block's warps have none, and yet no force call of leaves of 1 to 16
// moonlets takes longer than with a block of 128 threads per leaf (N = 1e5,
// leaves of one: 8.4 -> 6.3 ms).
// N = 1e5, p = 6, beside M2L: 3.57 ms one way (a block per leaf and share, 97 %
// of the lanes at work), 2.6 ms this way; both near their instructions' time.
// With a warp's items cut by entries instead (few sources, many targets)
// 3.2 ms, and at N = 1e4 twice the one-way time.
constexpr int NEAR64_SHARE = 64 / NEAR_WARPS, NEAR64_SUMS = 3 * NEAR64_SHARE;   // targets and sums of a warp

struct __align__(16) NearShared64 {             // of a warp
    double t[4][NEAR64_SHARE];                  // x, y, z, mu of its targets
    double sum[3][NEAR64_SUMS];                 // pulls on them: copies of m sums
};

__global__ void __launch_bounds__(NEAR_THREADS, 6) k_near_f64(NearArgs A) {
    __shared__ NearShared64 s_warp[NEAR_WARPS];
    __shared__ int s_item[2];
    if (aborted(A.ctl)) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    NearShared64 &S = s_warp[warp];
    const int n_items = min(A.ctl->n_near, A.item_cap);
    for (int turn = 0;; turn ^= 1) {
        if (threadIdx.x == 0) s_item[turn] = atomicAdd(A.work, 1);
        __syncthreads();   // (the item before last, of this slot, has been read by every thread)
        const int li = s_item[turn];
        if (li >= n_items) break;
        const NearItem I(__ldg(&A.items[li]));
        // the warp's share of the item's targets (at most 64)
        const int first = I.first + I.count * warp / NEAR_WARPS, m = I.first + I.count * (warp + 1) / NEAR_WARPS - first;
        if (m == 0) continue;
        if (lane < m) {
            S.t[0][lane] = A.x[first + lane];
            S.t[1][lane] = A.y[first + lane];
            S.t[2][lane] = A.z[first + lane];
            S.t[3][lane] = A.G * A.m[first + lane];
        }
#pragma unroll
        for (int d = 0; d < 3; d++) S.sum[d][lane] = S.sum[d][16 + lane] = 0.0;
        const int copy = lane / m, i_first = lane - copy * m;   // (32 lanes, m <= 16: places 0 to 31, the last copy cut)
        __syncwarp();
        NearWindow W;
        for (int at = I.s0; at < I.s1; at += 32) {
            // the window's entries: later leaves, and the targets' own
            int2 e = make_int2(0, 0);
            if (at + lane < I.s1) e = __ldg(&A.p2p_src[at + lane]);
            const bool own = e.x <= I.first && I.first < e.x + e.y;
            const unsigned which = __ballot_sync(0xffffffffu, own);
            const int o0 = __shfl_sync(0xffffffffu, e.x, __ffs(which) - 1);
            const int o1 = o0 + __shfl_sync(0xffffffffu, e.y, __ffs(which) - 1);
            const unsigned keep = __ballot_sync(0xffffffffu, e.y > 0 && (own || e.x > I.first));
            const unsigned from = __fns(keep, 0, lane + 1);   // (a window's entries are not empty)
            e.x = __shfl_sync(0xffffffffu, e.x, from & 31);
            e.y = __shfl_sync(0xffffffffu, e.y, from & 31);
            W.set(from < 32 ? e : make_int2(0, 0), lane);
            for (int pos = 0; pos < W.total; pos += 32) {
                const int j = W.moonlet(pos, lane);
                const bool valid = j >= 0, both = valid && !(which && j >= o0 && j < o1);
                double X = 0.0, Y = 0.0, Z = 0.0, M = 0.0, ax = 0.0, ay = 0.0, az = 0.0;
                if (valid) {
                    X = A.x[j];
                    Y = A.y[j];
                    Z = A.z[j];
                    M = A.G * A.m[j];
                }
                for (int s = 0, i = i_first; s < m; s++) {
                    const int q = copy * m + i;
                    const double mu = S.t[3][i];
                    const double dx = X - S.t[0][i], dy = Y - S.t[1][i], dz = Z - S.t[2][i];
                    double fi, fj;   // mu r^-3 of the source's pull on the target and of the target's on the source
                    p2p_f64_both(dx * dx + dy * dy + dz * dz, M, mu, fi, fj);
                    if (!valid) fi = 0.0;   // (a lane past the sources)
                    const double sx = S.sum[0][q], sy = S.sum[1][q], sz = S.sum[2][q];
                    S.sum[0][q] = sx + dx * fi;
                    S.sum[1][q] = sy + dy * fi;
                    S.sum[2][q] = sz + dz * fi;
                    ax -= dx * fj;
                    ay -= dy * fj;
                    az -= dz * fj;
                    i = i + 1 < m ? i + 1 : 0;
                    __syncwarp();   // the next lane's turn at this target
                }
                if (both) near_store(A, j, false, ax, ay, az);
            }
        }
        if (lane < m) {   // the copies of the sums
            double v[3] = {0.0, 0.0, 0.0};
            for (int q = lane; q < NEAR64_SUMS; q += m)
#pragma unroll
                for (int d = 0; d < 3; d++) v[d] += S.sum[d][q];
            near_store(A, first + lane, false, v[0], v[1], v[2]);
        }
        __syncwarp();   // the sums have been read
    }
}

void launch_near(ncorp_ctx *c, const ParticleSet &P, bool mixed, double G) {
    NearArgs A;
    A.items = c->wl.near_items; A.item_cap = c->wl.near_cap;
    A.p2p_src = c->wl.p2p_src;
    A.x = P.x; A.y = P.y; A.z = P.z; A.m = P.m;
    A.hi4 = P.hi4; A.lo4 = P.lo4;
    A.G = G;
    A.nx = c->amx; A.ny = c->amy; A.nz = c->amz;   // the far kernel overwrites them in place
    A.work = c->work_counter;
    A.ctl = c->ctl;
    const void *kern = mixed ? reinterpret_cast<const void *>(k_near_f32) : reinterpret_cast<const void *>(k_near_f64);
    int per_sm = 0;
    NCORP_CUDA_CHECK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, NEAR_THREADS, 0));
    if (per_sm < 1) per_sm = 1;
    void *args[] = {&A};
    NCORP_CUDA_CHECK(cudaLaunchKernel(kern, dim3(per_sm * c->num_sms), dim3(NEAR_THREADS), args, 0, c->stream));
    c->launches++;
}

}  // namespace ncorp
