// grid.cu -- preconditioned conjugate gradients in one persistent launch
// (Section 1.1), one thread block per SM, for systems whose parts fit on chip.
//
// The forest's contraction tree is cut as for the binned solve (bins.cu), but
// into as many equal "parts" as there are thread blocks: a part is a set of
// whole contraction subtrees of at most `bmax` vertices, packed in spatial
// order; the vertices whose subtree is larger are the "top" (a few hundred).
// Block b keeps its part's slice of every solver vector for the whole solve
// and runs, per iteration,
//   q = Gamma p on its rows (its own p and the rows of other parts that its
//     rows name, the "halo", in shared memory), p^T q
//   r -= alpha q, x += alpha p, |r|^2, its part's forward levels
//   z at the top vertices it reaches or owns, from the rows and columns of the
//     top's L^-1 that these need
//   its part's backward levels, r^T z, p = z + beta p
// Between the blocks travel p of the halo, the parts' sums for the top with
// the top's r, and three sums (p^T q, |r|^2, r^T z).
//
// Values that other blocks wait for travel in packets of 8-byte words, half
// data, half the number of the exchange: the value and its arrival are one
// memory access, with no fence and no flag.  A sum is exchanged all to all
// (every block reads the packets of all others), so each block adds the same
// numbers in the same order and takes the same decisions.  Every wait is
// bounded; one that gives up sets the error word and the launch ends.  The
// launch is cooperative: all its blocks are resident.
//
// Levels are stored as the instructions a warp runs ("slots", see
// k_gr_segments): records and blocks in the order of use, so that a level
// costs its reads of the vector and a barrier.
//
// The top's rows and columns of L^-1 (a few hundred vertices, once per factor)
// replace its 2 x 10 levels, which every block ran for itself.
//
// What bounds it: the levels of a part (about 10 each way; 200-300 clocks
// each, a chain of shared-memory reads, products and a barrier), the
// exchanges (about 1.2 us each) and the wait for the largest part, up to
// about 3e5 cells in FP32; FP64 by its issue rate (1/64 of FP32's); at 1e6
// cells also the stream of matrix rows and blocks from HBM.
// Measured per iteration against the multi-launch paths it replaces (product,
// vector kernels and level kernels or bins; tol 1e-10): FP64 lattice of 1e4
// cells 30.6 us (104), FP32 spheroid of 1e5 27.5 us (63), FP32 sheet of 2.5e5
// 34 us (76), FP64 spheroid of 3e5 121 us (282), FP32 spheroid of 1e6 122 us
// (181); block Jacobi, FP64, 2e5 cells 54 us (81).
#include <algorithm>
#include <cmath>
#include <cstddef>
#include <cstring>
#include <type_traits>

#include "solver_common.cuh"

namespace {

constexpr int GT = 512;          // threads of a part's block
constexpr int GW = GT / 32;
constexpr int PMAX = 160;        // parts
constexpr int NBIG = 32, NSWEEP = 24;   // large subtrees of a part; rounds of handing them over
constexpr int NTOP = 2048;       // top vertices
constexpr int NREC = 8190;       // cells that a slot's record can name (13 bits, one spare)
constexpr int CMAX = 48;         // entries of a column of the top's X
constexpr int TLONG = 32;        // a row of X with more entries has a warp, others 8 lanes
constexpr int GRID_SMEM = 226 * 1024;   // of 227, beside up to 0.8 KB of static shared memory
constexpr int MS_ITEMS = 4096;   // items per block of the stable split

constexpr int LMAX = 64;         // contraction levels
constexpr int NCLS = 8;          // segment classes: 8 sources or more, 7, ... 1

// header of a part (entry P: the top); Q_NSF, Q_NSB: slots of its programs;
// Q_NA, Q_NL: rows of the top that it forms and how many are long; Q_XR, Q_XC:
// entries of those rows and of the columns of its outputs (padded)
enum { Q_SOFF, Q_NV, Q_ROFF, Q_NR, Q_T0, Q_NP, Q_POFF, Q_NZ, Q_ZOFF, Q_DOFF, Q_NSF, Q_SF, Q_NSB, Q_SB,
       Q_NA, Q_AOFF, Q_NL, Q_XR, Q_XC, Q_N = 24 };
// totals and maxima over the parts
enum { T_NT, T_NR, T_P, T_Z, T_D, T_SF, T_SB, T_MNR, T_MNZ, T_MSF, T_MSB, T_MDZ, T_MNF, T_MNB, T_MNO,
       T_RE, T_CE, T_A, T_MNA, T_MX, T_ERR, T_N = 32 };
// a matrix's rows on the parts: slots and halo cells of each part with their
// offsets; behind the parts the totals and the largest halo
enum { R_NS, R_SLOT, R_NH, R_HOFF, R_N };
// streams of a program: first slot of every warp's wide levels, of the narrow
// levels, the end; wide levels
enum { W_NARROW = GW, W_END, W_LEVELS, W_N = GW + 4 };

__host__ __device__ __forceinline__ int32_t pad32(int32_t x) { return (x + 31) & ~31; }
__host__ __device__ __forceinline__ int32_t pad8(int32_t x) { return (x + 7) & ~7; }

// Block-wide exclusive scan of one int per thread; *total gets the sum.
template <int BS>
__device__ __forceinline__ int32_t gscan(int32_t v, int32_t *sh, int32_t *total)
{
    const int l = threadIdx.x & 31, w = threadIdx.x >> 5;
    int32_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (l >= o) x += y;
    }
    if (l == 31) sh[w] = x;
    __syncthreads();
    if (w == 0) {
        int32_t t = (l < BS / 32) ? sh[l] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            int32_t y = __shfl_up_sync(0xffffffffu, t, o);
            if (l >= o) t += y;
        }
        if (l < BS / 32) sh[l] = t;
    }
    __syncthreads();
    int32_t before = (w > 0 ? sh[w - 1] : 0) + x - v;
    *total = sh[BS / 32 - 1];
    __syncthreads();
    return before;
}

// ------------------------------------------------------------- structure
// parent in the contraction tree: the receiver eliminated first
__global__ void k_gr_parent(int32_t n, const int32_t *__restrict__ pr_ptr, const int32_t *__restrict__ pr_q,
                            const int32_t *__restrict__ pos, int32_t *par, int32_t *sz)
{
    int32_t t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n) return;
    int32_t best = -1;
    for (int32_t p = pr_ptr[t]; p < pr_ptr[t + 1]; ++p) {
        int32_t u = pos[pr_q[p]];
        if (best < 0 || u < best) best = u;
    }
    par[t] = best;
    sz[t] = 1;
}
// subtree sizes of one level's vertices added to their parents
__global__ void k_gr_size(int32_t p0, int32_t cnt, const int32_t *__restrict__ par, int32_t *sz)
{
    int32_t k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= cnt) return;
    int32_t t = p0 + k, u = par[t];
    if (u >= 0) atomicAdd(sz + u, sz[t]);
}
// the same for all remaining (short) levels in one block
__global__ void __launch_bounds__(1024) k_gr_size_rest(const int32_t *__restrict__ lp, int l0, int LV,
                                                       const int32_t *__restrict__ par, int32_t *sz)
{
    for (int l = l0; l < LV; ++l) {
        for (int32_t t = lp[l] + threadIdx.x; t < lp[l + 1]; t += blockDim.x) {
            const int32_t u = par[t];
            if (u >= 0) atomicAdd(sz + u, atomicAdd(sz + t, 0));
        }
        __threadfence();
        __syncthreads();
    }
}
// top: subtree above bmax; roots carry their subtree's size, by vertex (and
// again those of at most `small` vertices alone)
__global__ void k_gr_class(int32_t n, int32_t bmax, int32_t small, const int32_t *__restrict__ sz,
                           const int32_t *__restrict__ par, const int32_t *__restrict__ ord, int32_t *wv, int32_t *wsm)
{
    int32_t t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n) return;
    const int32_t s = sz[t], u = par[t], w = (s <= bmax && (u < 0 || sz[u] > bmax)) ? s : 0;
    wv[ord[t]] = w;
    wsm[ord[t]] = w <= small ? w : 0;
}
// The parts of the roots.  A root goes by its subtree's middle in the running
// total of sizes (vertices are in spatial order, so parts are compact), which
// leaves a part short or over by half a subtree at either end.  Then
// neighbouring parts hand large subtrees over (k_gr_balance), and the small
// ones fill all parts up to a common level, in order (k_gr_fill, k_gr_small).
// The parts run in step, so the largest one sets the pace.  Largest part by
// the middles alone and so (rows; the mean): FP32 1e5 cells 838 and 725 (658),
// sheet of 2.5e5 2174 and 1767 (1645), FP64 3e5 2757 and 2208 (1974).
// anc: itself for roots and top vertices (seg: P for the top), else its parent
// (a batch: instance s has the vertices [irow[s], irow[s+1]) and the parts
// [ipart[s], ipart[s+1]), and its top vertices are segment P + s)
__global__ void k_gr_roots(int32_t n, int32_t bmax, int32_t P, int32_t NI, const int32_t *__restrict__ irow,
                           const int32_t *__restrict__ ipart, const int32_t *__restrict__ sz,
                           const int32_t *__restrict__ par, const int32_t *__restrict__ ord,
                           const int32_t *__restrict__ pre, int32_t small, int32_t *load, int32_t *cnt, int32_t *list,
                           int32_t *anc, int32_t *seg)
{
    int32_t t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n) return;
    const int32_t s = sz[t], u = par[t];
    const bool tp = s > bmax, rt = !tp && (u < 0 || sz[u] > bmax);
    anc[t] = (tp || rt) ? t : u;
    int32_t b = -1;
    if (tp || rt) {
        const int32_t v = ord[t];
        int32_t lo = 0, hi = NI;   // the instance: the last one that starts at or before v
        while (hi - lo > 1) {
            const int32_t mid = (lo + hi) >> 1;
            if (irow[mid] <= v) lo = mid; else hi = mid;
        }
        if (tp) {
            b = P + lo;
        } else {
            const int32_t p0 = ipart[lo], np = ipart[lo + 1] - p0, before = pre[irow[lo]];
            const int64_t total = max(pre[irow[lo + 1]] - before, 1);
            b = p0 + (int32_t)min((int64_t)np - 1, ((int64_t)(pre[v] - before) + s / 2) * np / total);
            atomicAdd(load + b, s);
            if (s <= small) {
                b = -2 - lo;
            } else {
                const int32_t k = atomicAdd(cnt + b, 1);
                if (k < NBIG) list[b * NBIG + k] = t;
            }
        }
    }
    seg[t] = b;
}
// Large subtrees move between neighbouring parts of one instance, from the
// heavier to the lighter, alone or against a smaller one, a warp per pair:
// whatever leaves the smallest difference.  load: all the parts' sizes in, the large subtrees' sizes out.
__global__ void __launch_bounds__(1024) k_gr_balance(int32_t P, int32_t NI, const int32_t *__restrict__ ipart,
                                                     const int32_t *__restrict__ sz, const int32_t *__restrict__ cnt,
                                                     const int32_t *__restrict__ list, int32_t *load, int32_t *seg)
{
    __shared__ int32_t st[PMAX][NBIG], ss[PMAX][NBIG], sc[PMAX], sl[PMAX], first[PMAX];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int32_t b = w; b < P; b += 32) {
        // in the order of their vertices (the list's depends on timing)
        const int32_t c = cnt[b] <= NBIG ? cnt[b] : 0, t = lane < c ? list[b * NBIG + lane] : INT32_MAX;
        int32_t rank = 0;
        for (int k = 0; k < c; ++k) rank += __shfl_sync(0xffffffffu, t, k) < t;
        if (lane < c) {
            st[b][rank] = t;
            ss[b][rank] = sz[t];
        }
        if (lane == 0) {
            sc[b] = c;
            sl[b] = load[b];
            first[b] = 0;
        }
    }
    __syncthreads();
    for (int32_t s = threadIdx.x; s < NI; s += 1024)
        if (ipart[s + 1] > ipart[s]) first[ipart[s]] = 1;
    __syncthreads();
    int still = 0;   // sweeps without a move, both parities in turn
    for (int r = 0; r < NSWEEP && still < 2; ++r) {
        int moved = 0;
        for (int32_t b = 2 * w + (r & 1); b + 1 < P; b += 64) {
            if (first[b + 1]) continue;
            const int32_t d = sl[b] - sl[b + 1], from = d > 0 ? b : b + 1, to = d > 0 ? b + 1 : b, D = abs(d), c = sc[from],
                          c2 = sc[to];
            const int32_t x = lane < c ? ss[from][lane] : 0;
            int32_t left = INT32_MAX, other = -1;   // the best against this lane's subtree: none, or one of the lighter part
            if (x > 0)
                for (int32_t k = c2 < NBIG ? -1 : 0; k < c2; ++k) {
                    const int32_t y = x - (k < 0 ? 0 : ss[to][k]);
                    if (y > 0 && y < D && abs(D - 2 * y) < left) {
                        left = abs(D - 2 * y);
                        other = k;
                    }
                }
            const int32_t best = __reduce_min_sync(0xffffffffu, left);
            if (best >= D) continue;
            moved = 1;
            const int k = __ffs(__ballot_sync(0xffffffffu, left == best)) - 1;
            if (lane == k) {
                const int32_t t = st[from][k];
                if (other >= 0) {
                    const int32_t y = ss[to][other];
                    st[from][k] = st[to][other];
                    ss[from][k] = y;
                    st[to][other] = t;
                    ss[to][other] = x;
                    sl[from] -= x - y;
                    sl[to] += x - y;
                } else {
                    st[from][k] = st[from][c - 1];
                    ss[from][k] = ss[from][c - 1];
                    st[to][c2] = t;
                    ss[to][c2] = x;
                    sc[from] = c - 1;
                    sc[to] = c2 + 1;
                    sl[from] -= x;
                    sl[to] += x;
                }
            }
            __syncwarp();
        }
        still = __syncthreads_or(moved) ? 0 : still + 1;
    }
    for (int32_t b = w; b < P; b += 32) {
        // a part with more large subtrees than the list holds keeps them all
        const bool over = cnt[b] > NBIG;
        int32_t x = 0;
        if (lane < sc[b]) {
            seg[st[b][lane]] = b;
            x = ss[b][lane];
        }
        x = __reduce_add_sync(0xffffffffu, x);
        if (lane == 0) load[b] = over ? sl[b] : x;
    }
}
// A warp per instance: the level up to which its small subtrees fill its
// parts, and each part's room, as a running total.
__global__ void __launch_bounds__(256) k_gr_fill(int32_t NI, const int32_t *__restrict__ irow, const int32_t *__restrict__ ipart,
                                                 const int32_t *__restrict__ psm, const int32_t *__restrict__ load,
                                                 int32_t *room)
{
    const int lane = threadIdx.x & 31;
    for (int32_t s = threadIdx.x >> 5; s < NI; s += 8) {
        const int32_t p0 = ipart[s], np = ipart[s + 1] - p0, want = psm[irow[s + 1]] - psm[irow[s]];
        constexpr int K = (PMAX + 31) / 32;   // parts per lane, consecutive
        int32_t l[K] = {}, hi = 0;
        const int32_t k = (np + 31) / 32, b0 = lane * k;
#pragma unroll
        for (int u = 0; u < K; ++u) {
            l[u] = u < k && b0 + u < np ? load[p0 + b0 + u] : INT32_MAX;
            hi = max(hi, l[u] == INT32_MAX ? 0 : l[u]);
        }
        int32_t lo = -1;   // the lowest level with room for all of them
        hi = __reduce_max_sync(0xffffffffu, hi) + want;
        while (hi - lo > 1) {
            const int32_t mid = lo + (hi - lo) / 2;
            int32_t c = 0;
#pragma unroll
            for (int u = 0; u < K; ++u) c += min(max(mid - l[u], 0), want);
            c = __reduce_add_sync(0xffffffffu, min(c, want));
            if (c >= want) hi = mid; else lo = mid;
        }
        int32_t c = 0, own = 0;
#pragma unroll
        for (int u = 0; u < K; ++u) own += max(hi - l[u], 0);
        int32_t x = own;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int32_t y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        c = x - own;
#pragma unroll
        for (int u = 0; u < K; ++u) {
            if (u >= k || b0 + u >= np) break;
            room[p0 + b0 + u] = c;
            c += max(hi - l[u], 0);
        }
    }
}
// small roots: the part in whose room the subtree's middle lies
__global__ void k_gr_small(int32_t n, const int32_t *__restrict__ irow, const int32_t *__restrict__ ipart,
                           const int32_t *__restrict__ sz, const int32_t *__restrict__ ord, const int32_t *__restrict__ psm,
                           const int32_t *__restrict__ room, int32_t *seg)
{
    int32_t t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n || seg[t] > -2) return;
    const int32_t s = -2 - seg[t], x = psm[ord[t]] - psm[irow[s]] + sz[t] / 2;
    int32_t lo = ipart[s], hi = ipart[s + 1];
    while (hi - lo > 1) {
        const int32_t mid = (lo + hi) >> 1;
        if (room[mid] <= x) lo = mid; else hi = mid;
    }
    seg[t] = lo;
}
__global__ void k_gr_jump(int32_t n, const int32_t *__restrict__ a, int32_t *b)
{
    int32_t t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < n) b[t] = a[a[t]];
}
__global__ void k_gr_seg(int32_t n, const int32_t *__restrict__ anc, const int32_t *__restrict__ rootseg, int32_t *seg)
{
    int32_t t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < n) seg[t] = rootseg[anc[t]];
}

// Stable split of items by segment (seg[i] in [0, ns)): counts per block of
// items, a scan over (segment, block), then ranks by warp matches.
__global__ void __launch_bounds__(GT) k_gr_split_count(int32_t n, int32_t ns, const int32_t *__restrict__ seg,
                                                       int32_t *hist)
{
    __shared__ int32_t h[2 * PMAX];
    for (int i = threadIdx.x; i < ns; i += GT) h[i] = 0;
    __syncthreads();
    const int32_t i0 = blockIdx.x * MS_ITEMS;
    for (int32_t i = i0 + threadIdx.x; i < min(n, i0 + MS_ITEMS); i += GT) atomicAdd(h + seg[i], 1);
    __syncthreads();
    for (int i = threadIdx.x; i < ns; i += GT) hist[(size_t)i * gridDim.x + blockIdx.x] = h[i];
}
__global__ void __launch_bounds__(GT) k_gr_split_place(int32_t n, int32_t ns, const int32_t *__restrict__ seg,
                                                       const int32_t *__restrict__ off, int32_t *out, int32_t *lpos)
{
    __shared__ int32_t wc[GW][2 * PMAX];
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    for (int i = threadIdx.x; i < GW * 2 * PMAX; i += GT) (&wc[0][0])[i] = 0;
    __syncthreads();
    constexpr int PER = MS_ITEMS / GW;   // consecutive items of a warp
    const int32_t i0 = blockIdx.x * MS_ITEMS + w * PER;
    for (int r = 0; r < PER; r += 32) {
        const int32_t i = i0 + r + l;
        if (i < n) atomicAdd(&wc[w][seg[i]], 1);
    }
    __syncthreads();
    for (int s = threadIdx.x; s < ns; s += GT) {
        int32_t at = off[(size_t)s * gridDim.x + blockIdx.x];
        for (int k = 0; k < GW; ++k) {
            const int32_t c = wc[k][s];
            wc[k][s] = at;
            at += c;
        }
    }
    __syncthreads();
    for (int r = 0; r < PER; r += 32) {
        const int32_t i = i0 + r + l;
        const int32_t s = i < n ? seg[i] : ns;
        const unsigned m = __match_any_sync(0xffffffffu, s);
        const int32_t rank = __popc(m & ((1u << l) - 1u));
        int32_t at = 0;
        if (s < ns) at = wc[w][s] + rank;
        __syncwarp();
        if (s < ns && rank == 0) wc[w][s] = at + __popc(m);
        __syncwarp();
        if (s < ns) {
            out[at] = i;
            if (lpos) lpos[i] = at - off[(size_t)s * gridDim.x];
        }
    }
}

// a batch: the instances' top segments become one, in order
__global__ void k_gr_top_merge(int32_t n, int32_t P, int32_t nblk, const int32_t *__restrict__ off, int32_t *seg, int32_t *lpos)
{
    int32_t t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n || seg[t] <= P) return;
    lpos[t] += off[(size_t)seg[t] * nblk] - off[(size_t)P * nblk];
    seg[t] = P;
}

// Row segments: part b's vertices, then the top vertices it owns, padded to
// 32 rows; the top's own header.
__global__ void __launch_bounds__(256) k_gr_rows(int32_t P, int32_t NI, const int32_t *__restrict__ ipart, int32_t nblk,
                                                 const int32_t *__restrict__ off, int32_t *hdr, int32_t *tot)
{
    __shared__ int32_t sh[8];
    const int b = threadIdx.x;
    const int32_t s0 = off[(size_t)P * nblk], s1 = off[(size_t)(P + NI) * nblk];
    const int32_t nt = s1 - s0;
    int32_t nv = 0, nto = 0, t0 = 0, so = 0;
    if (b < P) {
        so = off[(size_t)b * nblk];
        nv = off[(size_t)(b + 1) * nblk] - so;
        int32_t lo = 0, hi = NI;   // the part's instance and its top vertices
        while (hi - lo > 1) {
            const int32_t mid = (lo + hi) >> 1;
            if (ipart[mid] <= b) lo = mid; else hi = mid;
        }
        const int32_t ta = off[(size_t)(P + lo) * nblk] - s0, te = off[(size_t)(P + lo + 1) * nblk] - s0,
                      np = ipart[lo + 1] - ipart[lo], tc = (te - ta + np - 1) / max(np, 1);
        t0 = min(te, ta + (b - ipart[lo]) * tc);
        nto = min(te, t0 + tc) - t0;
    }
    int32_t total;
    const int32_t ro = gscan<256>(pad32(nv + nto), sh, &total);
    if (b <= P) {
        int32_t *h = hdr + (size_t)Q_N * b;
        for (int k = 0; k < Q_N; ++k) h[k] = 0;
        h[Q_SOFF] = b < P ? so : s0;
        h[Q_NV] = b < P ? nv : nt;
        h[Q_ROFF] = b < P ? ro : total;
        h[Q_NR] = nv + nto;
        h[Q_T0] = t0;
    }
    if (b == 0) {
        tot[T_NT] = nt;
        tot[T_NR] = total;
        if (nt > NTOP) tot[T_ERR] = 1;
    }
}

// parts of U consecutive rows (no forest)
__global__ void __launch_bounds__(256) k_gr_rows_plain(int32_t n, int32_t P, int32_t U, int32_t *hdr, int32_t *tot)
{
    const int b = threadIdx.x;
    if (b > P) return;
    int32_t *h = hdr + (size_t)Q_N * b;
    for (int k = 0; k < Q_N; ++k) h[k] = 0;
    const int32_t r0 = min(n, b * U), nr = b < P ? min(n, r0 + U) - r0 : 0;
    h[Q_SOFF] = r0;
    h[Q_NV] = h[Q_NR] = nr;
    h[Q_ROFF] = b * pad32(U);
    if (b == P) {
        tot[T_NR] = (P - 1) * pad32(U) + pad32(n - (P - 1) * U);
        tot[T_MNR] = U;
    }
}

struct GBuild {
    int32_t n, P, LV;
    int32_t NRW;                             // halo bitmap words per part
    const int32_t *lp;                       // level boundaries of positions
    const int32_t *ord, *pos, *pr_ptr, *pr_q, *pr_c;
    const int32_t *seg, *sp, *lpos;
    const int32_t *row_ptr, *col;            // the matrix's rows (internal order)
    const float2 *col32;                     // MIXED: the column of a slot is in its record
    int32_t *hdr, *tot, *vm, *rh;            // rh: R_N per part
    int32_t *i_of_t, *t_of_i, *d_src;
    int32_t *dcnt, *plist, *sgk, *sgd, *sgf, *sgn; // per receiver counts; pairs by receiver; segments
    int32_t *nseg;                           // segments of each part
    int32_t *kb;                             // first segment of every (program, level, class) inside its level
    int32_t *st;                             // first step of every (program, level): 2 x (LMAX + 1) per part
    int32_t *sp_slot[2], *sp_n[2];           // every step's first slot, and its slots | barriers before << 16
    int32_t *ws;                             // streams: 2 x W_N per part
    int32_t lps;                             // receivers per step of a part: 32, or 10 with a lane per row
    int32_t *glen, *gso;
    uint16_t *perm;
    uint32_t *hb;                            // halo bitmap
    int32_t *hpre;                           // its running count, per word
    int32_t *hl;                             // halo rows
    uint8_t *xflag;                          // rows other parts read
    char *prog[2];                           // slots of the parts
    int32_t *msrc[2];                        // source pair of every slot's lane
    int32_t *zslot, *tlk;
    int32_t *clen, *rlen, *cptr, *rptr;      // the top's X: entries of its columns and rows, and where they start
    int32_t *cidx;                           // rows of every column's entries, CMAX per column
    double *cx;                              // and their blocks
    int32_t *xi;                             // the other index of every entry: rows, then columns
    int4 *alist, *outs;                      // per part: rows of X, outputs (see k_gr_part_top)
    int identity, halo;
};

__device__ __forceinline__ int level_of(const int32_t *lp, int LV, int32_t t)
{
    int lo = 0, hi = LV;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (lp[mid] <= t) lo = mid; else hi = mid;
    }
    return lo;
}

// rows of every part <-> internal rows
__global__ void __launch_bounds__(GT) k_gr_row_maps(GBuild g)
{
    const int32_t *h = g.hdr + (size_t)Q_N * blockIdx.x;
    const int32_t nv = h[Q_NV], nr = h[Q_NR], ro = h[Q_ROFF];
    const int32_t st = g.identity ? 0 : g.hdr[(size_t)Q_N * g.P + Q_SOFF] + h[Q_T0] - nv;
    for (int32_t l = blockIdx.y * GT + threadIdx.x; l < pad32(nr); l += GT * gridDim.y) {
        int32_t v = -1, t = -1;
        if (l < nr) {
            if (g.identity) {
                v = h[Q_SOFF] + l;
            } else {
                t = g.sp[l < nv ? h[Q_SOFF] + l : st + l];
                v = g.ord[t];
            }
            g.t_of_i[v] = ro + l;
        }
        g.i_of_t[ro + l] = v;
        if (!g.identity) g.d_src[ro + l] = l < nv ? t : -1;
    }
}

// One part: its pairs and the distinct top vertices it reaches, numbered in
// top order.
__global__ void __launch_bounds__(GT) k_gr_part_count(GBuild g)
{
    __shared__ int32_t sh[GW];
    __shared__ int32_t s_np;
    const int b = blockIdx.x;
    int32_t *h = g.hdr + (size_t)Q_N * b;
    const int32_t so = h[Q_SOFF], nv = h[Q_NV], nt = g.tot[T_NT];
    if (g.tot[T_ERR]) return;
    int32_t *vm = g.vm + (size_t)b * nt;
    if (threadIdx.x == 0) s_np = 0;
    for (int32_t i = threadIdx.x; i < nt; i += GT) vm[i] = 0;
    __syncthreads();
    int32_t c = 0;
    for (int32_t l = threadIdx.x; l < nv; l += GT) {
        const int32_t t = g.sp[so + l];
        for (int32_t p = g.pr_ptr[t]; p < g.pr_ptr[t + 1]; ++p) {
            ++c;
            const int32_t u = g.pos[g.pr_q[p]];
            if (g.seg[u] == g.P) vm[g.lpos[u]] = 1;
        }
    }
    if (c) atomicAdd(&s_np, c);
    __syncthreads();
    int32_t cz = 0;
    for (int32_t base = 0; base < nt; base += GT) {
        const int32_t i = base + threadIdx.x;
        const int32_t f = i < nt ? vm[i] : 0;
        int32_t tz;
        const int32_t ez = gscan<GT>(f, sh, &tz);
        if (i < nt) vm[i] = f ? 1 + cz + ez : 0;
        cz += tz;
    }
    if (threadIdx.x == 0) {
        h[Q_NP] = s_np;
        h[Q_NZ] = cz;
    }
}

// running offsets of one header field over the parts
__device__ __forceinline__ void hdr_scan(int32_t n, int32_t *hdr, int32_t *tot, int f, int fo, int t, int extra, int32_t *sh)
{
    const int b = threadIdx.x;
    int32_t *h = hdr + (size_t)Q_N * b;
    int32_t total;
    const int32_t o = gscan<256>(b < n ? h[f] + extra : 0, sh, &total);
    if (b < n) h[fo] = o;
    if (b == 0) tot[t] = total;
}
__global__ void __launch_bounds__(256) k_gr_offsets1(int32_t P, int32_t *hdr, int32_t *tot)
{
    __shared__ int32_t sh[8];
    hdr_scan(P, hdr, tot, Q_NP, Q_POFF, T_P, 0, sh);
    hdr_scan(P, hdr, tot, Q_NZ, Q_ZOFF, T_Z, 0, sh);
    const int b = threadIdx.x;
    int32_t *h = hdr + (size_t)Q_N * b;
    int32_t total;
    const int32_t o = gscan<256>(b < P ? h[Q_NR] + h[Q_NZ] + 1 : 0, sh, &total);
    if (b < P) h[Q_DOFF] = o;
    if (b == 0) tot[T_D] = total;
}
__global__ void __launch_bounds__(256) k_gr_offsets2(int32_t P, int32_t *hdr, int32_t *tot, const int32_t *ws)
{
    __shared__ int32_t sh[8];
    hdr_scan(P, hdr, tot, Q_NSF, Q_SF, T_SF, 0, sh);
    hdr_scan(P, hdr, tot, Q_NSB, Q_SB, T_SB, 0, sh);
    hdr_scan(P, hdr, tot, Q_NA, Q_AOFF, T_A, 0, sh);
    if (threadIdx.x < P) {
        const int32_t *h = hdr + (size_t)Q_N * threadIdx.x;
        atomicMax(tot + T_MNR, h[Q_NR]);
        atomicMax(tot + T_MNZ, h[Q_NZ]);
        atomicMax(tot + T_MSF, h[Q_NSF]);
        atomicMax(tot + T_MSB, h[Q_NSB]);
        atomicMax(tot + T_MDZ, h[Q_NR] + h[Q_NZ]);
        atomicMax(tot + T_MNO, h[Q_NZ] + h[Q_NR] - h[Q_NV]);
        atomicMax(tot + T_MNA, h[Q_NA]);
        atomicMax(tot + T_MX, h[Q_XR] + h[Q_XC]);
        if (ws) {
            const int32_t *f = ws + (size_t)threadIdx.x * 2 * W_N;
            atomicMax(tot + T_MNF, f[W_END] - f[W_NARROW]);
            atomicMax(tot + T_MNB, f[W_N + W_END] - f[W_N + W_NARROW]);
        }
    }
}

__device__ __forceinline__ int seg_class(int32_t n) { return NCLS - min(n, NCLS); }
// local index of a pair's receiver
__device__ __forceinline__ int32_t pair_dst(const GBuild &g, int b, int32_t nr, const int32_t *vm, int32_t p)
{
    const int32_t u = g.pos[g.pr_q[p]];
    return g.seg[u] == b ? g.lpos[u] : nr + vm[g.lpos[u]] - 1;
}

// The programs of one part: w[dst] -= sum M w[src], level by level.  The pairs of one receiver (forward) or vertex (backward) in one
// level are a segment; the segments of a level, by descending size, are cut
// into steps of lps receivers, one lane (or three, one per row) each; a step
// is as many slots as its largest segment has pairs, and a slot holds one
// pair per receiver.  Levels with more than one step are wide: their steps go
// to the warps in turn, every warp's slots stored in the order it runs them;
// narrow levels are run by warp 0.  Forward programs start wide and end
// narrow, backward ones the other way around.
// This kernel: pairs grouped by receiver (in elimination order), cut into
// segments by level; the steps and the streams.
__global__ void __launch_bounds__(GT) k_gr_segments(GBuild g)
{
    __shared__ int32_t sh[GW], hist[2][LMAX * NCLS], lmax[LMAX];
    const int b = blockIdx.x;
    int32_t *h = g.hdr + (size_t)Q_N * b;
    if (g.tot[T_ERR]) return;
    for (int i = threadIdx.x; i < LMAX; i += GT) lmax[i] = 0;
    const int32_t so = h[Q_SOFF], nv = h[Q_NV], nr = h[Q_NR], nt = g.tot[T_NT], po = h[Q_POFF], nd = nr + h[Q_NZ],
                  lps = g.lps;
    const int32_t *vm = g.vm + (size_t)b * nt;
    int32_t *dc = g.dcnt + h[Q_DOFF];
    for (int i = threadIdx.x; i < 2 * LMAX * NCLS; i += GT) (&hist[0][0])[i] = 0;
    for (int32_t d = threadIdx.x; d <= nd; d += GT) dc[d] = 0;
    __syncthreads();
    for (int32_t l = threadIdx.x; l < nv; l += GT) {
        const int32_t t = g.sp[so + l], p0 = g.pr_ptr[t], p1 = g.pr_ptr[t + 1];
        for (int32_t p = p0; p < p1; ++p) atomicAdd(dc + pair_dst(g, b, nr, vm, p), 1);
        if (p1 > p0) atomicAdd(&hist[1][(g.LV - 1 - level_of(g.lp, g.LV, t)) * NCLS + seg_class(p1 - p0)], 1);
    }
    __syncthreads();
    int32_t carry = 0;
    for (int32_t base = 0; base <= nd; base += GT) {
        const int32_t d = base + threadIdx.x;
        const int32_t c = d < nd ? dc[d] : 0;
        int32_t tot;
        const int32_t ex = gscan<GT>(c, sh, &tot);
        if (d <= nd) dc[d] = carry + ex;
        carry += tot;
    }
    __syncthreads();
    // placed behind the running start of each receiver (which ends at the
    // next one's start: shifted back by the counts below)
    for (int32_t l = threadIdx.x; l < nv; l += GT) {
        const int32_t t = g.sp[so + l];
        for (int32_t p = g.pr_ptr[t]; p < g.pr_ptr[t + 1]; ++p)
            g.plist[po + atomicAdd(dc + pair_dst(g, b, nr, vm, p), 1)] = p;
    }
    __syncthreads();
    int32_t cs = 0;
    for (int32_t base = 0; base < nd; base += GT) {
        const int32_t d = base + threadIdx.x;
        int32_t ns = 0, a0 = 0, a1 = 0;
        if (d < nd) {
            a0 = d > 0 ? dc[d - 1] : 0;
            a1 = dc[d];
            int32_t *L = g.plist + po;
            for (int32_t i = a0 + 1; i < a1; ++i) {   // pair ids ascending: elimination order
                const int32_t x = L[i];
                int32_t j = i - 1;
                while (j >= a0 && L[j] > x) {
                    L[j + 1] = L[j];
                    --j;
                }
                L[j + 1] = x;
            }
        }
        auto lev = [&](int32_t i) { return level_of(g.lp, g.LV, g.pos[g.pr_c[g.plist[po + i]]]); };
        for (int32_t i = a0, lv = -1; i < a1; ++i) {
            const int l2 = lev(i);
            ns += l2 != lv;
            lv = l2;
        }
        int32_t tot;
        int32_t at = cs + gscan<GT>(ns, sh, &tot);
        for (int32_t i = a0; i < a1;) {
            const int lv = lev(i);
            int32_t e = i + 1;
            while (e < a1 && lev(e) == lv) ++e;
            const int32_t n = e - i;
            if (n >= NCLS) atomicMax(lmax + lv, n);
            const int32_t key = lv * NCLS + seg_class(n);
            atomicAdd(&hist[0][key], 1);
            g.sgk[po + at] = key;
            g.sgd[po + at] = d;
            g.sgf[po + at] = i;
            g.sgn[po + at] = n;
            ++at;
            i = e;
        }
        cs += tot;
    }
    __syncthreads();
    __shared__ int32_t lst[2][LMAX + 1], wlen[2][GW + 1], cutl[2];
    if (threadIdx.x < 2) {
        const int q = threadIdx.x;
        int32_t *kb = g.kb + ((size_t)b * 2 + q) * LMAX * NCLS, *st = g.st + ((size_t)b * 2 + q) * (LMAX + 1);
        int32_t steps = 0, wide0 = g.LV, wide1 = 0;
        for (int l = 0; l < g.LV; ++l) {
            int32_t c = 0;
            st[l] = lst[q][l] = steps;
            for (int k = 0; k < NCLS; ++k) {
                kb[l * NCLS + k] = c;
                c += hist[q][l * NCLS + k];
            }
            const int32_t ns = (c + lps - 1) / lps;
            if (ns > 1) {
                wide0 = min(wide0, l);
                wide1 = l + 1;
            }
            steps += ns;
        }
        for (int l = g.LV; l <= LMAX; ++l) st[l] = lst[q][l] = steps;
        // forward: wide levels [0, cut); backward: wide levels [cut, LV)
        cutl[q] = q ? wide0 : wide1;
        if (q == 0) g.nseg[b] = cs;
    }
    __syncthreads();
    // slots of a step: its largest segment, the first one of its class order
    auto slots = [&](int q, int l, int32_t s) {
        int32_t at = (s - lst[q][l]) * lps, k = 0;
        while (k < NCLS - 1 && at >= hist[q][l * NCLS + k]) at -= hist[q][l * NCLS + k++];
        return k == 0 ? lmax[l] : NCLS - k;
    };
    // lengths of the streams, then the steps' places in them
    for (int pass = 0; pass < 2; ++pass) {
        if (threadIdx.x < 2 * (GW + 1)) {
            const int q = threadIdx.x / (GW + 1), w = threadIdx.x % (GW + 1);
            const int32_t c = cutl[q];
            int32_t at = 0, bars = 0;
            if (pass)
                for (int v = 0; v < w; ++v) at += wlen[q][v];
            const int32_t at0 = at;
            const bool nar = w == GW;
            const int la = nar ? (q ? 0 : c) : (q ? c : 0), lb = nar ? (q ? c : g.LV) : (q ? g.LV : c);
            for (int l = la; l < lb; ++l) {
                const int32_t s0 = lst[q][l], s1 = lst[q][l + 1];
                if (s0 == s1) continue;
                for (int32_t s = s0 + (nar ? 0 : w); s < s1; s += nar ? 1 : GW) {
                    const int32_t n = slots(q, l, s);
                    if (pass) {
                        if (bars > 31 || n > 0xffff) atomicOr(g.tot + T_ERR, 4);
                        g.sp_slot[q][po + b + s] = at;
                        g.sp_n[q][po + b + s] = n | (nar ? 0 : min(bars, 31)) << 16;
                    }
                    at += n;
                    bars = 0;
                }
                ++bars;
            }
            if (!pass) {
                wlen[q][w] = at;
            } else {
                int32_t *ws = g.ws + ((size_t)b * 2 + q) * W_N;
                ws[w] = at0;
                if (nar) {
                    ws[W_END] = at;
                    int32_t nl = 0;
                    for (int l = q ? c : 0; l < (q ? g.LV : c); ++l) nl += lst[q][l + 1] > lst[q][l];
                    ws[W_LEVELS] = nl;
                    h[q ? Q_NSB : Q_NSF] = at;
                }
            }
        }
        __syncthreads();
    }
}

// Rows of one part by descending length (lengths from 63 up count as one
// class), stable; per group of 32 rows its padded length and slot offset.
__global__ void __launch_bounds__(GT) k_gr_part_rows(GBuild g)
{
    __shared__ int32_t cls[64], wc[GW][64], sh[GW];
    const int b = blockIdx.x, w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int32_t *h = g.hdr + (size_t)Q_N * b;
    const int32_t nr = h[Q_NR], ro = h[Q_ROFF], ng = pad32(nr) / 32;
    for (int i = threadIdx.x; i < 64; i += GT) cls[i] = 0;
    __syncthreads();
    auto len = [&](int32_t l) {
        const int32_t v = g.i_of_t[ro + l];
        return g.row_ptr[v + 1] - g.row_ptr[v];
    };
    for (int32_t l = threadIdx.x; l < nr; l += GT) atomicAdd(cls + min(len(l), 63), 1);
    __syncthreads();
    if (threadIdx.x == 0) {
        int32_t at = 0;
        for (int k = 63; k >= 0; --k) {
            const int32_t c = cls[k];
            cls[k] = at;
            at += c;
        }
    }
    for (int32_t base = 0; base < nr; base += GT) {
        for (int i = threadIdx.x; i < GW * 64; i += GT) (&wc[0][0])[i] = 0;
        __syncthreads();
        const int32_t l = base + threadIdx.x;
        const int k = l < nr ? min(len(l), 63) : 64;
        const unsigned m = __match_any_sync(0xffffffffu, k);
        const int32_t rank = __popc(m & ((1u << lane) - 1u));
        if (k < 64 && rank == 0) wc[w][k] = __popc(m);
        __syncthreads();
        for (int c = threadIdx.x; c < 64; c += GT) {
            int32_t at = cls[c];
            for (int q = 0; q < GW; ++q) {
                const int32_t x = wc[q][c];
                wc[q][c] = at;
                at += x;
            }
            cls[c] = at;
        }
        __syncthreads();
        if (k < 64) g.perm[ro + wc[w][k] + rank] = (uint16_t)l;
        __syncthreads();
    }
    for (int32_t l = nr + threadIdx.x; l < 32 * ng; l += GT) g.perm[ro + l] = 0xffff;
    __syncthreads();
    int32_t carry = 0;
    for (int32_t gb = 0; gb < ng; gb += GW) {
        const int32_t gi = gb + w;
        int32_t mx = 0;
        if (gi < ng) {
            const int32_t l = g.perm[ro + 32 * gi + lane];
            mx = l != 0xffff ? len(l) : 0;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        }
        int32_t tot;
        const int32_t ex = gscan<GT>(lane == 0 ? mx : 0, sh, &tot);
        if (gi < ng && lane == 0) {
            g.glen[ro / 32 + gi] = mx;
            g.gso[ro / 32 + gi] = carry + ex;
        }
        carry += tot;
    }
    if (threadIdx.x == 0) g.rh[R_N * b + R_NS] = carry;
}

// The rows of other parts that a part's rows name ("halo"): marked in a
// bitmap, then counted word by word.
__device__ __forceinline__ int32_t slot_col(const GBuild &g, int32_t s)
{
    return g.col32 ? __float_as_int(g.col32[s].y) : g.col[s];
}
__global__ void __launch_bounds__(GT) k_gr_halo_mark(GBuild g)
{
    const int b = blockIdx.x;
    const int32_t *h = g.hdr + (size_t)Q_N * b;
    const int32_t nr = h[Q_NR], ro = h[Q_ROFF];
    uint32_t *hb = g.hb + (size_t)b * g.NRW;
    for (int32_t l = blockIdx.y * GT + threadIdx.x; l < nr; l += GT * gridDim.y) {
        const int32_t v = g.i_of_t[ro + l];
        for (int32_t s = g.row_ptr[v]; s < g.row_ptr[v + 1]; ++s) {
            const int32_t t = g.t_of_i[slot_col(g, s)];
            if (t < ro || t >= ro + nr) {
                atomicOr(hb + (t >> 5), 1u << (t & 31));
                g.xflag[t] = 1;
            }
        }
    }
}
__global__ void __launch_bounds__(1024) k_gr_halo_count(GBuild g)
{
    __shared__ int32_t sh[32];
    const int b = blockIdx.x;
    const uint32_t *hb = g.hb + (size_t)b * g.NRW;
    int32_t *hp = g.hpre + (size_t)b * g.NRW;
    const int32_t nw = g.tot[T_NR] / 32;
    int32_t carry = 0;
    for (int32_t base = 0; base < nw; base += 4096) {
        int32_t c[4], s = 0;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int32_t w = base + 4 * threadIdx.x + u;
            c[u] = w < nw ? __popc(hb[w]) : 0;
            s += c[u];
        }
        int32_t tot;
        int32_t at = carry + gscan<1024>(s, sh, &tot);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int32_t w = base + 4 * threadIdx.x + u;
            if (w < nw) hp[w] = at;
            at += c[u];
        }
        carry += tot;
    }
    if (threadIdx.x == 0) g.rh[R_N * b + R_NH] = carry;
}
__global__ void __launch_bounds__(256) k_gr_row_offsets(GBuild g)
{
    __shared__ int32_t sh[8];
    const int b = threadIdx.x;
    int32_t *rh = g.rh + R_N * b, *t = g.rh + R_N * g.P, total;
    if (b < R_N) t[b] = 0;
    int32_t o = gscan<256>(b < g.P ? rh[R_NS] : 0, sh, &total);
    if (b < g.P) rh[R_SLOT] = o;
    if (b == 0) t[0] = total;
    o = gscan<256>(b < g.P ? rh[R_NH] : 0, sh, &total);
    if (b < g.P) {
        rh[R_HOFF] = o;
        atomicMax(t + 2, rh[R_NH]);
    }
    if (b == 0) t[1] = total;
}
__global__ void __launch_bounds__(GT) k_gr_halo_list(GBuild g)
{
    const int b = blockIdx.x;
    const uint32_t *hb = g.hb + (size_t)b * g.NRW;
    const int32_t *hp = g.hpre + (size_t)b * g.NRW;
    int32_t *hl = g.hl + g.rh[R_N * b + R_HOFF];
    const int32_t nw = g.tot[T_NR] / 32;
    for (int32_t w = blockIdx.y * GT + threadIdx.x; w < nw; w += GT * gridDim.y) {
        uint32_t m = hb[w];
        int32_t at = hp[w];
        while (m) {
            const int k = __ffs(m) - 1;
            m &= m - 1;
            hl[at++] = 32 * w + k;
        }
    }
}

// A slot: 32 records, then the blocks in planes of 32 values (all nine
// entries, or the lane's row).  rec = source | receiver << 13 | block barriers
// before the slot << 26.  Idle lanes work on a spare cell behind the vectors
// with a zero block.
template <typename T>
struct SlotSize;
template <>
struct SlotSize<float> {
    static constexpr int B = 128 + 9 * 128, LPS = 32;
};
template <>
struct SlotSize<double> {
    static constexpr int B = 128 + 3 * 256, LPS = 10;
};
template <typename T>
__global__ void __launch_bounds__(GT) k_gr_program(GBuild g)
{
    __shared__ uint16_t wc[GW][LMAX * NCLS];
    __shared__ int32_t base_s[LMAX * NCLS];
    constexpr int B = SlotSize<T>::B, LPS = SlotSize<T>::LPS, R = LPS == 32 ? 1 : 3;
    const int b = blockIdx.x, q = blockIdx.y, w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int32_t *h = g.hdr + (size_t)Q_N * b;
    const int32_t so = h[Q_SOFF], nv = h[Q_NV], nr = h[Q_NR], nt = g.tot[T_NT], po = h[Q_POFF], nd = nr + h[Q_NZ];
    const int32_t *vm = g.vm + (size_t)b * nt;
    const int32_t *kb = g.kb + ((size_t)b * 2 + q) * LMAX * NCLS, *st = g.st + ((size_t)b * 2 + q) * (LMAX + 1);
    const int32_t *sslot = g.sp_slot[q] + po + b, *sn = g.sp_n[q] + po + b;
    const int32_t slot0 = h[q ? Q_SB : Q_SF], nsteps = st[LMAX];
    char *prog = g.prog[q] + (size_t)B * slot0;
    int32_t *msrc = g.msrc[q] + 32 * (size_t)slot0;
    auto rec = [&](int32_t slot, int32_t ln) -> uint32_t & { return reinterpret_cast<uint32_t *>(prog + (size_t)B * slot)[ln]; };
    for (int32_t s = w; s < nsteps; s += GW) {
        const int32_t a = sslot[s], n = sn[s] & 0xffff, bars = sn[s] >> 16;
        for (int32_t j = 0; j < n; ++j) {
            rec(a + j, lane) = (uint32_t)nd | (uint32_t)nd << 13 | (j == 0 ? (uint32_t)bars << 26 : 0u);
            msrc[32 * (a + j) + lane] = -1;
        }
    }
    const int nk = g.LV * NCLS;
    for (int k = threadIdx.x; k < nk; k += GT) base_s[k] = kb[k];
    const int32_t items = q ? nv : g.nseg[b];
    for (int32_t ib = 0; ib < items; ib += GT) {
        for (int i = threadIdx.x; i < GW * LMAX * NCLS; i += GT) (&wc[0][0])[i] = 0;
        __syncthreads();
        const int32_t i = ib + threadIdx.x;
        int key = LMAX * NCLS;
        int32_t p0 = 0, n = 0, dst = 0;
        if (i < items) {
            if (q) {
                const int32_t t = g.sp[so + i];
                p0 = g.pr_ptr[t];
                n = g.pr_ptr[t + 1] - p0;
                dst = i;
                if (n > 0) key = (g.LV - 1 - level_of(g.lp, g.LV, t)) * NCLS + seg_class(n);
            } else {
                key = g.sgk[po + i];
                dst = g.sgd[po + i];
                n = g.sgn[po + i];
                p0 = g.sgf[po + i];
            }
        }
        const unsigned m = __match_any_sync(0xffffffffu, key);
        const int32_t rank = __popc(m & ((1u << lane) - 1u));
        if (key < nk && rank == 0) wc[w][key] = (uint16_t)__popc(m);
        __syncthreads();
        for (int k = threadIdx.x; k < nk; k += GT) {
            int32_t at = base_s[k];
            for (int v = 0; v < GW; ++v) {
                const int32_t x = wc[v][k];
                wc[v][k] = (uint16_t)at;
                at += x;
            }
            base_s[k] = at;
        }
        __syncthreads();
        if (key < nk) {
            const int32_t at = wc[w][key] + rank, s = st[key / NCLS] + at / LPS, ln = (at % LPS) * R;
            const int32_t a = sslot[s], ns = sn[s] & 0xffff;
            for (int32_t j = 0; j < ns; ++j) {
                int32_t src = dst, p = -1;
                if (j < n) {
                    p = q ? p0 + j : g.plist[po + p0 + j];
                    src = q ? pair_dst(g, b, nr, vm, p) : g.lpos[g.pos[g.pr_c[p]]];
                }
                for (int c = 0; c < R; ++c) {
                    uint32_t &r = rec(a + j, ln + c);
                    r = (r & 0xfc000000u) | (uint32_t)src | (uint32_t)dst << 13;
                    msrc[32 * (a + j) + ln + c] = p;
                }
            }
        }
        __syncthreads();
    }
}

// ---- the top.  Its forest solve is z = X^T D^-1 X r with X = L^-1 of the top
// alone: row j has an entry for every vertex whose elimination reaches j, the
// column of a vertex one for itself and for each of its receivers' columns.  A
// vertex has two receivers at most and meets two at a time on its way up, so
// columns are short (6 or 7 entries, 11 at most, at 1e4 to 1e6 cells).  A part
// forms the rows that its outputs' columns name (30 of some 340) and these
// columns: a third of the work of the same outputs' rows of the inverse
// X^T D^-1 X, which this replaces because in the inverse the 1 / gamma0 of the
// roots swamps the rest (rounded to FP32 it is no longer positive definite:
// sheets with gamma0 = 1e-10 broke down).  In this form the operator is
// positive definite however X is rounded.
// Whole steps with the inverse's rows and so: FP64 lattice of 1e4 cells 7.7 and
// 7.7 ms, MIXED 1e5 13.0 and 13.4, 1e6 59.0 and 59.4, 48 instances 13.8 and 12.6.

// One lane per component of a column, by its elimination steps in FP64.
__global__ void k_gr_cols(GBuild g, const double *__restrict__ L)
{
    const int32_t k = blockIdx.x * blockDim.x + threadIdx.x, i = k / 3, c = k % 3;
    if (g.tot[T_ERR] || i >= g.tot[T_NT]) return;
    constexpr int W = 4;
    int32_t f[W], n = 1, len = 0;   // vertices met, by position, and X's column c in their rows
    double y[W][3] = {};
    f[0] = g.sp[g.hdr[(size_t)Q_N * g.P + Q_SOFF] + i];
    y[0][0] = c == 0; y[0][1] = c == 1; y[0][2] = c == 2;
    bool bad = false;
    while (n > 0 && !bad) {
        int m = 0;
        for (int a = 1; a < n; ++a)
            if (f[a] < f[m]) m = a;
        const int32_t t = f[m];
        const double y0 = y[m][0], y1 = y[m][1], y2 = y[m][2];
        --n;
        f[m] = f[n];
        for (int r = 0; r < 3; ++r) y[m][r] = y[n][r];
        if (len == CMAX) {
            bad = true;
            break;
        }
        const int32_t j = g.lpos[t];
        double *x = g.cx + ((size_t)i * CMAX + len) * 9 + c;
        x[0] = y0; x[3] = y1; x[6] = y2;
        if (c == 0) {
            g.cidx[(size_t)i * CMAX + len] = j;
            atomicAdd(g.rlen + j, 1);
        }
        ++len;
        for (int32_t p = g.pr_ptr[t]; p < g.pr_ptr[t + 1]; ++p) {
            const int32_t u = g.pos[g.pr_q[p]];
            int a = 0;
            while (a < n && f[a] != u) ++a;
            if (a == W) {
                bad = true;
                break;
            }
            if (a == n) {
                f[n] = u;
                y[n][0] = y[n][1] = y[n][2] = 0.0;
                ++n;
            }
            const double *l = L + 9 * (size_t)p;
            for (int r = 0; r < 3; ++r) y[a][r] = fma(-l[3 * r + 2], y2, fma(-l[3 * r + 1], y1, fma(-l[3 * r], y0, y[a][r])));
        }
    }
    if (c == 0) g.clen[i] = len;
    if (bad) atomicOr(g.tot + T_ERR, 8);
}
// where the rows and columns start (padded to 8 entries)
__global__ void __launch_bounds__(1024) k_gr_top_offsets(GBuild g)
{
    __shared__ int32_t sh[32];
    const int32_t nt = min(g.tot[T_NT], NTOP);
    int32_t cr = 0, cc = 0;
    for (int32_t base = 0; base < nt; base += 1024) {
        const int32_t i = base + threadIdx.x;
        int32_t tr, tc;
        const int32_t er = gscan<1024>(i < nt ? pad8(g.rlen[i]) : 0, sh, &tr);
        const int32_t ec = gscan<1024>(i < nt ? pad8(g.clen[i]) : 0, sh, &tc);
        if (i < nt) {
            g.rptr[i] = cr + er;
            g.cptr[i] = cc + ec;
        }
        cr += tr;
        cc += tc;
    }
    if (threadIdx.x == 0) {
        g.tot[T_RE] = cr;
        g.tot[T_CE] = cc;
    }
}
// A part's share: its outputs (the top vertices that it reaches, then those
// that it owns) and the rows that their columns name, the long ones first.  On
// chip the part's rows, then its columns, are packed ("local" starts).
//   alist: row, start, local start, length
//   outs:  column's start, local start, length
template <bool FILL>
__global__ void __launch_bounds__(GT) k_gr_part_top(GBuild g)
{
    __shared__ int32_t sh[GW];
    __shared__ uint8_t in[NTOP];
    const int b = blockIdx.x;
    int32_t *h = g.hdr + (size_t)Q_N * b;
    if (g.tot[T_ERR]) return;   // (nothing of this launch writes it)
    const int32_t nt = g.tot[T_NT], nz = h[Q_NZ], nout = nz + h[Q_NR] - h[Q_NV], t0 = h[Q_T0];
    const int32_t *vm = g.vm + (size_t)b * nt;
    int4 *outs = FILL ? g.outs + h[Q_ZOFF] + t0 : nullptr;
    for (int32_t i = threadIdx.x; i < nt; i += GT) in[i] = 0;
    __syncthreads();
    int32_t xc = 0;
    for (int32_t base = 0; base < nt; base += GT) {
        const int32_t i = base + threadIdx.x;
        const bool own = i < nt && i >= t0 && i - t0 < nout - nz;
        const bool reach = i < nt && vm[i] != 0;
        int32_t n = 0;
        if (own || reach) {
            n = g.clen[i];
            for (int32_t k = 0; k < n; ++k) in[g.cidx[(size_t)i * CMAX + k]] = 1;
        }
        // a vertex that is reached and owned has two outputs
        const int32_t e = pad8(n) * ((own ? 1 : 0) + (reach ? 1 : 0));
        int32_t tot;
        const int32_t at = xc + gscan<GT>(e, sh, &tot);
        if (FILL) {
            const int32_t st = (own || reach) ? g.tot[T_RE] + g.cptr[i] : 0;
            if (reach) outs[vm[i] - 1] = make_int4(st, h[Q_XR] + at, n, 0);
            if (own) outs[nz + i - t0] = make_int4(st, h[Q_XR] + at + (reach ? pad8(n) : 0), n, 0);
        }
        xc += tot;
    }
    __syncthreads();
    int32_t nl = 0, ns = 0, xr = 0;
    for (int32_t base = 0; base < nt; base += GT) {
        const int32_t j = base + threadIdx.x;
        const int32_t n = j < nt && in[j] ? g.rlen[j] : 0;
        int32_t tl, ts, tx;
        const int32_t l = nl + gscan<GT>(n > TLONG, sh, &tl), k = ns + gscan<GT>(n > 0 && n <= TLONG, sh, &ts),
                      x0 = xr + gscan<GT>(pad8(n), sh, &tx);
        if (FILL && n > 0) g.alist[h[Q_AOFF] + (n > TLONG ? l : h[Q_NL] + k)] = make_int4(j, g.rptr[j], x0, n);
        nl += tl;
        ns += ts;
        xr += tx;
    }
    if (!FILL && threadIdx.x == 0) {
        h[Q_NA] = nl + ns;
        h[Q_NL] = nl;
        h[Q_XR] = xr;
        h[Q_XC] = xc;
    }
}
// X by rows (a block each: the columns that hold it, in order) and by columns:
// planes of the nine entries over the padded length
template <typename T>
__global__ void __launch_bounds__(128) k_gr_top_fill(GBuild g, T *X)
{
    __shared__ int32_t sh[4];
    const int32_t nt = g.tot[T_NT], re = g.tot[T_RE];
    for (int32_t j = blockIdx.x; j < nt; j += gridDim.x) {
        const int32_t st = g.rptr[j], lp = pad8(g.rlen[j]);
        int32_t done = 0;
        for (int32_t base = 0; base <= j; base += 128) {
            const int32_t i = base + threadIdx.x;
            int32_t k = -1;
            if (i <= j)
                for (int32_t e = g.clen[i] - 1; e >= 0 && k < 0; --e)
                    if (g.cidx[(size_t)i * CMAX + e] == j) k = e;
            int32_t tot;
            const int32_t at = done + gscan<128>(k >= 0 ? 1 : 0, sh, &tot);
            if (k >= 0) {
                g.xi[st + at] = i;
                const double *x = g.cx + ((size_t)i * CMAX + k) * 9;
                T *o = X + 9 * (size_t)st + at;
#pragma unroll
                for (int a = 0; a < 9; ++a) o[(size_t)a * lp] = (T)x[a];
            }
            done += tot;
        }
        const int32_t cs = re + g.cptr[j], n = g.clen[j], lc = pad8(n);
        for (int32_t e = threadIdx.x; e < n; e += 128) {
            g.xi[cs + e] = g.cidx[(size_t)j * CMAX + e];
            const double *x = g.cx + ((size_t)j * CMAX + e) * 9;
            T *o = X + 9 * (size_t)cs + e;
#pragma unroll
            for (int a = 0; a < 9; ++a) o[(size_t)a * lc] = (T)x[a];
        }
    }
}

// Slots of the parts' sums for the top, grouped by top vertex, parts ascending.
__global__ void __launch_bounds__(1024) k_gr_slots(GBuild g)
{
    __shared__ int32_t sh[32];
    const int32_t nt = g.tot[T_NT];
    int32_t carry = 0;
    for (int32_t base = 0; base < nt; base += 1024) {
        const int32_t i = base + threadIdx.x;
        int32_t c = 0;
        if (i < nt) {
#pragma unroll 8
            for (int32_t b = 0; b < g.P; ++b) c += g.vm[(size_t)b * nt + i] != 0;
        }
        int32_t tot;
        const int32_t ex = gscan<1024>(c, sh, &tot);
        if (i < nt) {
            g.tlk[i] = carry + ex;
            int32_t at = carry + ex;
#pragma unroll 8
            for (int32_t b = 0; b < g.P; ++b) {
                const int32_t k = g.vm[(size_t)b * nt + i];
                if (k) g.zslot[g.hdr[(size_t)Q_N * b + Q_ZOFF] + k - 1] = at++;
            }
        }
        carry += tot;
    }
    if (threadIdx.x == 0) g.tlk[nt] = carry;
}

// ---- numeric layout
// D^-1 in groups of 32 rows, one plane of 32 values per entry (a source of
// -1 gives a zero block).  FP32: times a power of two where gamma0 is far from
// 1.  PCG's iterates do not depend on the preconditioner's size, but r^T z and
// p^T q do (|r|^2 / gamma0 and less), and FP32 sums of them leave FP32's range
// where FP64 ones do not: coefficients of 1e-34 broke down.  With 1 / gamma0
// held to 2^80 at most and 2^-40 at least, both stay inside for coefficients
// from 1e-34 to 1e34.  (A gamma0 that is small beside the contacts alone needs no
// scale, and a small one does it no harm.)
template <typename T>
double pivot_scale(const sgp_matrix *M)
{
    const int e = std::ilogb(M->gamma0), k = e < -80 ? e + 80 : e > 40 ? e - 40 : 0;
    return sizeof(T) == 4 ? std::ldexp(1.0, k) : 1.0;
}
template <typename T>
__global__ void k_gr_pivots(int32_t cnt, const int32_t *__restrict__ src, const double *__restrict__ from, double scale,
                            T *to)
{
    int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= cnt) return;
    const int32_t s = src[i];
    T *o = to + (size_t)(i >> 5) * 192 + (i & 31);
#pragma unroll
    for (int a = 0; a < 6; ++a) o[32 * a] = s >= 0 ? (T)(scale * from[(size_t)6 * s + a]) : T(0);
}
// The programs' blocks: -L of the lane's pair, transposed in the backward
// program (TR); FP64 lanes hold one row.
template <typename T, bool TR>
__global__ void k_gr_blocks(int32_t lanes, const int32_t *__restrict__ src, const double *__restrict__ L, char *prog)
{
    int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= lanes) return;
    const int32_t s = src[i], ln = i & 31;
    T *o = reinterpret_cast<T *>(prog + (size_t)(i >> 5) * SlotSize<T>::B + 128) + ln;
    if (sizeof(T) == 4) {
#pragma unroll
        for (int a = 0; a < 9; ++a) o[32 * (TR ? 3 * (a % 3) + a / 3 : a)] = s >= 0 ? (T)-L[(size_t)9 * s + a] : T(0);
    } else {
        const int r = ln % 3;
#pragma unroll
        for (int c = 0; c < 3; ++c) o[32 * c] = s >= 0 ? (T)-L[(size_t)9 * s + (TR ? 3 * c + r : 3 * r + c)] : T(0);
    }
}

// The matrix's rows of every part, slot by slot in groups of 32 rows; the
// column is the local row inside the part, rows + halo index outside it, or
// -1 - row when the halo is read from memory.  Padding slots hold a zero
// block and the row's own column.
__device__ __forceinline__ int32_t sell_col(const GBuild &g, int b, int32_t t, int32_t ro, int32_t nr)
{
    const int32_t l = t - ro;
    if (l >= 0 && l < nr) return l;
    if (!g.halo) return -1 - t;
    const size_t w = (size_t)b * g.NRW + (t >> 5);
    return nr + g.hpre[w] + __popc(g.hb[w] & ((1u << (t & 31)) - 1u));
}
__global__ void __launch_bounds__(GT) k_gr_sell32(GBuild g, const float4 *__restrict__ a, const float2 *__restrict__ bb,
                                                  float4 *at, float2 *bt)
{
    const int32_t *h = g.hdr + (size_t)Q_N * blockIdx.x;
    const int32_t ro = h[Q_ROFF], nr = h[Q_NR], ng = pad32(nr) / 32, lane = threadIdx.x & 31;
    for (int32_t gi = blockIdx.y * GW + (threadIdx.x >> 5); gi < ng; gi += GW * gridDim.y) {
        const int32_t l = g.perm[ro + 32 * gi + lane];
        const int32_t v = l != 0xffff ? g.i_of_t[ro + l] : -1;
        const int32_t b0 = v >= 0 ? g.row_ptr[v] : 0, n = v >= 0 ? g.row_ptr[v + 1] - b0 : 0;
        const size_t o = (size_t)(g.rh[R_N * blockIdx.x + R_SLOT] + g.gso[ro / 32 + gi]) * 32 + lane;
        const int32_t gl = g.glen[ro / 32 + gi];
        for (int32_t k = 0; k < gl; ++k) {
            float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
            float2 y = make_float2(0.f, __int_as_float(l != 0xffff ? l : 0));
            if (k < n) {
                x = a[b0 + k];
                y = bb[b0 + k];
                y.y = __int_as_float(sell_col(g, blockIdx.x, g.t_of_i[__float_as_int(y.y)], ro, nr));
            }
            at[o + 32 * (size_t)k] = x;
            bt[o + 32 * (size_t)k] = y;
        }
    }
}
__global__ void __launch_bounds__(GT) k_gr_sell64(GBuild g, const double *__restrict__ blk,
                                                  const int32_t *__restrict__ col, double2 *bt, int32_t *ct)
{
    const int32_t *h = g.hdr + (size_t)Q_N * blockIdx.x;
    const int32_t ro = h[Q_ROFF], nr = h[Q_NR], ng = pad32(nr) / 32, lane = threadIdx.x & 31;
    for (int32_t gi = blockIdx.y * GW + (threadIdx.x >> 5); gi < ng; gi += GW * gridDim.y) {
        const int32_t l = g.perm[ro + 32 * gi + lane];
        const int32_t v = l != 0xffff ? g.i_of_t[ro + l] : -1;
        const int32_t b0 = v >= 0 ? g.row_ptr[v] : 0, n = v >= 0 ? g.row_ptr[v + 1] - b0 : 0;
        const size_t o = (size_t)(g.rh[R_N * blockIdx.x + R_SLOT] + g.gso[ro / 32 + gi]);
        const int32_t gl = g.glen[ro / 32 + gi];
        for (int32_t k = 0; k < gl; ++k) {
            double2 x[3] = {{0.0, 0.0}, {0.0, 0.0}, {0.0, 0.0}};
            int32_t j = l != 0xffff ? l : 0;
            if (k < n) {
                const double2 *q = reinterpret_cast<const double2 *>(blk + 6 * (size_t)(b0 + k));
                x[0] = q[0]; x[1] = q[1]; x[2] = q[2];
                j = sell_col(g, blockIdx.x, g.t_of_i[col[b0 + k]], ro, nr);
            }
            const size_t r = o + k;
#pragma unroll
            for (int c = 0; c < 3; ++c) bt[(3 * r + c) * 32 + lane] = x[c];
            ct[r * 32 + lane] = j;
        }
    }
}

// Every index the solve uses lies inside its arrays (checked once per
// build; a failure is a library bug and the build reports it).
__global__ void __launch_bounds__(GT) k_gr_check(GBuild g)
{
    const int b = blockIdx.x;
    int bad = 0;
    const int32_t nt = g.tot[T_NT], xe = g.tot[T_RE] + g.tot[T_CE];
    const int32_t *h = g.hdr + (size_t)Q_N * b;
    const int32_t nv = h[Q_NV], nr = h[Q_NR], nz = h[Q_NZ], nd = nr + nz, ro = h[Q_ROFF], nout = nz + nr - nv,
                  xl = h[Q_XR] + h[Q_XC];
    for (int q = 0; q < 2; ++q) {
        const int32_t ns = h[q ? Q_NSB : Q_NSF], B = g.lps == 32 ? SlotSize<float>::B : SlotSize<double>::B;
        const char *prog = g.prog[q] + (size_t)B * h[q ? Q_SB : Q_SF];
        for (int32_t i = threadIdx.x; i < 32 * ns; i += GT) {
            const uint32_t r = reinterpret_cast<const uint32_t *>(prog + (size_t)B * (i >> 5))[i & 31];
            if ((int32_t)(r & 8191) > nd || (int32_t)(r >> 13 & 8191) > nd) bad = 32;
        }
        const int32_t *ws = g.ws + ((size_t)b * 2 + q) * W_N;
        for (int k = threadIdx.x; k < W_END; k += GT)
            if (ws[k] < 0 || ws[k] > ws[k + 1] || ws[k + 1] > ns) bad = 64;
    }
    // the top: every row and column that the part reads, and its entries
    auto entries = [&](int32_t st, int32_t n, int32_t lp, int32_t loc) {
        bool in = n >= 0 && n <= lp && st >= 0 && st + lp <= xe && loc >= 0 && loc + lp <= xl;
        for (int32_t e = 0; in && e < n; ++e) in = g.xi[st + e] >= 0 && g.xi[st + e] < nt;
        return in;
    };
    for (int32_t k = threadIdx.x; k < h[Q_NA]; k += GT) {
        const int4 t = g.alist[h[Q_AOFF] + k];
        if (t.x < 0 || t.x >= nt || !entries(t.y, t.w, pad8(t.w), t.z)) bad = 256;
    }
    for (int32_t z = threadIdx.x; z < nout; z += GT) {
        const int4 t = g.outs[h[Q_ZOFF] + h[Q_T0] + z];
        if (!entries(t.x, t.z, pad8(t.z), t.y)) bad = 512;
    }
    for (int32_t z = threadIdx.x; z < nz; z += GT) {
        const int32_t k = g.zslot[h[Q_ZOFF] + z];
        if (k < 0 || k >= g.tlk[nt]) bad = 512;
    }
    for (int32_t l = threadIdx.x; l < pad32(nr); l += GT) {
        const int32_t q = g.perm[ro + l];
        if (q != 0xffff && q >= nr) bad = 1024;
    }
    if (g.halo)
        for (int32_t k = threadIdx.x; k < g.rh[R_N * b + R_NH]; k += GT) {
            const int32_t t = g.hl[g.rh[R_N * b + R_HOFF] + k];
            if (t < 0 || t >= g.tot[T_NR] || !g.xflag[t]) bad = 2048;
        }
    if (bad) atomicOr(g.tot + T_ERR, bad);
}

// ------------------------------------------------------------------ solve
template <typename T>
struct Mat;
template <>
struct Mat<float> {
    const float4 *a;
    const float2 *b;
};
template <>
struct Mat<double> {
    const double2 *a;
    const int32_t *b;
};

// Placement: byte offsets into shared memory (-1: the array stays in global
// memory).
struct GridPlace {
    int32_t o_p, o_w, o_t, o_u, o_misc, o_X, o_tab, o_nar[2], o_all[2], o_D, o_r, o_x, o_perm, o_hl;
    int32_t xe;   // entries of X on chip (o_X: their blocks, then their indices)
    int32_t bytes;
};
struct GridArgs {
    int32_t P, nt, x_given, timing, halo, nslots;
    const int32_t *grp;        // per part: first and end part of its system, the system (NULL: one system)
    const double *gtol2;       // per system: tol^2, or below 0 for none to solve (NULL: tol2 for all)
    const int32_t *hdr, *rh, *ws, *glen, *gso, *i_of_t, *zslot, *tlk, *hl;
    const int4 *alist, *outs;   // the top: see k_gr_part_top
    const int32_t *xi;
    const char *prog[2];
    const uint16_t *perm;
    const uint8_t *xflag;
    const void *D, *X, *tD;    // pivots, the top's X and pivots, of the solve's type
    const void *jac;           // block-Jacobi inverses, part order planes
    const void *ma, *mb;       // the matrix's rows
    const void *F;             // right-hand side, internal order
    void *x;                   // iterate, internal order
    void *pg, *r, *xt;         // part-order workspaces
    unsigned long long *pk, *px, *lx;   // packets: sums; p of exported rows; sums for the top, then the top's r
    double gamma0, tol2, tolE2, mu;
    long long maxit;
    int stopE;
    int *err;
    int *gave_up;              // a forest solve alone: the context's word (host memory) for a wait that gave up
    unsigned skew;             // block 0 numbers its packets from here (0; tests: waits that run out)
    Scal *sc;
    unsigned long long *ns;    // phase times (timing)
    GridPlace pl;
};

// Vectors addressed at random live in shared memory, VB bytes per cell: FP64
// 24; FP32 16 (one load per cell), or 12 where that makes room for the halo
// (1e6 cells: the product's gathers of other parts' rows then stay on chip).
template <typename T, int VB>
struct V3;
template <>
struct V3<float, 16> {
    static __device__ __forceinline__ void ld(uint32_t a, float *v)
    {
        float pad;
        asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(pad) : "r"(a) : "memory");
        asm volatile("" ::"f"(pad));
    }
    static __device__ __forceinline__ void st(uint32_t a, const float *v)
    {
        asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(a), "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(0.f) : "memory");
    }
};
template <>
struct V3<float, 12> {
    static __device__ __forceinline__ void ld(uint32_t a, float *v)
    {
        asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v[0]) : "r"(a) : "memory");
        asm volatile("ld.shared.f32 %0, [%1+4];" : "=f"(v[1]) : "r"(a) : "memory");
        asm volatile("ld.shared.f32 %0, [%1+8];" : "=f"(v[2]) : "r"(a) : "memory");
    }
    static __device__ __forceinline__ void st(uint32_t a, const float *v)
    {
        asm volatile("st.shared.f32 [%0], %1;" ::"r"(a), "f"(v[0]) : "memory");
        asm volatile("st.shared.f32 [%0+4], %1;" ::"r"(a), "f"(v[1]) : "memory");
        asm volatile("st.shared.f32 [%0+8], %1;" ::"r"(a), "f"(v[2]) : "memory");
    }
};
template <>
struct V3<double, 24> {
    static __device__ __forceinline__ void ld(uint32_t a, double *v)
    {
        asm volatile("ld.shared.f64 %0, [%1];" : "=d"(v[0]) : "r"(a) : "memory");
        asm volatile("ld.shared.f64 %0, [%1+8];" : "=d"(v[1]) : "r"(a) : "memory");
        asm volatile("ld.shared.f64 %0, [%1+16];" : "=d"(v[2]) : "r"(a) : "memory");
    }
    static __device__ __forceinline__ void st(uint32_t a, const double *v)
    {
        asm volatile("st.shared.f64 [%0], %1;" ::"r"(a), "d"(v[0]) : "memory");
        asm volatile("st.shared.f64 [%0+8], %1;" ::"r"(a), "d"(v[1]) : "memory");
        asm volatile("st.shared.f64 [%0+16], %1;" ::"r"(a), "d"(v[2]) : "memory");
    }
};

template <typename T>
struct Cell;   // one component of a cell
template <>
struct Cell<float> {
    static __device__ __forceinline__ void st(uint32_t a, float v) { asm volatile("st.shared.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory"); }
};
template <>
struct Cell<double> {
    static __device__ __forceinline__ void st(uint32_t a, double v) { asm volatile("st.shared.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory"); }
};

// Sums of products.  FP64: fused multiply-adds.  FP32: the product and the
// running sum each as a pair of floats (exact product, compensated sum), so
// that no thread spends FP64 issue slots (1/64 of the FP32 rate) on them and
// the sum is as good as an FP64 one.  warp() leaves the warp's sum in lane 0.
template <typename T>
struct Acc;
template <>
struct Acc<double> {
    double v = 0.0;
    __device__ __forceinline__ void mul(double a, double b) { v = fma(a, b, v); }
    __device__ __forceinline__ void warp()
    {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    }
    __device__ __forceinline__ double pair() const { return v; }
    __device__ __forceinline__ void join(double x) { v += x; }
};
template <>
struct Acc<float> {
    float h = 0.f, l = 0.f;
    __device__ __forceinline__ void add(float x, float e)
    {
        const float s = __fadd_rn(h, x), t = __fsub_rn(s, h);
        const float d = __fadd_rn(__fsub_rn(h, __fsub_rn(s, t)), __fsub_rn(x, t));
        h = s;
        l = __fadd_rn(l, __fadd_rn(d, e));
    }
    __device__ __forceinline__ void mul(float a, float b)
    {
        const float p = __fmul_rn(a, b);
        add(p, __fmaf_rn(a, b, -p));
    }
    __device__ __forceinline__ void warp()
    {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const float oh = __shfl_xor_sync(0xffffffffu, h, o), ol = __shfl_xor_sync(0xffffffffu, l, o);
            add(oh, ol);
        }
    }
    __device__ __forceinline__ float2 pair() const { return make_float2(h, l); }
    __device__ __forceinline__ void join(float2 x) { add(x.x, x.y); }
};
template <typename T>
struct Part;   // a partial sum in shared memory and in packets
template <>
struct Part<float> {
    using type = float2;
    static __device__ __forceinline__ void split(float2 v, unsigned &a, unsigned &b)
    {
        a = __float_as_uint(v.x);
        b = __float_as_uint(v.y);
    }
    static __device__ __forceinline__ float2 unite(unsigned a, unsigned b)
    {
        return make_float2(__uint_as_float(a), __uint_as_float(b));
    }
};
template <>
struct Part<double> {
    using type = double;
    static __device__ __forceinline__ void split(double v, unsigned &a, unsigned &b)
    {
        const unsigned long long x = (unsigned long long)__double_as_longlong(v);
        a = (unsigned)x;
        b = (unsigned)(x >> 32);
    }
    static __device__ __forceinline__ double unite(unsigned a, unsigned b)
    {
        return __longlong_as_double((long long)((unsigned long long)b << 32 | a));
    }
};

__device__ __forceinline__ unsigned long long now_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
__device__ __forceinline__ void ld_words(const unsigned long long *p, unsigned long long &a, unsigned long long &b)
{
    asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "l"(p) : "memory");
}
__device__ __forceinline__ unsigned long long ld_word(const unsigned long long *p)
{
    unsigned long long a;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(a) : "l"(p) : "memory");
    return a;
}
__device__ __forceinline__ void st_words(unsigned long long *p, unsigned long long a, unsigned long long b)
{
    asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(p), "l"(a), "l"(b) : "memory");
}
__device__ __forceinline__ void st_word(unsigned long long *p, unsigned long long a)
{
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(a) : "memory");
}

// Values that other blocks wait for travel in packets: 8-byte words of the
// exchange's number (high half) and 32 bits of data, so that a value and its
// arrival are one memory access: no fence, no separate flag, and a torn read
// is seen as such.  A cell's vector takes 4 words in FP32 (the last unused)
// and 6 in FP64.
template <typename T>
struct Pkt;
template <>
struct Pkt<float> {
    static constexpr int W = 4;
    static __device__ __forceinline__ void put(unsigned long long *p, unsigned long long e, const float *v)
    {
        st_words(p, e | __float_as_uint(v[0]), e | __float_as_uint(v[1]));
        st_word(p + 2, e | __float_as_uint(v[2]));
    }
    static __device__ __forceinline__ bool get(const unsigned long long *p, unsigned ep, float *v)
    {
        unsigned long long a, b, c;
        ld_words(p, a, b);
        c = ld_word(p + 2);
        v[0] = __uint_as_float((unsigned)a);
        v[1] = __uint_as_float((unsigned)b);
        v[2] = __uint_as_float((unsigned)c);
        return (unsigned)(a >> 32) == ep && (unsigned)(b >> 32) == ep && (unsigned)(c >> 32) == ep;
    }
};
template <>
struct Pkt<double> {
    static constexpr int W = 6;
    static __device__ __forceinline__ void put(unsigned long long *p, unsigned long long e, const double *v)
    {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const unsigned long long x = (unsigned long long)__double_as_longlong(v[c]);
            st_words(p + 2 * c, e | (x & 0xffffffffull), e | (x >> 32));
        }
    }
    static __device__ __forceinline__ bool get(const unsigned long long *p, unsigned ep, double *v)
    {
        bool ok = true;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            unsigned long long a, b;
            ld_words(p + 2 * c, a, b);
            v[c] = __longlong_as_double((long long)((a & 0xffffffffull) | (b << 32)));
            ok = ok && (unsigned)(a >> 32) == ep && (unsigned)(b >> 32) == ep;
        }
        return ok;
    }
};
constexpr int WAIT_MAX = 1 << 21;   // polls: about two seconds
// gives up (returns true) after WAIT_MAX polls, or when another block has.  (The
// limit as an argument costs 0.5 to 0.8 us an iteration.)
__device__ __forceinline__ bool give_up(int it, int *err)
{
    if (it >= WAIT_MAX || ((it & 1023) == 1023 && *(volatile int *)err != 0)) {
        atomicOr(err, 1);
        return true;
    }
    return false;
}
template <typename T>
__device__ __forceinline__ bool wait_packet(const unsigned long long *p, unsigned ep, T *v, int *err)
{
    for (int it = 0; !Pkt<T>::get(p, ep, v); ++it)
        if (give_up(it, err)) return false;
    return true;
}

// One exchange of sums, run by warp 0: publishes the block's NV partial sums
// and returns the sums over all blocks, added in the same order everywhere.
// Two alternating packet sets are enough: a block writes exchange e only
// after all blocks have written e - 1, that is, after they have read e - 2.
constexpr int PK = (PMAX + 31) / 32;
template <typename T, int NV>
__device__ __forceinline__ bool exchange(unsigned long long *pk, int p0, int P, unsigned epoch, int *err, Acc<T> *v)
{
    const int lane = threadIdx.x & 31;
    unsigned long long *set = pk + (size_t)(epoch & 1u) * PMAX * 4;
    const unsigned long long e = (unsigned long long)epoch << 32;
    if (lane == 0) {
#pragma unroll
        for (int k = 0; k < NV; ++k) {
            unsigned x, y;
            Part<T>::split(v[k].pair(), x, y);
            st_words(set + 4 * blockIdx.x + 2 * k, e | x, e | y);
        }
    }
    // lanes without a packet of their own watch their block's
    const unsigned long long *at[PK];
#pragma unroll
    for (int u = 0; u < PK; ++u) at[u] = set + 4 * (lane + 32 * u < P ? p0 + lane + 32 * u : (int)blockIdx.x);
    unsigned long long a[NV][PK], b[NV][PK];
    bool ok = true;
    for (int it = 0;; ++it) {
        unsigned off = 0;
#pragma unroll
        for (int u = 0; u < PK; ++u)
#pragma unroll
            for (int k = 0; k < NV; ++k) ld_words(at[u] + 2 * k, a[k][u], b[k][u]);
#pragma unroll
        for (int u = 0; u < PK; ++u)
#pragma unroll
            for (int k = 0; k < NV; ++k) off |= ((unsigned)(a[k][u] >> 32) ^ epoch) | ((unsigned)(b[k][u] >> 32) ^ epoch);
        if (!__any_sync(0xffffffffu, off != 0)) break;
        if (__any_sync(0xffffffffu, give_up(it, err))) {
            ok = false;
            break;
        }
    }
#pragma unroll
    for (int k = 0; k < NV; ++k) {
        v[k] = Acc<T>();
#pragma unroll
        for (int u = 0; u < PK; ++u)
            if (lane + 32 * u < P) v[k].join(Part<T>::unite((unsigned)a[k][u], (unsigned)b[k][u]));
        v[k].warp();
    }
    return ok;
}

// A lane's share of a slot: w[receiver] += M w[source] (M = -L); FP32 lanes
// hold a whole block, FP64 lanes one row of it (an FP64 instruction of one
// warp takes 64 clocks here, so a level's chain is its number of FP64
// instructions).
template <typename T>
struct Lane;
template <>
struct Lane<float> {
    uint32_t rec;
    float M[9];
    __device__ __forceinline__ void load(const char *slot, int lane)
    {
        rec = reinterpret_cast<const uint32_t *>(slot)[lane];
        const float *m = reinterpret_cast<const float *>(slot + 128) + lane;
#pragma unroll
        for (int a = 0; a < 9; ++a) M[a] = m[32 * a];
    }
    template <int VB>
    __device__ __forceinline__ void step(uint32_t w) const
    {
        float x[3], y[3];
        const uint32_t d = w + (rec >> 13 & 8191u) * VB;
        V3<float, VB>::ld(w + (rec & 8191u) * VB, x);
        V3<float, VB>::ld(d, y);
#pragma unroll
        for (int r = 0; r < 3; ++r) y[r] = fmaf(M[3 * r + 2], x[2], fmaf(M[3 * r + 1], x[1], fmaf(M[3 * r], x[0], y[r])));
        V3<float, VB>::st(d, y);
    }
};
template <>
struct Lane<double> {
    uint32_t rec;
    double M[3];
    __device__ __forceinline__ void load(const char *slot, int lane)
    {
        rec = reinterpret_cast<const uint32_t *>(slot)[lane];
        const double *m = reinterpret_cast<const double *>(slot + 128) + lane;
#pragma unroll
        for (int a = 0; a < 3; ++a) M[a] = m[32 * a];
    }
    template <int VB>
    __device__ __forceinline__ void step(uint32_t w) const
    {
        double x[3], y;
        const uint32_t d = w + (rec >> 13 & 8191u) * VB + (threadIdx.x & 31) % 3 * 8u;
        V3<double, VB>::ld(w + (rec & 8191u) * VB, x);
        asm volatile("ld.shared.f64 %0, [%1];" : "=d"(y) : "r"(d) : "memory");
        y = fma(M[2], x[2], fma(M[1], x[1], fma(M[0], x[0], y)));
        asm volatile("st.shared.f64 [%0], %1;" ::"r"(d), "d"(y) : "memory");
    }
};
// n slots of a warp from `slot` on; NARROW: each step is a level, else the
// records say where the block barriers lie (`levels` in all).  DEPTH slots
// are in flight; each buffer is refilled as soon as it is used.
template <typename T, int VB, bool NARROW>
__device__ __forceinline__ void run_stream(const char *slot, int32_t n, int levels, uint32_t w)
{
    constexpr int D = 4, B = SlotSize<T>::B;
    const int lane = threadIdx.x & 31;
    // zero first: a register that a skipped load might leave as it was would
    // count as live through the whole solve
    Lane<T> k[D] = {};
#pragma unroll
    for (int d = 0; d < D; ++d)
        if (d < n) k[d].load(slot + d * B, lane);
    const char *next = slot + D * B;
    for (; n > 0;) {
#pragma unroll
        for (int d = 0; d < D; ++d) {
            if (n <= 0) break;
            if (!NARROW)
                for (uint32_t bars = k[d].rec >> 26 & 31u; bars > 0; --bars) {
                    __syncthreads();
                    --levels;
                }
            k[d].template step<VB>(w);
            if (NARROW) __syncwarp();
            if (n > D) k[d].load(next, lane);
            next += B;
            --n;
        }
    }
    if (!NARROW)
        for (; levels > 0; --levels) __syncthreads();
}
// A program in place: its streams (W_*), the slots in shared or global memory.
struct Prog {
    const int32_t *ws;
    const char *wide, *narrow;
};
template <typename T, int VB, bool FWD>
__device__ __forceinline__ void run(const Prog &g, uint32_t w)
{
    const int warp = threadIdx.x >> 5;
    constexpr int B = SlotSize<T>::B;
    if (!FWD) {
        if (warp == 0) run_stream<T, VB, true>(g.narrow, g.ws[W_END] - g.ws[W_NARROW], 0, w);
        __syncthreads();
    }
    const int32_t a = g.ws[warp];
    run_stream<T, VB, false>(g.wide + (size_t)B * a, g.ws[warp + 1] - a, g.ws[W_LEVELS], w);
    if (FWD) {
        if (warp == 0) run_stream<T, VB, true>(g.narrow, g.ws[W_END] - g.ws[W_NARROW], 0, w);
        __syncthreads();
    }
}

// One lane's slot of the matrix.
template <typename T>
struct Slot;
template <>
struct Slot<float> {
    float4 a;
    float2 b;
    __device__ __forceinline__ void load(const Mat<float> &M, size_t row, int lane)
    {
        a = __ldg(M.a + row * 32 + lane);
        b = __ldg(M.b + row * 32 + lane);
    }
    __device__ __forceinline__ int32_t col() const { return __float_as_int(b.y); }
    __device__ __forceinline__ void add(const float *d, float *y) const
    {
        // the six entries of Upsilon = g_perp I + (g_par - g_perp) u u^T
        const float dx = a.y * a.z, dy = a.y * a.w;
        const float s0 = fmaf(dx, a.z, a.x), s1 = dx * a.w, s2 = dx * b.x, s3 = fmaf(dy, a.w, a.x), s4 = dy * b.x,
                    s5 = fmaf(a.y * b.x, b.x, a.x);
        y[0] = fmaf(s0, d[0], y[0]); y[0] = fmaf(s1, d[1], y[0]); y[0] = fmaf(s2, d[2], y[0]);
        y[1] = fmaf(s1, d[0], y[1]); y[1] = fmaf(s3, d[1], y[1]); y[1] = fmaf(s4, d[2], y[1]);
        y[2] = fmaf(s2, d[0], y[2]); y[2] = fmaf(s4, d[1], y[2]); y[2] = fmaf(s5, d[2], y[2]);
    }
};
template <>
struct Slot<double> {
    double2 a, b, c;
    int32_t j;
    __device__ __forceinline__ void load(const Mat<double> &M, size_t row, int lane)
    {
        a = __ldg(M.a + (3 * row) * 32 + lane);
        b = __ldg(M.a + (3 * row + 1) * 32 + lane);
        c = __ldg(M.a + (3 * row + 2) * 32 + lane);
        j = __ldg(M.b + row * 32 + lane);
    }
    __device__ __forceinline__ int32_t col() const { return j; }
    __device__ __forceinline__ void add(const double *d, double *y) const
    {
        y[0] = fma(a.x, d[0], y[0]); y[0] = fma(a.y, d[1], y[0]); y[0] = fma(b.x, d[2], y[0]);
        y[1] = fma(a.y, d[0], y[1]); y[1] = fma(b.y, d[1], y[1]); y[1] = fma(c.x, d[2], y[1]);
        y[2] = fma(b.x, d[0], y[2]); y[2] = fma(c.x, d[1], y[2]); y[2] = fma(c.y, d[2], y[2]);
    }
};
// q = Gamma p on the part's rows (into w), p^T q: a warp takes 32 rows of
// nearly equal length, U slots in flight per lane; p from shared memory (its
// own rows and the halo), or the halo from global memory.
template <typename T, int VB>
__device__ __forceinline__ Acc<T> product(const GridArgs &a, const Mat<T> &M, int32_t ro, int32_t nr, int32_t slot0,
                                       const uint16_t *perm, const int32_t *glen, const int32_t *gso, const T *ps,
                                       uint32_t w)
{
    constexpr int U = sizeof(T) == 4 ? 8 : 2;
    const int lane = threadIdx.x & 31, ng = pad32(nr) / 32;
    const T g0 = (T)a.gamma0;
    const T *pg = reinterpret_cast<const T *>(a.pg);
    Acc<T> acc;
    for (int g = threadIdx.x >> 5; g < ng; g += GW) {
        const int32_t l = perm[32 * g + lane], len = glen[g];
        const size_t row = (size_t)slot0 + gso[g];
        const bool live = l != 0xffff;
        T v[3] = {0, 0, 0}, y[3] = {0, 0, 0};
        if (live) {
            v[0] = ps[3 * l]; v[1] = ps[3 * l + 1]; v[2] = ps[3 * l + 2];
        }
        for (int32_t k = 0; k < len; k += U) {
            Slot<T> s[U];
            T d[U][3];
#pragma unroll
            for (int u = 0; u < U; ++u) s[u].load(M, row + min(k + u, len - 1), lane);
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int32_t j = s[u].col();
                const T *q = j >= 0 ? ps + 3 * j : pg + 3 * (size_t)(-1 - j);
                if (j >= 0) {
                    d[u][0] = q[0]; d[u][1] = q[1]; d[u][2] = q[2];
                } else {
                    d[u][0] = __ldcg(q); d[u][1] = __ldcg(q + 1); d[u][2] = __ldcg(q + 2);
                }
            }
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (k + u < len) {
                    d[u][0] = v[0] - d[u][0]; d[u][1] = v[1] - d[u][1]; d[u][2] = v[2] - d[u][2];
                    s[u].add(d[u], y);
                }
        }
        if (live) {
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                y[c] = fma(g0, v[c], y[c]);
                acc.mul(v[c], y[c]);
            }
            V3<T, VB>::st(w + l * VB, y);
        }
    }
    acc.warp();
    return acc;
}

// D^-1 w of every vertex
template <typename T, int VB>
__device__ __forceinline__ void pivots(const T *D, int32_t nv, uint32_t w)
{
    for (int32_t i = threadIdx.x; i < nv; i += GT) {
        T B[6], x[3], z[3];
        const T *d = D + (size_t)(i >> 5) * 192 + (i & 31);
#pragma unroll
        for (int a = 0; a < 6; ++a) B[a] = d[32 * a];
        V3<T, VB>::ld(w + i * VB, x);
        sym_mv(B, x, z);
        V3<T, VB>::st(w + i * VB, z);
    }
}

// The scalars of a block's solve; warp 0 alone changes them.
template <typename T>
struct Solve {
    Scal S;
    typename Part<T>::type red[2][GW];   // the warps' partial sums
    typename Part<T>::type rho, stop2, rr;   // FP32 keeps these as pairs of floats
    T al, be;
    int go, bad;                         // the solve goes on; a wait gave up
    int p0, np;                          // the system's parts
    double tol2;
    unsigned epoch;
};
enum { OP_START, OP_RHO, OP_PQ, OP_RR, OP_RR_RZ, OP_RZ, OP_NONE };

// The decisions on a sum, in one thread.  FP64: on the Scal as in the
// multi-launch solve.
__device__ __forceinline__ void decide(const GridArgs &a, Solve<double> &Z, int op, double t, double t1)
{
    Scal &S = Z.S;
    switch (op) {
    case OP_START:
        S.FF = t;
        S.rr = t1;
        S.stop2 = Z.tol2 * t;
        S.done = t == 0.0 || t1 <= S.stop2;
        break;
    case OP_RHO:
        S.rho = S.rz = t;
        S.est = S.phi * t;
        if (!(t > 0.0) || !isfinite(t)) {
            S.status = SGP_ERR_NOT_SPD;
            S.done = 1;
        }
        break;
    case OP_PQ:
        S.pq = t;
        if (!(t > 0.0) || !isfinite(t)) {
            S.status = SGP_ERR_NOT_SPD;
            S.done = 1;
        } else {
            Z.al = S.alpha = S.rho / t;
        }
        break;
    case OP_RR:
    case OP_RR_RZ:
        S.rr = t;
        S.it += 1;
        if (t <= S.stop2) {
            S.done = 1;
        } else if (S.it >= S.maxit) {
            S.done = 1;
            S.status = SGP_ERR_NO_CONVERGENCE;
        }
        if (op == OP_RR || S.done) break;
        rz_finish(&S, t1);
        Z.be = S.beta;
        break;
    case OP_RZ:
        rz_finish(&S, t);
        Z.be = S.beta;
        break;
    }
}
// FP32 (inner solves: no error bound): on pairs of floats, so that the chain
// behind every exchange holds no FP64 instruction (64 clocks and more each
// for one warp; a division is ten of them).
__device__ __forceinline__ float pair_ratio(float2 x, float2 y)
{
    const float q = x.x / y.x;
    return q + (fmaf(-q, y.x, x.x) + fmaf(-q, y.y, x.y)) / y.x;
}
__device__ __forceinline__ void decide(const GridArgs &a, Solve<float> &Z, int op, float2 t, float2 t1)
{
    Scal &S = Z.S;
    switch (op) {
    case OP_START: {
        S.FF = (double)t.x + (double)t.y;
        const double st = Z.tol2 * S.FF;
        Z.stop2.x = (float)st;
        Z.stop2.y = (float)(st - (double)Z.stop2.x);
        S.stop2 = st;
        Z.rr = t1;
        S.done = S.FF == 0.0 || (double)t1.x + (double)t1.y <= st;
        break;
    }
    case OP_RHO:
        Z.rho = t;
        if (!(t.x > 0.f) || !isfinite(t.x)) {
            S.status = SGP_ERR_NOT_SPD;
            S.done = 1;
        }
        break;
    case OP_PQ:
        if (!(t.x > 0.f) || !isfinite(t.x)) {
            S.status = SGP_ERR_NOT_SPD;
            S.done = 1;
        } else {
            Z.al = pair_ratio(Z.rho, t);
        }
        break;
    case OP_RR:
    case OP_RR_RZ:
        Z.rr = t;
        S.it += 1;
        if ((t.x - Z.stop2.x) + (t.y - Z.stop2.y) <= 0.f) {
            S.done = 1;
        } else if (S.it >= S.maxit) {
            S.done = 1;
            S.status = SGP_ERR_NO_CONVERGENCE;
        }
        if (op == OP_RR || S.done) break;
        t = t1;
        // fall through
    case OP_RZ:
        if (!(t.x > 0.f) || !isfinite(t.x)) {
            S.status = SGP_ERR_NOT_SPD;
            S.done = 1;
        } else {
            Z.be = pair_ratio(t, Z.rho);
            Z.rho = t;
        }
        break;
    }
}
__device__ __forceinline__ double pair_value(double x) { return x; }
__device__ __forceinline__ double pair_value(float2 x) { return (double)x.x + (double)x.y; }

// Warp 0, after the barrier behind the partial sums: their sums over the
// grid, and the step's decision.
template <typename T>
__device__ __noinline__ void sums(const GridArgs &a, Solve<T> &Z, int op)
{
    const int lane = threadIdx.x & 31;
    const unsigned epoch = Z.epoch + 1;
    const bool two = op == OP_START || op == OP_RR_RZ;
    Acc<T> v[2];
    if (lane < GW && op != OP_NONE) v[0].join(Z.red[0][lane]);
    v[0].warp();
    if (two) {
        if (lane < GW) v[1].join(Z.red[1][lane]);
        v[1].warp();
    }
    const bool ok = two ? exchange<T, 2>(a.pk, Z.p0, Z.np, epoch, a.err, v) : exchange<T, 1>(a.pk, Z.p0, Z.np, epoch, a.err, v);
    if (lane) return;
    Z.epoch = epoch;
    if (!ok) {
        Z.bad = 1;
        return;
    }
    decide(a, Z, op, v[0].pair(), v[1].pair());
    Z.go = Z.S.done ? 0 : 1;
}

// A part's numbers: its vertices, rows (with its top vertices), the top
// vertices that it reaches and their offset, its first top vertex.  It needs
// z of `nout` top vertices (those it reaches, then those it owns), for which it
// forms `na` rows of the top, `nl` of them long; [tb, te): its own system's top.
struct PartDims {
    int32_t nv, nr, ro, t0, nz, zo, nout, na, nl, tb, te;
};
__device__ __forceinline__ PartDims part_of(const GridArgs &a)
{
    const int32_t *h = a.hdr + (size_t)Q_N * blockIdx.x;
    PartDims g{h[Q_NV], h[Q_NR], h[Q_ROFF], h[Q_T0], h[Q_NZ], h[Q_ZOFF], 0, h[Q_NA], h[Q_NL], 0, a.nt};
    if (a.grp && a.nt > 0) {
        const int32_t *h0 = a.hdr + (size_t)Q_N * a.grp[3 * blockIdx.x], *h1 = a.hdr + (size_t)Q_N * (a.grp[3 * blockIdx.x + 1] - 1);
        g.tb = h0[Q_T0];
        g.te = h1[Q_T0] + h1[Q_NR] - h1[Q_NV];
    }
    g.nout = g.nz + g.nr - g.nv;
    return g;
}
// The top's tables and X as the part reads them (in shared or global memory).
template <typename T>
struct Top {
    const int4 *alist, *outs;
    const T *X, *D;
    const int32_t *xi;
    bool local;   // X packed on chip
};
template <typename T>
__device__ __forceinline__ Top<T> top_of(const GridArgs &a, const PartDims &g)
{
    const int32_t *h = a.hdr + (size_t)Q_N * blockIdx.x;
    return Top<T>{a.alist + h[Q_AOFF], a.outs + g.zo + g.t0, reinterpret_cast<const T *>(a.X),
                  reinterpret_cast<const T *>(a.tD), a.xi, false};
}

// One forest solve, in three steps (w: the right-hand side in, the solution
// out).  First the r of the part's top rows to the others, the forward levels,
// the part's sums for the top, its pivots.
template <typename T, int VB>
__device__ __forceinline__ void tree_up(const GridArgs &a, const PartDims &g, const Prog *s_prog, const T *D, uint32_t w,
                                        unsigned long long *trx, unsigned ep)
{
    // (in registers: the cells' accesses below are volatile, so that a field
    // read from shared memory is read again at every use)
    const int32_t nv = g.nv, nr = g.nr, nz = g.nz, zo = g.zo, t0 = g.t0;
    const unsigned long long e = (unsigned long long)ep << 32;
    const T zero[3] = {0, 0, 0};
    for (int32_t z = (int)threadIdx.x; z < nz; z += GT) V3<T, VB>::st(w + (nr + z) * VB, zero);
    __syncthreads();
    for (int32_t i = nv + (int)threadIdx.x; i < nr; i += GT) {
        T v[3];
        V3<T, VB>::ld(w + i * VB, v);
        Pkt<T>::put(trx + (size_t)Pkt<T>::W * (t0 + i - nv), e, v);
    }
    run<T, VB, true>(s_prog[0], w);
    for (int32_t z = (int)threadIdx.x; z < nz; z += GT) {
        T v[3];
        V3<T, VB>::ld(w + (nr + z) * VB, v);
        Pkt<T>::put(a.lx + (size_t)Pkt<T>::W * __ldg(a.zslot + zo + z), e, v);
    }
    pivots<T, VB>(D, nv, w);
}

// Then, by the threads from `first` on, the parts' sums and the top's r.
template <typename T, int VB>
__device__ __forceinline__ bool gather_top(const GridArgs &a, const PartDims &g, uint32_t tw, const unsigned long long *trx, unsigned ep,
                                           int first)
{
    const int tid = threadIdx.x;
    const int32_t te = g.te;
    bool ok = true;
    for (int32_t i = g.tb + tid - first; i < te; i += GT - first) {
        const int32_t k0 = __ldg(a.tlk + i), k1 = __ldg(a.tlk + i + 1);
        // r and the first two sums in flight together
        const unsigned long long *pv = trx + (size_t)Pkt<T>::W * i, *p0 = a.lx + (size_t)Pkt<T>::W * k0,
                                 *p1 = k0 + 1 < k1 ? p0 + Pkt<T>::W : p0;
        if (k0 >= k1) p0 = p1 = pv;
        T v[3], y0[3], y1[3];
        for (int it = 0; ok; ++it) {
            const bool a0 = Pkt<T>::get(pv, ep, v), a1 = Pkt<T>::get(p0, ep, y0),
                       a2 = Pkt<T>::get(p1, ep, y1);
            if (a0 && a1 && a2) break;
            ok = !give_up(it, a.err);
        }
        if (k0 < k1) {
            v[0] += y0[0]; v[1] += y0[1]; v[2] += y0[2];
        }
        if (k0 + 1 < k1) {
            v[0] += y1[0]; v[1] += y1[1]; v[2] += y1[2];
        }
        for (int32_t k = k0 + 2; k < k1 && ok; ++k) {
            ok = wait_packet<T>(a.lx + (size_t)Pkt<T>::W * k, ep, y0, a.err);
            v[0] += y0[0]; v[1] += y0[1]; v[2] += y0[2];
        }
        V3<T, VB>::st(tw + i * VB, v);
    }
    return ok;
}

// Then (after a barrier) the top, as far as the part needs it: u = D^-1 X r in
// the rows that its outputs' columns name, a warp or 8 lanes per row; z = X^T u,
// 8 lanes per output; then the part's backward levels.
template <typename T, int VB>
__device__ __forceinline__ void tree_down(const PartDims &g, const Prog *s_prog, const Top<T> &top, uint32_t w, uint32_t tw, uint32_t tu)
{
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, l8 = lane & 7;
    const int32_t nout = g.nout, nl = g.nl, na = g.na, nz = g.nz, nr = g.nr, nv = g.nv, items = nl + (na - nl + 3) / 4;
    const bool loc = top.local;
    constexpr int N = sizeof(T) == 4 ? 4 : 2;   // blocks in flight per lane
    for (int32_t it = warp; it < items; it += GW) {
        const bool lng = it < nl;
        const int32_t k = lng ? it : nl + 4 * (it - nl) + (lane >> 3), G = lng ? 32 : 8, l = lng ? lane : l8;
        const int4 t = k < na ? top.alist[k] : make_int4(0, 0, 0, 0);
        const int32_t len = t.w, lp = pad8(len), st = loc ? t.z : t.y;
        const int32_t *xi = top.xi + st;
        const T *x = top.X + 9 * (size_t)st;
        // row l of D^-1 (its six entries: 00 01 02 11 12 22)
        T d[3] = {0, 0, 0};
        if (l < 3 && k < na) {
            const T *D = top.D + (size_t)(t.x >> 5) * 192 + (t.x & 31);
            d[0] = __ldg(D + 32 * l);
            d[1] = __ldg(D + 32 * (l == 0 ? 1 : l + 2));
            d[2] = __ldg(D + 32 * (l == 0 ? 2 : l + 3));
        }
        const int32_t most = __reduce_max_sync(0xffffffffu, len);
        T y[3] = {0, 0, 0};
        for (int32_t e0 = 0; e0 < most; e0 += G * N) {
            T m[N][9];
            int32_t i[N];
#pragma unroll
            for (int u = 0; u < N; ++u) {
                const int32_t e = e0 + G * u + l;
                i[u] = e < len ? xi[e] : -1;
#pragma unroll
                for (int c = 0; c < 9; ++c) m[u][c] = e < len ? x[(size_t)c * lp + e] : T(0);
            }
#pragma unroll
            for (int u = 0; u < N; ++u) {
                if (e0 + G * u >= most) break;
                T r[3] = {0, 0, 0};
                if (i[u] >= 0) V3<T, VB>::ld(tw + i[u] * VB, r);
#pragma unroll
                for (int c = 0; c < 3; ++c)
                    y[c] = fma(m[u][3 * c + 2], r[2], fma(m[u][3 * c + 1], r[1], fma(m[u][3 * c], r[0], y[c])));
            }
        }
        if (lng)
#pragma unroll
            for (int b = 16; b > 4; b >>= 1)
#pragma unroll
                for (int c = 0; c < 3; ++c) y[c] += __shfl_xor_sync(0xffffffffu, y[c], b);
#pragma unroll
        for (int b = 4; b > 0; b >>= 1)
#pragma unroll
            for (int c = 0; c < 3; ++c) y[c] += __shfl_xor_sync(0xffffffffu, y[c], b);
        if (l < 3 && k < na) Cell<T>::st(tu + t.x * VB + l * sizeof(T), fma(d[2], y[2], fma(d[1], y[1], d[0] * y[0])));
    }
    __syncthreads();
    for (int32_t base = 4 * warp; base < nout; base += 4 * GW) {
        const int32_t o = base + (lane >> 3);
        const int4 t = o < nout ? top.outs[o] : make_int4(0, 0, 0, 0);
        const int32_t len = t.z, lp = pad8(len), st = loc ? t.y : t.x;
        const int32_t *xi = top.xi + st;
        const T *x = top.X + 9 * (size_t)st;
        T z[3] = {0, 0, 0};
        for (int32_t e = l8; e < len; e += 8) {
            T u[3];
            V3<T, VB>::ld(tu + xi[e] * VB, u);
#pragma unroll
            for (int c = 0; c < 3; ++c)
                z[c] = fma(x[(size_t)(6 + c) * lp + e], u[2], fma(x[(size_t)(3 + c) * lp + e], u[1], fma(x[(size_t)c * lp + e], u[0], z[c])));
        }
        __syncwarp();
#pragma unroll
        for (int b = 4; b > 0; b >>= 1)
#pragma unroll
            for (int c = 0; c < 3; ++c) z[c] += __shfl_xor_sync(0xffffffffu, z[c], b);
        if (l8 == 0 && o < nout) V3<T, VB>::st(w + (o < nz ? nr + o : nv + o - nz) * VB, z);
    }
    __syncthreads();
    run<T, VB, false>(s_prog[1], w);
}

template <typename T, int VB, int PREC>
__global__ void __launch_bounds__(GT, 1) k_pcg_grid(const __grid_constant__ GridArgs a)
{
    extern __shared__ __align__(16) unsigned char sm[];
    __shared__ Solve<T> Z;
    __shared__ Prog s_prog[2];   // the part's forward and backward programs
    __shared__ int32_t s_ws[2][W_N];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int32_t *h = a.hdr + (size_t)Q_N * blockIdx.x;
    const int32_t p0 = a.grp ? a.grp[3 * blockIdx.x] : 0, gid = a.grp ? a.grp[3 * blockIdx.x + 2] : 0;
    const double tol2 = a.gtol2 ? a.gtol2[gid] : a.tol2;
    if (a.gtol2 && tol2 < 0.0) return;   // nothing to solve
    // in registers, but where those are shortest (VB = 12; us per iteration in
    // registers and in shared memory: 1e5 cells FP32 27.1 and 27.9, 3e5 FP64
    // 136.1 and 136.2, 1e6 FP32 133.9 and 130.8)
    __shared__ PartDims sg;
    const PartDims rg = part_of(a);
    if (VB == 12 && tid == 0) sg = rg;
    if (VB == 12) __syncthreads();
    const PartDims &g = VB == 12 ? sg : rg;
    const int32_t nv = g.nv, nr = g.nr, ro = g.ro, slot0 = a.rh[R_N * blockIdx.x + R_SLOT],
                  nh = a.rh[R_N * blockIdx.x + R_NH];
    T *ps = reinterpret_cast<T *>(sm + a.pl.o_p);
    const uint32_t sm0 = (uint32_t)__cvta_generic_to_shared(sm);
    const uint32_t w = sm0 + a.pl.o_w, tw = sm0 + a.pl.o_t;
    auto put = [&](auto *src, int32_t off, int32_t cnt) {
        using E = typename std::remove_const<typename std::remove_reference<decltype(*src)>::type>::type;
        if (off < 0) return (const E *)src;
        E *d = reinterpret_cast<E *>(sm + off);
        for (int32_t i = tid; i < cnt; i += GT) d[i] = src[i];
        return (const E *)d;
    };
    const int ng = pad32(nr) / 32;
    const uint16_t *perm = put(a.perm + ro, a.pl.o_perm, 32 * ng);
    int32_t *glen = reinterpret_cast<int32_t *>(sm + a.pl.o_misc), *gso = glen + ng;
    for (int i = tid; i < ng; i += GT) {
        glen[i] = a.glen[ro / 32 + i];
        gso[i] = a.gso[ro / 32 + i];
    }
    const int32_t *hl = put(a.hl + a.rh[R_N * blockIdx.x + R_HOFF], a.pl.o_hl, a.halo ? nh : 0);
    const T *D = nullptr;
    Top<T> top{};
    if (PREC == 0) {
        D = put(reinterpret_cast<const T *>(a.D) + 6 * (size_t)ro, a.pl.o_D, 6 * pad32(nv));
        constexpr int B = SlotSize<T>::B;
        for (int i = tid; i < 2 * W_N; i += GT) s_ws[i / W_N][i % W_N] = a.ws[(size_t)blockIdx.x * 2 * W_N + i];
        __syncthreads();
        for (int q = 0; q < 2; ++q) {
            // slots in shared memory: the narrow levels, or the whole program
            const char *pg = a.prog[q] + (size_t)B * h[q ? Q_SB : Q_SF];
            const int32_t nn = s_ws[q][W_END] - s_ws[q][W_NARROW];
            const int4 *all = put(reinterpret_cast<const int4 *>(pg), a.pl.o_all[q], (B / 16) * s_ws[q][W_END]);
            const int4 *nar = a.pl.o_all[q] >= 0 ? all + (size_t)(B / 16) * s_ws[q][W_NARROW]
                                                 : put(reinterpret_cast<const int4 *>(pg) + (size_t)(B / 16) * s_ws[q][W_NARROW],
                                                       a.pl.o_nar[q], (B / 16) * nn);
            if (tid == 0) s_prog[q] = Prog{s_ws[q], reinterpret_cast<const char *>(all), reinterpret_cast<const char *>(nar)};
        }
        if (tid == 0) {   // the spare cell
            const T zero[3] = {0, 0, 0};
            V3<T, VB>::st(w + (nr + g.nz) * VB, zero);
        }
        top = top_of<T>(a, g);
        if (a.pl.o_tab >= 0) {
            top.alist = put(top.alist, a.pl.o_tab, g.na);
            top.outs = put(top.outs, a.pl.o_tab + 16 * g.na, g.nout);
        }
        // the rows and columns of X that the part needs, when they fit
        if (a.pl.o_X >= 0) {
            T *xd = reinterpret_cast<T *>(sm + a.pl.o_X);
            int32_t *xi = reinterpret_cast<int32_t *>(sm + a.pl.o_X + 9 * sizeof(T) * (size_t)a.pl.xe);
            for (int32_t k = warp; k < g.na + g.nout; k += GW) {
                const int4 t = k < g.na ? a.alist[h[Q_AOFF] + k] : a.outs[g.zo + g.t0 + k - g.na];
                const int32_t from = k < g.na ? t.y : t.x, at = k < g.na ? t.z : t.y, n = pad8(k < g.na ? t.w : t.z);
                for (int32_t e = lane; e < n; e += 32) xi[at + e] = top.xi[from + e];
                for (int32_t e = lane; e < 9 * n; e += 32) xd[9 * (size_t)at + e] = top.X[9 * (size_t)from + e];
            }
            top.X = xd;
            top.xi = xi;
            top.local = true;
        }
    }
    T *r = a.pl.o_r >= 0 ? reinterpret_cast<T *>(sm + a.pl.o_r) : reinterpret_cast<T *>(a.r) + 3 * (size_t)ro;
    T *x = a.pl.o_x >= 0 ? reinterpret_cast<T *>(sm + a.pl.o_x) : reinterpret_cast<T *>(a.xt) + 3 * (size_t)ro;
    unsigned long long *trx = a.lx + (size_t)Pkt<T>::W * a.nslots;
    Mat<T> M;
    M.a = reinterpret_cast<decltype(M.a)>(a.ma);
    M.b = reinterpret_cast<decltype(M.b)>(a.mb);
    unsigned ep = blockIdx.x == 0 ? a.skew : 0u;   // steps started: the number of this step's packets
    unsigned long long tk = 0, t_spmv = 0, t_tree = 0, t_vec = 0;
    const bool clk = a.timing && blockIdx.x == 0 && tid == 0;
    auto lap = [&](unsigned long long &sum) {
        if (clk) {
            const unsigned long long t = now_ns();
            sum += t - tk;
            tk = t;
        }
    };
    auto partial = [&](int k, Acc<T> &acc) {
        acc.warp();
        if (lane == 0) Z.red[k][warp] = acc.pair();
    };
    // z = H r of the row-wise preconditioners
    auto diag = [&](int32_t i, const T *q, T *z) {
        if (PREC == 1) {
            T B[6];
            const T *d = reinterpret_cast<const T *>(a.jac) + (size_t)((ro + i) >> 5) * 192 + (i & 31);
#pragma unroll
            for (int k = 0; k < 6; ++k) B[k] = __ldg(d + 32 * k);
            sym_mv(B, q, z);
        } else {
            z[0] = q[0]; z[1] = q[1]; z[2] = q[2];
        }
    };
    const T *F = reinterpret_cast<const T *>(a.F);
    T *xo = reinterpret_cast<T *>(a.x);
    if (tid == 0) {
        memset(&Z.S, 0, sizeof(Z.S));
        Z.S.maxit = a.maxit;
        Z.tol2 = tol2;
        Z.p0 = p0;
        Z.np = (a.grp ? a.grp[3 * blockIdx.x + 1] : a.P) - p0;
        Z.S.mu = a.mu;
        Z.S.phi = a.mu > 0.0 ? 1.0 / a.mu : 0.0;
        Z.S.stopE = a.stopE;
        Z.S.tolE2 = a.tolE2;
        Z.go = 1;
        Z.bad = 0;
        Z.epoch = ep;
    }
    // x = 0 or given; without it the first pass skips the product
    for (int32_t i = tid; i < nr; i += GT) {
        const int32_t v = __ldg(a.i_of_t + ro + i);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const T x0 = a.x_given ? xo[3 * (size_t)v + c] : T(0);
            ps[3 * i + c] = x0;
            x[3 * i + c] = x0;
        }
    }
    __syncthreads();
    // phase 0: r = F - Gamma x, the thresholds, z = H r, rho, p = z;
    // from phase 1 on: the steps
    for (int phase = a.x_given ? 0 : -1;; phase = 1) {
        if (phase >= 0) {
            // p of the exported rows to the other parts, theirs into the halo
            ++ep;
            if (a.halo) {
                const unsigned long long e = (unsigned long long)ep << 32;
                for (int32_t i = tid; i < nr; i += GT)
                    if (a.xflag[ro + i]) Pkt<T>::put(a.px + (size_t)Pkt<T>::W * (ro + i), e, ps + 3 * i);
                for (int32_t k = tid; k < nh; k += GT)
                    if (!wait_packet<T>(a.px + (size_t)Pkt<T>::W * hl[k], ep, ps + 3 * (nr + k), a.err)) Z.bad = 1;
                __syncthreads();
            } else {
                T *o = reinterpret_cast<T *>(a.pg) + 3 * (size_t)ro;
                for (int32_t i = tid; i < 3 * nr; i += GT) o[i] = ps[i];
                __threadfence();
                __syncthreads();
                if (warp == 0) {
                    sums<T>(a, Z, OP_NONE);
                    __threadfence();
                }
                __syncthreads();
            }
            if (Z.bad) return;
            lap(t_vec);
            Acc<T> pq = product<T, VB>(a, M, ro, nr, slot0, perm, glen, gso, ps, w);
            if (lane == 0) Z.red[0][warp] = pq.pair();
            __syncthreads();
        }
        if (phase <= 0) {
            Acc<T> ff, rr;
            for (int32_t i = tid; i < nr; i += GT) {
                const int32_t v = __ldg(a.i_of_t + ro + i);
                T q[3] = {0, 0, 0}, z[3];
                if (phase == 0) V3<T, VB>::ld(w + i * VB, q);
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    const T f = F[3 * (size_t)v + c];
                    ff.mul(f, f);
                    q[c] = f - q[c];
                    rr.mul(q[c], q[c]);
                    r[3 * i + c] = q[c];
                }
                diag(i, q, z);
                V3<T, VB>::st(w + i * VB, z);
            }
            partial(0, ff);
            partial(1, rr);
            __syncthreads();
            if (warp == 0) sums<T>(a, Z, OP_START);
            __syncthreads();
            if (Z.bad) return;
            if (clk) tk = now_ns();
            if (!Z.go) break;
        } else {
            if (warp == 0) sums<T>(a, Z, OP_PQ);
            __syncthreads();
            if (Z.bad) return;
            lap(t_spmv);
            if (!Z.go) break;
            const T al = Z.al;
            Acc<T> rr, rz;
            constexpr int N = 2;   // rows in flight per thread
            for (int32_t b = tid; b < nr; b += N * GT) {
                T rv[N][3], xv[N][3];
#pragma unroll
                for (int u = 0; u < N; ++u) {
                    const int32_t i = b + u * GT;
#pragma unroll
                    for (int c = 0; c < 3; ++c) {
                        rv[u][c] = i < nr ? r[3 * i + c] : T(0);
                        xv[u][c] = i < nr ? x[3 * i + c] : T(0);
                    }
                }
#pragma unroll
                for (int u = 0; u < N; ++u) {
                    const int32_t i = b + u * GT;
                    if (i >= nr) break;
                    T q[3], z[3];
                    V3<T, VB>::ld(w + i * VB, q);
#pragma unroll
                    for (int c = 0; c < 3; ++c) {
                        q[c] = fma(-al, q[c], rv[u][c]);
                        rr.mul(q[c], q[c]);
                        r[3 * i + c] = q[c];
                        x[3 * i + c] = fma(al, ps[3 * i + c], xv[u][c]);
                    }
                    diag(i, q, z);
                    if (PREC != 0) {
#pragma unroll
                        for (int c = 0; c < 3; ++c) rz.mul(q[c], z[c]);
                    }
                    V3<T, VB>::st(w + i * VB, z);
                }
            }
            partial(0, rr);
            if (PREC != 0) partial(1, rz);
        }
        if (PREC == 0) {
            tree_up<T, VB>(a, g, s_prog, D, w, trx, ep + 1);
        } else {
            __syncthreads();
        }
        // |r|^2 and the stopping test by warp 0; the others gather the parts'
        // sums and the top's r
        const int first = phase > 0 ? 32 : 0;
        if (warp == 0 && phase > 0) {
            sums<T>(a, Z, PREC == 0 ? OP_RR : OP_RR_RZ);
        } else if (PREC == 0) {
            if (!gather_top<T, VB>(a, g, tw, trx, ep + 1, first)) Z.bad = 1;
        }
        __syncthreads();
        if (Z.bad) return;
        if (!Z.go) {
            lap(t_tree);
            break;
        }
        if (PREC == 0) {
            tree_down<T, VB>(g, s_prog, top, w, tw, sm0 + a.pl.o_u);
            if (sizeof(T) == 8 && a.pl.o_u == a.pl.o_p && phase > 0) {   // p's first rows again
                const T *o = reinterpret_cast<const T *>(a.pg) + 3 * (size_t)ro;
                for (int32_t i = tid; i < min(3 * nr, a.nt * (int)(VB / sizeof(T))); i += GT) ps[i] = __ldcg(o + i);
            }
        }
        if (PREC == 0 || phase <= 0) {
            Acc<T> acc;
            for (int32_t i = tid; i < nr; i += GT) {
                T z[3];
                V3<T, VB>::ld(w + i * VB, z);
                const T r0 = r[3 * i], r1 = r[3 * i + 1], r2 = r[3 * i + 2];
                acc.mul(r0, z[0]);
                acc.mul(r1, z[1]);
                acc.mul(r2, z[2]);
            }
            partial(0, acc);
            __syncthreads();
            if (warp == 0) sums<T>(a, Z, phase <= 0 ? OP_RHO : OP_RZ);
            __syncthreads();
            if (Z.bad) return;
            if (PREC == 0) lap(t_tree);
            if (!Z.go) break;
        }
        const T be = phase <= 0 ? T(0) : Z.be;
        for (int32_t i = tid; i < nr; i += GT) {
            T z[3];
            V3<T, VB>::ld(w + i * VB, z);
#pragma unroll
            for (int c = 0; c < 3; ++c) ps[3 * i + c] = phase <= 0 ? z[c] : fma(be, ps[3 * i + c], z[c]);
        }
        __syncthreads();
    }
    __syncthreads();
    for (int32_t i = tid; i < nr; i += GT) {
        const int32_t v = __ldg(a.i_of_t + ro + i);
#pragma unroll
        for (int c = 0; c < 3; ++c) xo[3 * (size_t)v + c] = x[3 * i + c];
    }
    if (blockIdx.x == p0 && tid == 0) {
        if (sizeof(T) == 4) Z.S.rr = pair_value(Z.rr);
        a.sc[gid] = Z.S;
        if (a.timing && blockIdx.x == 0) {
            a.ns[0] = t_spmv;
            a.ns[1] = t_tree;
            a.ns[2] = t_vec;
        }
    }
}

// One forest solve alone: x = P^-1 b in the caller's order (orig_of) or the
// internal one, the forest's part of one iteration above.  Everything is read once, so only what warp 0 reads
// in sequence (the narrow levels) is brought on chip first, while the right-
// hand side arrives.
template <typename T, int VB>
__global__ void __launch_bounds__(GT, 1) k_apply_grid(const __grid_constant__ GridArgs a, const int32_t *__restrict__ orig_of,
                                                    const int *__restrict__ done)
{
    extern __shared__ __align__(16) unsigned char sm[];
    __shared__ Prog s_prog[2];
    __shared__ int32_t s_ws[2][W_N];
    __shared__ int s_bad;
    const int tid = threadIdx.x;
    const int32_t *h = a.hdr + (size_t)Q_N * blockIdx.x;
    const PartDims g = part_of(a);
    const uint32_t sm0 = (uint32_t)__cvta_generic_to_shared(sm);
    const uint32_t w = sm0 + a.pl.o_w, tw = sm0 + a.pl.o_t;
    constexpr int B = SlotSize<T>::B;
    if (done && *done) return;
    const T *F = reinterpret_cast<const T *>(a.F);
    T *x = reinterpret_cast<T *>(a.x);
    for (int i = tid; i < 2 * W_N; i += GT) s_ws[i / W_N][i % W_N] = a.ws[(size_t)blockIdx.x * 2 * W_N + i];
    if (tid == 0) s_bad = 0;
    __syncthreads();
    for (int q = 0; q < 2; ++q) {
        const char *pg = a.prog[q] + (size_t)B * h[q ? Q_SB : Q_SF], *nar = pg + (size_t)B * s_ws[q][W_NARROW];
        if (a.pl.o_nar[q] >= 0) {
            const int32_t cnt = (B / 16) * (s_ws[q][W_END] - s_ws[q][W_NARROW]);
            int4 *d = reinterpret_cast<int4 *>(sm + a.pl.o_nar[q]);
            for (int32_t i = tid; i < cnt; i += GT) d[i] = reinterpret_cast<const int4 *>(nar)[i];
            nar = reinterpret_cast<const char *>(d);
        }
        if (tid == 0) s_prog[q] = Prog{s_ws[q], pg, nar};
    }
    constexpr int N = 4;   // rows in flight per thread
    for (int32_t b = tid; b < g.nr; b += N * GT) {
        int32_t v[N];
#pragma unroll
        for (int u = 0; u < N; ++u) v[u] = __ldg(a.i_of_t + g.ro + min(b + u * GT, g.nr - 1));
#pragma unroll
        for (int u = 0; u < N; ++u)
            if (orig_of) v[u] = __ldg(orig_of + v[u]);
        T q[N][3];
#pragma unroll
        for (int u = 0; u < N; ++u)
#pragma unroll
            for (int c = 0; c < 3; ++c) q[u][c] = F[3 * (size_t)v[u] + c];
#pragma unroll
        for (int u = 0; u < N; ++u)
            if (b + u * GT < g.nr) V3<T, VB>::st(w + (b + u * GT) * VB, q[u]);
    }
    const T zero[3] = {0, 0, 0};
    if (tid == 0) V3<T, VB>::st(w + (g.nr + g.nz) * VB, zero);   // the spare cell
    unsigned long long *trx = a.lx + (size_t)Pkt<T>::W * a.nslots;
    const unsigned ep = blockIdx.x == 0 ? a.skew + 1u : 1u;
    tree_up<T, VB>(a, g, s_prog, reinterpret_cast<const T *>(a.D) + 6 * (size_t)g.ro, w, trx, ep);
    if (!gather_top<T, VB>(a, g, tw, trx, ep, 0)) s_bad = 1;
    __syncthreads();
    const bool bad = s_bad != 0;
    if (bad && tid == 0) *(volatile int *)a.gave_up = 1;
    if (!bad)
        tree_down<T, VB>(g, s_prog, top_of<T>(a, g), w, tw, sm0 + a.pl.o_u);
    for (int32_t b = tid; b < g.nr; b += N * GT) {
        int32_t v[N];
#pragma unroll
        for (int u = 0; u < N; ++u) v[u] = __ldg(a.i_of_t + g.ro + min(b + u * GT, g.nr - 1));
#pragma unroll
        for (int u = 0; u < N; ++u)
            if (orig_of) v[u] = __ldg(orig_of + v[u]);
#pragma unroll
        for (int u = 0; u < N; ++u) {
            if (b + u * GT >= g.nr) break;
            T q[3];
            V3<T, VB>::ld(w + (b + u * GT) * VB, q);
#pragma unroll
            for (int c = 0; c < 3; ++c) x[3 * (size_t)v[u] + c] = bad ? T(NAN) : q[c];
        }
    }
}

}  // namespace

// ---------------------------------------------------------- host: building
namespace {

// Shared-memory placement (sized by the largest part, the same in every
// block): what is addressed at random always; then, as far as it fits, what
// is read most often.  False: the vectors alone do not fit.
bool place(const GridLayout &G, int32_t mnh, size_t sz, size_t vb, bool tree, bool halo, GridPlace *pl)
{
    const int32_t *t = G.tot;
    const size_t mnr = (size_t)t[T_MNR], nt = tree ? (size_t)t[T_NT] : 0;
    size_t at = 0;
    auto need = [&](size_t b) {
        const int32_t o = (int32_t)at;
        at += (b + 15) & ~size_t(15);
        return o;
    };
    auto opt = [&](size_t b) {
        const size_t r = (b + 15) & ~size_t(15);
        return r > 0 && at + r <= (size_t)GRID_SMEM ? need(b) : -1;
    };
    const size_t B = sz == 4 ? SlotSize<float>::B : SlotSize<double>::B;
    pl->o_p = need(3 * sz * (mnr + (halo ? (size_t)mnh : 0)));
    pl->o_w = need(vb * (size_t)(tree ? t[T_MDZ] + 1 : t[T_MNR]));
    pl->o_t = need(vb * nt);
    // the top's D^-1 X r; where it does not fit beside the rest and p is in
    // memory too (no halo on chip), in the place of p's first rows (sizes of
    // 530,000 to 640,000 cells, by their largest part; FP32 ends at NREC cells)
    const size_t misc = 8 * (mnr / 32 + 1);
    const bool in_p = tree && !halo && sz == 8 && at + vb * nt + misc + 32 > (size_t)GRID_SMEM && vb * nt <= 3 * sz * mnr;
    pl->o_u = in_p ? pl->o_p : need(vb * nt);
    pl->o_misc = need(misc);
    if (at > (size_t)GRID_SMEM) return false;
    for (int q = 0; q < 2; ++q) pl->o_nar[q] = pl->o_all[q] = -1;
    pl->o_D = pl->o_X = pl->o_tab = -1;
    pl->o_perm = opt(2 * (size_t)pad32((int32_t)mnr));
    pl->o_hl = halo ? opt(4 * (size_t)mnh) : -1;
    if (tree) {
        pl->o_tab = opt(16 * ((size_t)t[T_MNA] + (size_t)t[T_MNO]));
        // the whole programs when they fit beside r and x, else the narrow levels
        const size_t all = B * ((size_t)t[T_MSF] + (size_t)t[T_MSB]) + 6 * sz * mnr + 64;
        if (at + all <= (size_t)GRID_SMEM)
            for (int q = 0; q < 2; ++q) pl->o_all[q] = opt(B * (size_t)(q ? t[T_MSB] : t[T_MSF]));
        else
            for (int q = 0; q < 2; ++q) pl->o_nar[q] = opt(B * (size_t)(q ? t[T_MNB] : t[T_MNF]));
    }
    pl->o_r = opt(3 * sz * mnr);
    pl->o_x = opt(3 * sz * mnr);
    if (tree) {
        pl->o_D = opt(6 * sz * (size_t)pad32((int32_t)mnr));
        pl->xe = t[T_MX];
        pl->o_X = opt((9 * sz + 4) * (size_t)t[T_MX]);
        for (int q = 0; q < 2; ++q)
            if (pl->o_all[q] < 0) {
                // more room after all: one whole program
                const int32_t o = opt(B * (size_t)(q ? t[T_MSB] : t[T_MSF]));
                if (o >= 0) pl->o_all[q] = o;
            }
    }
    pl->bytes = (int32_t)at;
    return true;
}

// The same for one forest solve alone.
bool place_apply(const GridLayout &G, size_t sz, size_t vb, GridPlace *pl)
{
    const int32_t *t = G.tot;
    size_t at = 0;
    auto need = [&](size_t b) {
        const int32_t o = (int32_t)at;
        at += (b + 15) & ~size_t(15);
        return o;
    };
    const size_t B = sz == 4 ? SlotSize<float>::B : SlotSize<double>::B;
    *pl = GridPlace{};
    pl->o_X = pl->o_tab = -1;
    pl->o_w = need(vb * (size_t)(t[T_MDZ] + 1));
    pl->o_t = need(vb * (size_t)t[T_NT]);
    pl->o_u = need(vb * (size_t)t[T_NT]);
    if (at > (size_t)GRID_SMEM) return false;
    for (int q = 0; q < 2; ++q) {
        const size_t b = B * (size_t)(q ? t[T_MNB] : t[T_MNF]);
        pl->o_nar[q] = b > 0 && at + b + 16 <= (size_t)GRID_SMEM ? need(b) : -1;
    }
    pl->bytes = (int32_t)at;
    return true;
}

struct GScr {
    sgp_ctx *ctx;
    GridLayout *G;
    int nbuf = 0;
    template <typename U>
    sgp_status take(size_t count, U **p)
    {
        if (nbuf >= SGP_GRID_SCRATCH) return sgp_fail(ctx, SGP_ERR_OOM, "grid layout: out of scratch buffers");
        DBuf &b = G->scr[nbuf++];
        SGP_TRY(buf_ensure(ctx, b, sizeof(U) * std::max<size_t>(count, 16)));
        *p = reinterpret_cast<U *>(b.p);
        return SGP_OK;
    }
};

template <typename U>
sgp_status ensure(sgp_ctx *ctx, DBuf &b, size_t count, U **p)
{
    SGP_TRY(buf_ensure(ctx, b, sizeof(U) * std::max<size_t>(count, 16)));
    *p = reinterpret_cast<U *>(b.p);
    return SGP_OK;
}

// Parts for n rows: one block per SM, at least `umin` rows each.
int32_t part_count(const sgp_ctx *ctx, int32_t n, int32_t umin)
{
    return std::max(1, std::min(std::min(ctx->num_sms, PMAX), (n + umin - 1) / umin));
}

// The rows of a matrix on the parts of a layout, up to the counts (they go to
// the host with the next read of `R.tot`).
sgp_status rows_count(sgp_ctx *ctx, GridRows &R, GBuild &g, const sgp_matrix *M, size_t NRmax)
{
    const int32_t P = g.P;
    g.NRW = (int32_t)(NRmax / 32);
    SGP_TRY(ensure(ctx, R.rh, R_N * ((size_t)P + 1), &g.rh));
    SGP_TRY(ensure(ctx, R.glen, NRmax / 32 + 1, &g.glen));
    SGP_TRY(ensure(ctx, R.gso, NRmax / 32 + 1, &g.gso));
    SGP_TRY(ensure(ctx, R.perm, NRmax, &g.perm));
    SGP_TRY(ensure(ctx, R.xflag, NRmax, &g.xflag));
    SGP_TRY(ensure(ctx, R.hb, (size_t)P * g.NRW, &g.hb));
    SGP_TRY(ensure(ctx, R.hpre, (size_t)P * g.NRW, &g.hpre));
    SGP_CUDA(ctx, cudaMemsetAsync(g.hb, 0, sizeof(uint32_t) * (size_t)P * g.NRW, ctx->stream));
    SGP_CUDA(ctx, cudaMemsetAsync(g.xflag, 0, NRmax, ctx->stream));
    g.row_ptr = bp<const int32_t>(M->row_ptr);
    g.col = bp<const int32_t>(M->col);
    LAUNCH(ctx, k_gr_part_rows, P, GT, 0, g);
    const unsigned gy = (unsigned)std::max<size_t>(1, std::min<size_t>(8, NRmax / P / GT));
    SGP_TRY(sgp_launch(ctx, "k_gr_halo_mark", k_gr_halo_mark, dim3(P, gy), dim3(GT), 0, g));
    LAUNCH(ctx, k_gr_halo_count, P, 1024, 0, g);
    LAUNCH(ctx, k_gr_row_offsets, 1, 256, 0, g);
    return SGP_OK;
}

// Where the halo goes: on chip, in FP32 with packed vectors if need be, else
// read from memory.  False: nothing fits, or the padded rows are too many.
bool rows_place(const GridLayout &G, GridRows &R, const sgp_matrix *M, bool f32, bool tree)
{
    const size_t sz = f32 ? 4 : 8;
    GridPlace pl;
    if (G.tot[T_MNR] + R.tot[2] > 65535 ||
        (int64_t)R.tot[0] * 32 > 4 * (int64_t)M->m + 64 * (int64_t)M->n + 65536)
        return false;
    R.halo = 1;
    R.vb = f32 ? 16 : 24;
    if (place(G, R.tot[2], sz, R.vb, tree, true, &pl)) return true;
    if (f32) R.vb = 12;
    if (f32 && place(G, R.tot[2], sz, R.vb, tree, true, &pl)) return true;
    R.halo = 0;
    return place(G, R.tot[2], sz, R.vb, tree, false, &pl);
}

// The matrix's rows in part order (after the counts are known).
sgp_status rows_fill(sgp_ctx *ctx, const GridLayout &G, GridRows &R, GBuild &g, const sgp_matrix *M, bool f32)
{
    const int32_t P = g.P;
    const unsigned gy = (unsigned)std::max(1, std::min(8, G.tot[T_MNR] / GT));
    g.halo = R.halo;
    SGP_TRY(ensure(ctx, R.hl, R.tot[1], &g.hl));
    if (g.halo) SGP_TRY(sgp_launch(ctx, "k_gr_halo_list", k_gr_halo_list, dim3(P, gy), dim3(GT), 0, g));
    const size_t slots = 32 * (size_t)R.tot[0];
    if (f32) {
        float4 *at;
        float2 *bt;
        SGP_TRY(ensure(ctx, R.ma, slots, &at));
        SGP_TRY(ensure(ctx, R.mb, slots, &bt));
        const float4 *a4 = bp<const float4>(M->blk32);
        SGP_TRY(sgp_launch(ctx, "k_gr_sell32", k_gr_sell32, dim3(P, gy), dim3(GT), 0, g, a4,
                           reinterpret_cast<const float2 *>(a4 + 2 * M->m), at, bt));
    } else {
        double2 *at;
        int32_t *bt;
        SGP_TRY(ensure(ctx, R.ma, 3 * slots, &at));
        SGP_TRY(ensure(ctx, R.mb, slots, &bt));
        SGP_TRY(sgp_launch(ctx, "k_gr_sell64", k_gr_sell64, dim3(P, gy), dim3(GT), 0, g, bp<const double>(M->blk),
                           bp<const int32_t>(M->col), at, bt));
    }
    R.mgen = M->gen;
    R.ok = 1;
    return SGP_OK;
}

template <typename T>
sgp_status numeric(sgp_ctx *ctx, GridLayout &G, const sgp_factor *F, const sgp_matrix *M, const GBuild &g,
                   const int32_t *td_src)
{
    const double scale = pivot_scale<T>(M);
    const int32_t *t = G.tot;
    const double *L = bp<const double>(F->L), *Di = bp<const double>(F->Dinv);
    const int32_t nf = 32 * t[T_SF], nb = 32 * t[T_SB], nr = t[T_NR], nt = t[T_NT], B = SGP_BLOCK;
    T *D, *X, *tD;
    SGP_TRY(ensure(ctx, G.D, 6 * (size_t)nr, &D));
    SGP_TRY(ensure(ctx, G.X, 9 * ((size_t)t[T_RE] + (size_t)t[T_CE]), &X));
    SGP_TRY(ensure(ctx, G.tD, 6 * (size_t)pad32(nt), &tD));
    LAUNCH(ctx, (k_gr_blocks<T, false>), grid_for(nf, B), B, 0, nf, (const int32_t *)g.msrc[0], L, g.prog[0]);
    LAUNCH(ctx, (k_gr_blocks<T, true>), grid_for(nb, B), B, 0, nb, (const int32_t *)g.msrc[1], L, g.prog[1]);
    LAUNCH(ctx, k_gr_pivots<T>, grid_for(nr, B), B, 0, nr, (const int32_t *)g.d_src, Di, scale, D);
    if (nt == 0) return SGP_OK;
    LAUNCH(ctx, k_gr_top_fill<T>, nt, 128, 0, g, X);
    LAUNCH(ctx, k_gr_pivots<T>, grid_for(nt, B), B, 0, nt, td_src, Di, scale, tD);
    return SGP_OK;
}

}  // namespace

// Build the grid layout of a factor whose structure and numerics are done,
// in the factor's own precision, with the rows of `M`.  Leaves G.ok at 0
// when a part does not fit (the other solves then serve the factor).
sgp_status grid_build(sgp_ctx *ctx, sgp_factor *F, const sgp_matrix *M)
{
    GridLayout &G = F->gl;
    G.ok = G.rows.ok = 0;
    const int32_t n = (int32_t)F->n, LV = F->levels;
    if (n == 0 || LV == 0 || LV > LMAX || !M || M->n != n || M->precision != F->precision) return SGP_OK;
    const bool f32 = F->precision == SGP_PREC_MIXED;
    // At least 128 rows per part.  Measured (us per iteration, FP64 lattice of
    // 10,000 cells): 41.3 with 64 rows and 152 parts, 38.9 with 128, 42.9 with
    // 256, 53.9 with 512: more parts share the FP64 work, fewer exchange less.
    int32_t P = part_count(ctx, n, 128);
    int32_t U = (n + P - 1) / P;
    // a batch: no part holds rows of two instances, and U is the smallest at
    // which the instances' parts fit the device
    std::vector<int64_t> &irow = G.irow;
    irow.assign({0, (int64_t)n});
    if (M->batched) irow = M->inst_row;
    const int32_t NI = (int32_t)irow.size() - 1;
    if (NI < 1 || irow[0] != 0 || irow[NI] != n || NI > PMAX) return SGP_OK;
    G.ipart.assign(NI + 1, 0);
    if (NI > 1) {
        const int32_t most = std::min(ctx->num_sms, PMAX);
        auto parts = [&](int64_t u) {
            int64_t c = 0;
            for (int32_t s = 0; s < NI; ++s) c += (irow[s + 1] - irow[s] + u - 1) / u;
            return c;
        };
        int64_t lo = 127, hi = n;
        if (parts(hi) > most) return SGP_OK;   // more instances than SMs
        while (hi - lo > 1) {
            const int64_t mid = (lo + hi) / 2;
            if (parts(mid) <= most) hi = mid; else lo = mid;
        }
        U = (int32_t)hi;
        P = (int32_t)parts(U);
        for (int32_t s = 0; s < NI; ++s) G.ipart[s + 1] = G.ipart[s] + (int32_t)((irow[s + 1] - irow[s] + U - 1) / U);
    } else {
        G.ipart[1] = P;
    }
    // p and w of the largest part must fit; in FP64 w alone serves the forest
    // solve, whose launch has no p.  A slot's record counts 13 bits of cells.
    const auto too_large = [&](int32_t rows) { return (size_t)rows * 24 > (size_t)GRID_SMEM || rows > NREC; };
    if (too_large(U)) return SGP_OK;
    // The subtree bound trades the number of top vertices (every block reads
    // its rows and columns of their L^-1) and the length of the narrow levels against
    // what balancing can do (a part cannot be smaller than its largest
    // subtree).  Measured, us per iteration: FP64, U = 127 rows per part: 31.8
    // with bmax = U, 31.1 with 3U/2, 30.7 with 2U; U = 395: U/2 61, 3U/4 50, 3U/2
    // 49; U = 658: 0.6 U 63.4, 3U/4 57.8, U 57.8, 1.3 U 60.2; U = 1974: U/2 133,
    // 3U/4 125, U 124-130, 1.3 U 131.  FP32, U = 197: 20.7 with U, 20.2 with
    // 3U/2; U = 395: U/2 24, 3U/2 22.4; U = 658: U/2 25.8, U 26.1; U = 1645: U/2
    // 35, U 40; U = 3290: U/4 80, U/2 67-71, U 71-77; U = 6579: U/4 131, 0.35 U
    // 121-127, U/2 120-125, U 182 (the halo no longer fits on chip).
    const int32_t part = U <= 512 ? 3 * U / 2 : (f32 ? U / 2 : 3 * U / 4);
    const int32_t bmax = std::max(32, part);
    G.P = P;
    G.LV = LV;
    const int32_t NP = (int32_t)F->npairs;
    GScr S{ctx, &G};
    const int B = SGP_BLOCK;
    const int32_t nblk = (n + MS_ITEMS - 1) / MS_ITEMS;
    GBuild g{};
    g.n = n; g.P = P; g.LV = LV;
    g.ord = bp<const int32_t>(F->ord);
    g.pos = bp<const int32_t>(F->pos);
    g.pr_ptr = bp<const int32_t>(F->pr_ptr);
    g.pr_q = bp<const int32_t>(F->pr_q);
    g.pr_c = bp<const int32_t>(F->pr_c);
    int32_t *lp, *par, *sz_, *wv, *pre, *wsm, *psm, *load, *anc, *anc2, *rseg, *seg, *hist, *off, *sp, *lpos;
    SGP_TRY(S.take((size_t)LV + 1 + 2 * ((size_t)NI + 1), &lp));
    const int32_t *d_irow = lp + LV + 1, *d_ipart = d_irow + NI + 1;
    const int32_t NS = P + NI;   // segments: parts, then the instances' tops
    SGP_TRY(S.take(n, &par));
    SGP_TRY(S.take(n, &sz_));
    SGP_TRY(S.take(n, &wv));
    SGP_TRY(S.take((size_t)n + 1, &pre));
    SGP_TRY(S.take(n, &wsm));
    SGP_TRY(S.take((size_t)n + 1, &psm));
    SGP_TRY(S.take((3 + NBIG) * (size_t)P, &load));
    SGP_TRY(S.take(n, &anc));
    SGP_TRY(S.take(n, &anc2));
    SGP_TRY(S.take(n, &rseg));
    SGP_TRY(S.take(n, &seg));
    SGP_TRY(S.take((size_t)NS * nblk + 1, &hist));
    SGP_TRY(S.take((size_t)NS * nblk + 1, &off));
    SGP_TRY(S.take(n, &sp));
    SGP_TRY(S.take(n, &lpos));
    std::vector<int32_t> tab(F->lvl_ptr.begin(), F->lvl_ptr.begin() + LV + 1);
    tab.insert(tab.end(), irow.begin(), irow.end());
    tab.insert(tab.end(), G.ipart.begin(), G.ipart.end());
    SGP_CUDA(ctx, cudaMemcpyAsync(lp, tab.data(), sizeof(int32_t) * tab.size(), cudaMemcpyHostToDevice, ctx->stream));
    LAUNCH(ctx, k_gr_parent, grid_for(n, B), B, 0, n, g.pr_ptr, g.pr_q, g.pos, par, sz_);
    int l0 = 0;
    while (l0 < LV && F->lvl_ptr[l0 + 1] - F->lvl_ptr[l0] > 4096) {
        const int32_t p0 = F->lvl_ptr[l0], c = F->lvl_ptr[l0 + 1] - p0;
        LAUNCH(ctx, k_gr_size, grid_for(c, B), B, 0, p0, c, (const int32_t *)par, sz_);
        ++l0;
    }
    if (l0 < LV) LAUNCH(ctx, k_gr_size_rest, 1, 1024, 0, (const int32_t *)lp, l0, LV, (const int32_t *)par, sz_);
    // (U/8 against U/16: U = 658 FP64 57.8 and 59.6 us, FP32 25.8 and 26.4; U =
    // 1645 35.6 and 34.3, U = 3290 71.1 and 67.1, U = 6579 125.5 and 122.3)
    // A batch keeps the middles' parts: an instance has a few only, and the halo
    // that moved subtrees add costs more (48 instances of 3e5 cells, two draws:
    // solve 8.9 and 9.3 ms so, 8.4 and 10.6 ms balanced).
    const int32_t small = NI > 1 ? 0 : U <= 1024 ? U / 8 : U / 16;
    int32_t *cnt = load + P, *room = cnt + P, *list = room + P;
    SGP_CUDA(ctx, cudaMemsetAsync(load, 0, 2 * sizeof(int32_t) * P, ctx->stream));
    LAUNCH(ctx, k_gr_class, grid_for(n, B), B, 0, n, bmax, small, (const int32_t *)sz_, (const int32_t *)par, g.ord, wv, wsm);
    SGP_TRY(scan_exclusive_i32(ctx, wv, pre, n));
    SGP_TRY(scan_exclusive_i32(ctx, wsm, psm, n));
    LAUNCH(ctx, k_gr_roots, grid_for(n, B), B, 0, n, bmax, P, NI, d_irow, d_ipart, (const int32_t *)sz_, (const int32_t *)par, g.ord,
           (const int32_t *)pre, small, load, cnt, list, anc, rseg);
    if (NI == 1)
        LAUNCH(ctx, k_gr_balance, 1, 1024, 0, P, NI, d_ipart, (const int32_t *)sz_, (const int32_t *)cnt,
               (const int32_t *)list, load, rseg);
    LAUNCH(ctx, k_gr_fill, 1, 256, 0, NI, d_irow, d_ipart, (const int32_t *)psm, (const int32_t *)load, room);
    LAUNCH(ctx, k_gr_small, grid_for(n, B), B, 0, n, d_irow, d_ipart, (const int32_t *)sz_, g.ord, (const int32_t *)psm,
           (const int32_t *)room, rseg);
    for (int r = 0; (1 << r) <= LV + 1; ++r) {
        LAUNCH(ctx, k_gr_jump, grid_for(n, B), B, 0, n, (const int32_t *)anc, anc2);
        std::swap(anc, anc2);
    }
    LAUNCH(ctx, k_gr_seg, grid_for(n, B), B, 0, n, (const int32_t *)anc, (const int32_t *)rseg, seg);
    LAUNCH(ctx, k_gr_split_count, nblk, GT, 0, n, NS, (const int32_t *)seg, hist);
    SGP_TRY(scan_exclusive_i32(ctx, hist, off, (int64_t)NS * nblk));
    LAUNCH(ctx, k_gr_split_place, nblk, GT, 0, n, NS, (const int32_t *)seg, (const int32_t *)off, sp, lpos);
    if (NI > 1) LAUNCH(ctx, k_gr_top_merge, grid_for(n, B), B, 0, n, P, nblk, (const int32_t *)off, seg, lpos);
    const size_t NRmax = (size_t)pad32(n) + 32 * (size_t)P + 32, PB = (size_t)P + 1;
    SGP_TRY(ensure(ctx, G.hdr, (size_t)Q_N * PB, &g.hdr));
    SGP_TRY(ensure(ctx, G.dtot, T_N, &g.tot));
    SGP_TRY(ensure(ctx, G.i_of_t, NRmax, &g.i_of_t));
    SGP_TRY(ensure(ctx, G.t_of_i, n, &g.t_of_i));
    SGP_TRY(ensure(ctx, G.ws, PB * 2 * W_N, &g.ws));
    SGP_TRY(S.take(PB * 2 * (LMAX + 1), &g.st));
    for (int q = 0; q < 2; ++q) {
        SGP_TRY(S.take(NP + PB, &g.sp_slot[q]));
        SGP_TRY(S.take(NP + PB, &g.sp_n[q]));
    }
    SGP_TRY(S.take(NP, &g.sgn));
    g.lps = f32 ? SlotSize<float>::LPS : SlotSize<double>::LPS;
    SGP_TRY(S.take(NRmax, &g.d_src));
    SGP_TRY(S.take((size_t)P * NTOP, &g.vm));
    SGP_TRY(S.take(NRmax + NP + NTOP + PB, &g.dcnt));
    SGP_TRY(S.take(NP, &g.plist));
    SGP_TRY(S.take(NP, &g.sgk));
    SGP_TRY(S.take(NP, &g.sgd));
    SGP_TRY(S.take(NP, &g.sgf));
    SGP_TRY(S.take(PB, &g.nseg));
    SGP_TRY(S.take(PB * 2 * LMAX * NCLS, &g.kb));
    SGP_TRY(S.take(NTOP, &g.clen));
    SGP_TRY(S.take(NTOP, &g.rlen));
    SGP_TRY(S.take(NTOP, &g.cptr));
    SGP_TRY(S.take(NTOP, &g.rptr));
    SGP_TRY(S.take((size_t)NTOP * CMAX, &g.cidx));
    SGP_TRY(S.take((size_t)NTOP * CMAX * 9, &g.cx));
    SGP_CUDA(ctx, cudaMemsetAsync(g.rlen, 0, sizeof(int32_t) * NTOP, ctx->stream));
    g.lp = lp; g.seg = seg; g.sp = sp; g.lpos = lpos;
    if (f32) g.col32 = reinterpret_cast<const float2 *>(bp<const float4>(M->blk32) + 2 * M->m);
    SGP_CUDA(ctx, cudaMemsetAsync(g.tot, 0, sizeof(int32_t) * T_N, ctx->stream));
    LAUNCH(ctx, k_gr_rows, 1, 256, 0, P, NI, d_ipart, nblk, (const int32_t *)off, g.hdr, g.tot);
    if (U > NREC / 2) {
        // near the end of the range the largest part decides (a third over the
        // mean at 1e6 cells in FP64): not the rest of the layout for nothing
        // (factor of 1e6 cells, FP64: 3.22 ms with the whole layout, 2.76 so, 2.52
        // without any)
        std::vector<int32_t> hd((size_t)Q_N * P);
        SGP_TRY(read_back(ctx, hd.data(), g.hdr, sizeof(int32_t) * hd.size()));
        for (int32_t b = 0; b < P; ++b)
            if (too_large(hd[(size_t)Q_N * b + Q_NR])) return SGP_OK;
    }
    const unsigned gy = (unsigned)std::max(1, std::min(8, U / GT));
    SGP_TRY(sgp_launch(ctx, "k_gr_row_maps", k_gr_row_maps, dim3(P, gy), dim3(GT), 0, g));
    LAUNCH(ctx, k_gr_part_count, P, GT, 0, g);
    LAUNCH(ctx, k_gr_offsets1, 1, 256, 0, P, g.hdr, g.tot);
    LAUNCH(ctx, k_gr_cols, 3 * NTOP / 96, 96, 0, g, bp<const double>(F->L));
    LAUNCH(ctx, k_gr_top_offsets, 1, 1024, 0, g);
    LAUNCH(ctx, k_gr_part_top<false>, P, GT, 0, g);
    LAUNCH(ctx, k_gr_segments, P, GT, 0, g);
    GridRows &R = G.rows;
    SGP_TRY(rows_count(ctx, R, g, M, NRmax));
    LAUNCH(ctx, k_gr_offsets2, 1, 256, 0, P, g.hdr, g.tot, (const int32_t *)g.ws);
    // sizes to the host
    struct {
        int32_t t[T_N], top[Q_N];
    } hs;
    SGP_TRY(read_back(ctx, hs.t, g.tot, sizeof(hs.t)));
    SGP_TRY(read_back(ctx, hs.top, g.hdr + (size_t)Q_N * P, sizeof(hs.top)));
    SGP_TRY(read_back(ctx, R.tot, g.rh + R_N * P, sizeof(R.tot)));
    memcpy(G.tot, hs.t, sizeof(hs.t));
    if (G.tot[T_ERR] || G.tot[T_MDZ] > NREC) return SGP_OK;
    GridPlace pl;
    const bool rows = rows_place(G, R, M, f32, true), apply = !f32 && place_apply(G, 8, 24, &pl);
    if (!rows && !apply) return SGP_OK;
    G.nr_max = (int64_t)NRmax;
    for (int q = 0; q < 2; ++q) {
        const size_t slots = (size_t)G.tot[q ? T_SB : T_SF];
        SGP_TRY(ensure(ctx, G.prog[q], slots * (f32 ? SlotSize<float>::B : SlotSize<double>::B), &g.prog[q]));
        SGP_TRY(S.take(32 * slots, &g.msrc[q]));
    }
    SGP_TRY(ensure(ctx, G.alist, G.tot[T_A], &g.alist));
    SGP_TRY(ensure(ctx, G.outs, (size_t)G.tot[T_Z] + (size_t)G.tot[T_NT], &g.outs));
    SGP_TRY(ensure(ctx, G.xi, (size_t)G.tot[T_RE] + (size_t)G.tot[T_CE], &g.xi));
    SGP_TRY(ensure(ctx, G.zslot, G.tot[T_Z], &g.zslot));
    SGP_TRY(ensure(ctx, G.tlk, (size_t)G.tot[T_NT] + 1, &g.tlk));
    SGP_TRY(sgp_launch(ctx, "k_gr_program", f32 ? k_gr_program<float> : k_gr_program<double>, dim3(P, 2), dim3(GT), 0, g));
    LAUNCH(ctx, k_gr_part_top<true>, P, GT, 0, g);
    LAUNCH(ctx, k_gr_slots, 1, 1024, 0, g);
    if (rows) SGP_TRY(rows_fill(ctx, G, R, g, M, f32));
    const int32_t *td_src = sp + hs.top[Q_SOFF];
    if (f32)
        SGP_TRY(numeric<float>(ctx, G, F, M, g, td_src));
    else
        SGP_TRY(numeric<double>(ctx, G, F, M, g, td_src));
    LAUNCH(ctx, k_gr_check, P, GT, 0, g);
    SGP_TRY(read_back(ctx, hs.t, g.tot, sizeof(hs.t)));
    if (hs.t[T_ERR]) return sgp_fail(ctx, SGP_ERR_CUDA, "tree_factor: inconsistent grid layout (0x%x)", hs.t[T_ERR]);
    G.prec = F->precision;
    // packets of a forest solve alone (its callers' vectors are FP64)
    G.apply_bytes = 0;
    if (apply) {
        const size_t b = 8 * (size_t)Pkt<double>::W * ((size_t)G.tot[T_Z] + (size_t)G.tot[T_NT]) + 16;
        SGP_TRY(buf_ensure(ctx, G.apply, b));
        G.apply_bytes = b;
    }
    G.ok = 1;
    return SGP_OK;
}

// The rows of another matrix on a factor's parts (the augmented forest's P':
// its product, the factor's preconditioner).  R.ok is 0 when they do not fit.
// Nothing is done when R holds these already (generations are unique: of this
// assembly and this factor build).
sgp_status grid_rows(sgp_ctx *ctx, const sgp_factor *F, const sgp_matrix *M, GridRows &R)
{
    const GridLayout &G = F->gl;
    if (R.mgen == M->gen && R.fgen == F->gen) return SGP_OK;
    R.ok = 0;
    R.mgen = R.fgen = 0;
    const bool f32 = G.prec == SGP_PREC_MIXED;
    if (!G.ok || M->n != F->n || (f32 && M->precision != SGP_PREC_MIXED)) return SGP_OK;
    GBuild g{};
    g.n = (int32_t)M->n; g.P = G.P;
    g.hdr = bp<int32_t>(G.hdr); g.tot = bp<int32_t>(G.dtot);
    g.i_of_t = bp<int32_t>(G.i_of_t); g.t_of_i = bp<int32_t>(G.t_of_i);
    if (f32) g.col32 = reinterpret_cast<const float2 *>(bp<const float4>(M->blk32) + 2 * M->m);
    SGP_TRY(rows_count(ctx, R, g, M, (size_t)G.nr_max));
    SGP_TRY(read_back(ctx, R.tot, g.rh + R_N * g.P, sizeof(R.tot)));
    if (rows_place(G, R, M, f32, true)) SGP_TRY(rows_fill(ctx, G, R, g, M, f32));
    R.mgen = M->gen;
    R.fgen = F->gen;
    return SGP_OK;
}

// A matrix cut into parts of consecutive rows, for the row-wise
// preconditioners, in FP64 or (MIXED matrices) FP32; G.ok is 0 when the parts
// do not fit.  `jac`: the block-Jacobi inverses (internal order), or NULL.
// Nothing is done when G holds this assembly in this form already: 200,000
// cells, FP64, one more block-Jacobi solve of one step 0.36 -> 0.26 ms, of five
// 0.58 -> 0.47 (multi-launch 0.31 and 0.61).
sgp_status grid_plain(sgp_ctx *ctx, const sgp_matrix *M, bool f32, const double *jac, GridLayout &G)
{
    const int32_t n = (int32_t)M->n;
    GridRows &R = G.rows;
    const int prec = f32 ? SGP_PREC_MIXED : SGP_PREC_F64, diag = jac ? 1 : 0;
    if (R.mgen == M->gen && G.prec == prec && G.diag == diag) return SGP_OK;
    G.ok = 0;
    R.mgen = 0;
    G.prec = prec;
    G.diag = diag;
    // FP64 is bound by its issue rate: all SMs from 64 rows each on; FP32 from 128
    int32_t P = part_count(ctx, n, f32 ? 128 : 64);
    const int32_t U = (n + P - 1) / P;
    P = (n + U - 1) / U;
    if ((size_t)U * (f32 ? 24 : 48) > (size_t)GRID_SMEM) {
        R.mgen = M->gen;
        return SGP_OK;
    }
    G.P = P;
    G.nr_max = (int64_t)P * pad32(U) + 32;
    GBuild g{};
    g.n = n; g.P = P; g.identity = 1;
    SGP_TRY(ensure(ctx, G.hdr, (size_t)Q_N * (P + 1), &g.hdr));
    SGP_TRY(ensure(ctx, G.dtot, T_N, &g.tot));
    SGP_TRY(ensure(ctx, G.i_of_t, (size_t)G.nr_max, &g.i_of_t));
    SGP_TRY(ensure(ctx, G.t_of_i, n, &g.t_of_i));
    if (f32) g.col32 = reinterpret_cast<const float2 *>(bp<const float4>(M->blk32) + 2 * M->m);
    SGP_CUDA(ctx, cudaMemsetAsync(g.tot, 0, sizeof(int32_t) * T_N, ctx->stream));
    LAUNCH(ctx, k_gr_rows_plain, 1, 256, 0, n, P, U, g.hdr, g.tot);
    const unsigned gy = (unsigned)std::max(1, std::min(8, U / GT));
    SGP_TRY(sgp_launch(ctx, "k_gr_row_maps", k_gr_row_maps, dim3(P, gy), dim3(GT), 0, g));
    SGP_TRY(rows_count(ctx, R, g, M, (size_t)G.nr_max));
    SGP_TRY(read_back(ctx, R.tot, g.rh + R_N * P, sizeof(R.tot)));
    memset(G.tot, 0, sizeof(G.tot));
    G.tot[T_NR] = (P - 1) * pad32(U) + pad32(n - (P - 1) * U);   // the rows that k_gr_row_maps writes
    G.tot[T_MNR] = U;
    if (!rows_place(G, R, M, f32, false)) {
        R.mgen = M->gen;
        return SGP_OK;
    }
    SGP_TRY(rows_fill(ctx, G, R, g, M, f32));
    R.mgen = 0;   // until the diagonal is there
    if (jac) {
        const int32_t nr = G.tot[T_NR];
        SGP_TRY(buf_ensure(ctx, G.D, (f32 ? 4 : 8) * 6 * (size_t)nr));
        if (f32)
            LAUNCH(ctx, k_gr_pivots<float>, grid_for(nr, SGP_BLOCK), SGP_BLOCK, 0, nr, bp<const int32_t>(G.i_of_t), jac,
                   pivot_scale<float>(M), bp<float>(G.D));
        else
            LAUNCH(ctx, k_gr_pivots<double>, grid_for(nr, SGP_BLOCK), SGP_BLOCK, 0, nr, bp<const int32_t>(G.i_of_t), jac,
                   pivot_scale<double>(M), bp<double>(G.D));
    }
    R.mgen = M->gen;
    G.ok = 1;
    return SGP_OK;
}

void grid_rows_release(GridRows &R)
{
    for (DBuf *d : {&R.rh, &R.glen, &R.gso, &R.perm, &R.xflag, &R.hl, &R.ma, &R.mb, &R.hb, &R.hpre})
        if (d->p) cudaFree(d->p);
}
void grid_release(GridLayout &G)
{
    for (DBuf *d : {&G.hdr, &G.dtot, &G.ws, &G.alist, &G.outs, &G.xi, &G.zslot, &G.tlk, &G.i_of_t, &G.t_of_i, &G.prog[0], &G.prog[1], &G.D,
                    &G.X, &G.tD, &G.apply})
        if (d->p) cudaFree(d->p);
    for (DBuf &d : G.scr)
        if (d.p) cudaFree(d.p);
    grid_rows_release(G.rows);
}


// What serves a tree-preconditioned run in precision T: the factor's layout and
// the matrix's rows on its parts, the factor's own or, for another assembly (a
// factor kept for several steps), put there now; NULL where nothing does.
// (A layout cut for more SMs than the context's stream has cannot be resident.)
// MIXED solve of 1e5 cells with a factor of another assembly: 31.2 -> 11.2 ms
// (its own 10.7; bins 25.5); 1e6: 92.8 -> 54.8 (52.4; 77.5).
template <typename T>
sgp_status grid_serves(sgp_ctx *ctx, const sgp_factor *F, const sgp_matrix *M, const GridLayout **G, const GridRows **R)
{
    *G = nullptr;
    *R = nullptr;
    if (!ctx->fused || !F || !F->gl.ok || !F->gl.rows.ok || F->gl.P > ctx->num_sms || F->gl.prec != (sizeof(T) == 4 ? SGP_PREC_MIXED : SGP_PREC_F64))
        return SGP_OK;
    const GridRows *r = &F->gl.rows;
    if (r->mgen != M->gen) {
        SGP_TRY(grid_rows(ctx, F, M, ctx->grid_rows));
        r = &ctx->grid_rows;
        if (!r->ok) return SGP_OK;
    }
    *G = &F->gl;
    *R = r;
    return SGP_OK;
}
template sgp_status grid_serves<float>(sgp_ctx *, const sgp_factor *, const sgp_matrix *, const GridLayout **, const GridRows **);
template sgp_status grid_serves<double>(sgp_ctx *, const sgp_factor *, const sgp_matrix *, const GridLayout **, const GridRows **);

// The systems of a batched solve, offsets[0..n_inst], on the parts of a
// factor: per part its system's parts and the system.  False without a layout,
// or where a system does not begin and end with instances of the layout.
bool grid_groups(const GridLayout &G, int64_t n_inst, const int64_t *offsets, std::vector<int32_t> &grp)
{
    if (!G.ok) return false;
    grp.assign(3 * (size_t)G.P, 0);
    for (int64_t s = 0; s < n_inst; ++s) {
        if (offsets[s] == offsets[s + 1]) continue;
        const auto a = std::upper_bound(G.irow.begin(), G.irow.end(), offsets[s]) - 1,
                   e = std::lower_bound(G.irow.begin(), G.irow.end(), offsets[s + 1]);
        if (a < G.irow.begin() || *a != offsets[s] || e == G.irow.end() || *e != offsets[s + 1]) return false;
        const int32_t p0 = G.ipart[a - G.irow.begin()], p1 = G.ipart[e - G.irow.begin()];
        for (int32_t p = p0; p < p1; ++p) {
            grp[3 * p] = p0;
            grp[3 * p + 1] = p1;
            grp[3 * p + 2] = (int32_t)s;
        }
    }
    return true;
}

// Device workspace of one grid solve in bytes (element size sz, ng systems).
size_t grid_work_bytes(const GridLayout &G, size_t sz, int ng)
{
    if (!G.ok) return 0;
    const int32_t *t = G.tot;
    const size_t wb = sz == 4 ? 32 : 48, nr = (size_t)t[T_NR];
    return 3 * (3 * sz * nr + 256) + wb * (nr + (size_t)t[T_NT] + (size_t)t[T_Z]) + 512 + 2 * PMAX * 4 * 8 + 2048 +
           sizeof(Scal) * (size_t)ng;
}

static void top_args(const GridLayout &G, GridArgs &a)
{
    a.alist = bp<const int4>(G.alist); a.outs = bp<const int4>(G.outs);
    a.xi = bp<const int32_t>(G.xi);
    a.X = G.X.p; a.tD = G.tD.p;
}

// x = P^-1 b of an FP64 factor in one launch, without a host synchronisation;
// a wait that gives up leaves NaN and sets the context's word (gave_up).  orig_of: the caller's order, or NULL for
// the internal one; nothing is done when *done is set.
bool grid_apply_ready(const sgp_ctx *ctx, const sgp_factor *F)
{
    return ctx->fused && F->gl.ok && F->gl.prec == SGP_PREC_F64 && F->gl.apply_bytes > 0 && F->gl.P <= ctx->num_sms;
}
sgp_status grid_apply(sgp_ctx *ctx, const sgp_factor *F, const DBuf &ws, const double *b, double *x, const int32_t *orig_of,
                      const int *done)
{
    const GridLayout &G = F->gl;
    const int32_t *t = G.tot;
    GridArgs a{};
    if (!place_apply(G, 8, 24, &a.pl)) return sgp_fail(ctx, SGP_ERR_CUDA, "tree solve: the grid layout does not fit");
    a.P = G.P; a.nt = t[T_NT]; a.nslots = t[T_Z];
    a.hdr = bp<const int32_t>(G.hdr); a.ws = bp<const int32_t>(G.ws);
    a.i_of_t = bp<const int32_t>(G.i_of_t);
    top_args(G, a);
    a.zslot = bp<const int32_t>(G.zslot); a.tlk = bp<const int32_t>(G.tlk);
    for (int q = 0; q < 2; ++q) a.prog[q] = bp<const char>(G.prog[q]);
    a.D = G.D.p;
    a.F = b; a.x = x;
    a.err = bp<int>(ws);
    a.gave_up = ctx->d_gave_up;
    a.skew = ctx->skew;
    a.lx = reinterpret_cast<unsigned long long *>(ws.p) + 2;
    SGP_CUDA(ctx, cudaMemsetAsync(ws.p, 0, G.apply_bytes, ctx->stream));
    if (ctx->skew) SGP_CUDA(ctx, cudaMemsetAsync(a.err, 1, sizeof(int), ctx->stream));   // (waits that fail are short)
    void *args[] = {&a, &orig_of, &done};
    const auto kern = k_apply_grid<double, 24>;
    SGP_CUDA(ctx, cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, GRID_SMEM));
    SGP_CUDA(ctx, cudaLaunchCooperativeKernel((const void *)kern, dim3(G.P), dim3(GT), args, (size_t)a.pl.bytes, ctx->stream));
    ctx->launches++;
    return SGP_OK;
}

// One PCG run on Gamma x = F (vectors in the matrix's internal order) in one
// launch: the parts and the forest of `G` (precond TREE), or parts of rows
// (block Jacobi, none), the matrix's rows `R`; the final scalars go to *hs (a
// Scal).
template <typename T>
sgp_status grid_pcg(sgp_ctx *ctx, const sgp_matrix *M, const GridLayout &G, const GridRows &R, int precond, const T *F, T *x,
                    int x_given, double tol, int64_t maxit, void *work, void *hs, double mu, int stopE,
                    const GridGroups *groups)
{
    const int ng = groups ? groups->n : 1;
    const int32_t *t = G.tot;
    const bool tree = precond == SGP_PRECOND_TREE;
    GridArgs a{};
    if (!place(G, R.tot[2], sizeof(T), R.vb, tree, R.halo != 0, &a.pl))
        return sgp_fail(ctx, SGP_ERR_CUDA, "pcg: the grid layout does not fit");
    char *at = reinterpret_cast<char *>(work);
    auto take = [&](size_t b) {
        char *p = at;
        at += (b + 255) & ~size_t(255);
        return p;
    };
    struct Out {
        unsigned long long ns[4];
        int err, pad;
        Scal sc[1];
    };
    const size_t out_bytes = sizeof(Out) + sizeof(Scal) * (size_t)(ng - 1);
    const size_t wb = 8 * (size_t)Pkt<T>::W, nr = (size_t)t[T_NR];
    char *zero = take(0);
    a.pk = reinterpret_cast<unsigned long long *>(take(2 * PMAX * 4 * 8));
    a.lx = reinterpret_cast<unsigned long long *>(take(wb * ((size_t)t[T_Z] + (size_t)t[T_NT])));
    Out *out = reinterpret_cast<Out *>(take(out_bytes));
    if (R.halo) a.px = reinterpret_cast<unsigned long long *>(take(wb * nr));
    char *zend = take(0);
    if (!R.halo) a.pg = take(3 * sizeof(T) * nr);
    if (a.pl.o_r < 0) a.r = take(3 * sizeof(T) * nr);
    if (a.pl.o_x < 0) a.xt = take(3 * sizeof(T) * nr);
    a.P = G.P; a.nt = tree ? t[T_NT] : 0; a.x_given = x_given; a.timing = ctx->timing; a.halo = R.halo;
    a.nslots = t[T_Z];
    a.hdr = bp<const int32_t>(G.hdr); a.rh = bp<const int32_t>(R.rh); a.ws = bp<const int32_t>(G.ws);
    a.glen = bp<const int32_t>(R.glen); a.gso = bp<const int32_t>(R.gso); a.i_of_t = bp<const int32_t>(G.i_of_t);
    top_args(G, a);
    a.zslot = bp<const int32_t>(G.zslot); a.tlk = bp<const int32_t>(G.tlk);
    a.hl = bp<const int32_t>(R.hl);
    a.perm = bp<const uint16_t>(R.perm); a.xflag = bp<const uint8_t>(R.xflag);
    for (int q = 0; q < 2; ++q) a.prog[q] = bp<const char>(G.prog[q]);
    a.D = a.jac = G.D.p; a.ma = R.ma.p; a.mb = R.mb.p;
    a.F = F; a.x = x;
    a.gamma0 = M->gamma0;
    a.tol2 = stopE ? -1.0 : tol * tol;
    a.tolE2 = tol * tol;
    a.mu = mu;
    a.maxit = maxit;
    a.stopE = stopE;
    a.err = &out->err;
    a.skew = ctx->skew;
    a.sc = out->sc;
    if (groups) {
        a.grp = groups->grp;
        a.gtol2 = groups->tol2;
    }
    a.ns = out->ns;
    SGP_CUDA(ctx, cudaMemsetAsync(zero, 0, (size_t)(zend - zero), ctx->stream));
    if (ctx->skew) SGP_CUDA(ctx, cudaMemsetAsync(a.err, 1, sizeof(int), ctx->stream));
    void *args[] = {&a};
    auto go = [&](auto kern) -> sgp_status {
        SGP_CUDA(ctx, cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, GRID_SMEM));
        SGP_CUDA(ctx, cudaLaunchCooperativeKernel((const void *)kern, dim3(G.P), dim3(GT), args, (size_t)a.pl.bytes,
                                                  ctx->stream));
        return SGP_OK;
    };
    auto pick = [&](auto vb) -> sgp_status {
        constexpr int VB = decltype(vb)::value;
        if (precond == SGP_PRECOND_BLOCK_JACOBI) return go(k_pcg_grid<T, VB, 1>);
        if (precond == SGP_PRECOND_NONE) return go(k_pcg_grid<T, VB, 2>);
        return go(k_pcg_grid<T, VB, 0>);
    };
    if constexpr (sizeof(T) == 8)
        SGP_TRY(pick(std::integral_constant<int, 24>{}));
    else if (R.vb == 16)
        SGP_TRY(pick(std::integral_constant<int, 16>{}));
    else
        SGP_TRY(pick(std::integral_constant<int, 12>{}));
    ctx->launches++;
    std::vector<char> hb(out_bytes);
    SGP_TRY(read_back(ctx, hb.data(), out, out_bytes));
    Out h;
    std::memcpy(&h, hb.data(), sizeof(h));
    Scal *so = reinterpret_cast<Scal *>(hs);
    std::memcpy(so, hb.data() + offsetof(Out, sc), sizeof(Scal) * (size_t)ng);
    if (h.err)
        for (int k = 0; k < ng; ++k) {
            so[k].status = SGP_ERR_TIMEOUT;
            so[k].done = 1;
        }
    if (ctx->timing) {
        const int cls[3] = {SGP_KT_SPMV, SGP_KT_TREE_SOLVE, SGP_KT_PCG_VECTOR};
        for (int k = 0; k < 3; ++k) {
            if (!tree && k == 1) {   // no tree solve: the vector work
                ctx->kt_ms[SGP_KT_PCG_VECTOR] += 1e-6 * (double)h.ns[1];
                continue;
            }
            ctx->kt_ms[cls[k]] += 1e-6 * (double)h.ns[k];
            ctx->kt_n[cls[k]] += so[0].it + (k == 1);
        }
    }
    return SGP_OK;
}
#define GRID_PCG(T)                                                                                                      \
    template sgp_status grid_pcg<T>(sgp_ctx *, const sgp_matrix *, const GridLayout &, const GridRows &, int, const T *, \
                                    T *, int, double, int64_t, void *, void *, double, int, const GridGroups *);
GRID_PCG(float)
GRID_PCG(double)
