// Create-time kernels: internal cell numbering and the slab layout of the
// netlist for the wirelength kernel (k_wire.cu).  All of them run once per
// handle; nothing here is on the per-iteration path.
//
// Cell numbering: cells whose index is a multiple of kSeedStride start as
// region seeds labelled with their own index; each round, a net (of at most
// kRankMaxDegree pins) takes the smallest label among its cells and every
// cell the smallest label among its nets (Jacobi rounds, so the result does
// not depend on the order in which threads run).  A cell keeps the round in
// which its label last dropped as its distance.  The cells are then numbered
// by (label, distance, index): the cells of one region get consecutive
// numbers, and so do the pins of most nets.  Both orders of the layout (cells,
// and nets by degree and lowest cell number) come from a stable radix sort
// here, so they do not depend on scheduling either.
#include <utility>

#include "fftpl_internal.cuh"

namespace fftpl {

constexpr int kIntMax = 0x7fffffff;

__global__ void k_lp_init(int m, int stride, int* __restrict__ lab, int* __restrict__ next,
                          int* __restrict__ dist) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= m) return;
    bool seed = (i % stride) == 0;
    lab[i] = next[i] = seed ? i : kIntMax;
    dist[i] = seed ? 0 : kIntMax;
}

// netlab[e] = min label over the movable cells of net e (2 <= d <= maxd)
__global__ void k_lp_net(int E, const int* __restrict__ np, const int* __restrict__ pc, int m,
                         int maxd, const int* __restrict__ lab, int* __restrict__ netlab) {
    int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= E) return;
    int p0 = np[e], p1 = np[e + 1], v = kIntMax;
    if (p1 - p0 >= 2 && p1 - p0 <= maxd)
        for (int p = p0; p < p1; ++p) {
            int cc = pc[p];
            if (cc < m) v = min(v, lab[cc]);
        }
    netlab[e] = v;
}

// next[c] = min(next[c], netlab[e]) for every movable cell c of net e (next
// starts a round equal to lab: k_lp_step leaves them so)
__global__ void k_lp_cell(int E, const int* __restrict__ np, const int* __restrict__ pc, int m,
                          const int* __restrict__ netlab, int* __restrict__ next) {
    int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= E) return;
    int v = netlab[e];
    if (v == kIntMax) return;
    for (int p = np[e]; p < np[e + 1]; ++p) {
        int cc = pc[p];
        if (cc < m) atomicMin(next + cc, v);
    }
}

// lab <- next, distance = round + 1 where the label dropped
__global__ void k_lp_step(int m, int round, int* __restrict__ lab, const int* __restrict__ next,
                          int* __restrict__ dist) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= m) return;
    int a = lab[i], b = next[i];
    if (b < a) {
        lab[i] = b;
        dist[i] = round + 1;
    }
}

// key[e] = smallest internal number among the movable cells of net e (m if
// none), val[e] = e
__global__ void k_net_key(int E, const int* __restrict__ np, const int* __restrict__ pc, int m,
                          const int* __restrict__ rank, unsigned* __restrict__ key,
                          int* __restrict__ val) {
    int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= E) return;
    int v = m;
    for (int p = np[e]; p < np[e + 1]; ++p) {
        int cc = pc[p];
        if (cc < m) v = min(v, rank[cc]);
    }
    key[e] = (unsigned)v;
    val[e] = e;
}

// ------------------------------------------------------ stable radix sort
// Eight bits a pass, tiles of kSortTile items: counts per tile and digit, their
// exclusive scan (digits major), then every item to its place; a warp ranks
// its 256 consecutive items 32 at a time, so equal digits keep their order.
constexpr int kSortTile = 2048, kSortThreads = 256, kSortWarps = kSortThreads / 32;

__global__ void __launch_bounds__(kSortThreads)
k_sort_count(int n, int shift, const unsigned* __restrict__ key, int* __restrict__ counts) {
    __shared__ int hist[256];
    hist[threadIdx.x] = 0;
    __syncthreads();
    const int base = blockIdx.x * kSortTile;
    for (int i = threadIdx.x; i < kSortTile; i += kSortThreads)
        if (base + i < n) atomicAdd(&hist[(key[base + i] >> shift) & 255u], 1);
    __syncthreads();
    counts[threadIdx.x * gridDim.x + blockIdx.x] = hist[threadIdx.x];
}

// Exclusive scan of len counts (a multiple of 256) in place, one block, eight
// counts a thread and round.  (One count a thread took 250 us of a pass over
// 2.2M keys.)
__global__ void __launch_bounds__(1024) k_sort_scan(int len, int* __restrict__ counts) {
    __shared__ int warp_tot[32];
    __shared__ int carry;
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    if (threadIdx.x == 0) carry = 0;
    __syncthreads();
    for (int b = 0; b < len; b += 8192) {
        const int i = b + 8 * threadIdx.x;
        int4* at = reinterpret_cast<int4*>(counts + i);
        int4 u = make_int4(0, 0, 0, 0), v = u;
        if (i < len) {
            u = at[0];
            v = at[1];
        }
        const int sum = u.x + u.y + u.z + u.w + v.x + v.y + v.z + v.w;
        int x = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, x, o);
            if (l >= o) x += t;
        }
        if (l == 31) warp_tot[w] = x;
        __syncthreads();
        if (w == 0) {
            int t = warp_tot[l];
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int t2 = __shfl_up_sync(0xffffffffu, t, o);
                if (l >= o) t += t2;
            }
            warp_tot[l] = t;
        }
        __syncthreads();
        int run = carry + (w ? warp_tot[w - 1] : 0) + x - sum;
        if (i < len) {
            int4 q;
            q.x = run; run += u.x;
            q.y = run; run += u.y;
            q.z = run; run += u.z;
            q.w = run; run += u.w;
            at[0] = q;
            q.x = run; run += v.x;
            q.y = run; run += v.y;
            q.z = run; run += v.z;
            q.w = run;
            at[1] = q;
        }
        __syncthreads();
        if (threadIdx.x == 0) carry += warp_tot[31];
        __syncthreads();
    }
}

__global__ void __launch_bounds__(kSortThreads)
k_sort_scatter(int n, int shift, const unsigned* __restrict__ key, const int* __restrict__ val,
               const int* __restrict__ counts, unsigned* __restrict__ key_out,
               int* __restrict__ val_out) {
    __shared__ int at[kSortWarps][256];
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    for (int k = 0; k < kSortWarps; ++k) at[k][threadIdx.x] = 0;
    __syncthreads();
    const int base = blockIdx.x * kSortTile + w * (kSortTile / kSortWarps);
    constexpr int kSteps = kSortTile / kSortThreads;
    for (int k = 0; k < kSteps; ++k) {
        const int i = base + 32 * k + l;
        if (i < n) atomicAdd(&at[w][(key[i] >> shift) & 255u], 1);
    }
    __syncthreads();
    // where each warp's items of digit threadIdx.x go
    int run = counts[threadIdx.x * gridDim.x + blockIdx.x];
    for (int k = 0; k < kSortWarps; ++k) {
        const int c = at[k][threadIdx.x];
        at[k][threadIdx.x] = run;
        run += c;
    }
    __syncthreads();
    for (int k = 0; k < kSteps; ++k) {
        const int i = base + 32 * k + l;
        const unsigned act = __ballot_sync(0xffffffffu, i < n);
        if (i < n) {
            const unsigned kk = key[i], d = (kk >> shift) & 255u;
            const unsigned same = __match_any_sync(act, d);
            const int place = at[w][d] + __popc(same & ((1u << l) - 1u));
            __syncwarp(act);
            if (l == __ffs(same) - 1) at[w][d] += __popc(same);
            key_out[place] = kk;
            val_out[place] = val[i];
        }
        __syncwarp();
    }
}

// cells: sort key (label, distance), value index
__global__ void k_cell_key(int m, const int* __restrict__ lab, const int* __restrict__ dist,
                           unsigned* __restrict__ key, int* __restrict__ val) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= m) return;
    // labels are seeds' indices, multiples of kSeedStride; unreached cells last
    const unsigned l = lab[i] >= m ? (unsigned)(m + kSeedStride - 1) / kSeedStride
                                   : (unsigned)lab[i] / kSeedStride;
    const unsigned d = dist[i] > kLabelRounds ? kLabelRounds + 1 : dist[i];
    key[i] = l * (kLabelRounds + 2) + d;
    val[i] = i;
}

__global__ void k_cell_rank(int m, const int* __restrict__ order, int* __restrict__ rank) {
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q < m) rank[order[q]] = q;
}

// nets in the order given: descending degree, degrees below 2 last
__global__ void k_net_degree_key(int E, int maxd, const int* __restrict__ np,
                                 const int* __restrict__ order, unsigned* __restrict__ key) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= E) return;
    const int e = order[p], d = np[e + 1] - np[e];
    key[p] = (unsigned)(d >= 2 ? maxd - d : maxd - 1);
}

// Pin records in slab layout.  order: the nets of degree >= 2, largest degree
// first; by_degree[d]: place in it of the first net of degree d, and that
// degree's first slot.  With L lanes per net (1, or grp_lanes(d)) and 32 / L
// nets per slab, pin k of the j-th net of its degree is at slot
// first + (j / (32 / L)) 32 ceil(d / L) + (j % (32 / L)) L + 32 (k / L) + k % L.
// A pin on a movable cell stores its cell's internal number and its offset; a
// pin on a fixed cell stores -1 and its absolute coordinate fl32(centre +
// offset).  cslot (deterministic mode, else null): each pin's slot in the
// cell-ordered pin array.
__global__ void k_fill_slabs(int nets, const int* __restrict__ order,
                             const int2* __restrict__ by_degree, const int* __restrict__ np,
                             const int* __restrict__ pc, const float* __restrict__ dx,
                             const float* __restrict__ dy, int m, const int* __restrict__ rank,
                             const float* __restrict__ fix_x, const float* __restrict__ fix_y,
                             const int* __restrict__ cslot, int* __restrict__ spc,
                             float* __restrict__ sdx, float* __restrict__ sdy,
                             int* __restrict__ sslot) {
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= nets) return;
    const int e = order[q];
    const int p0 = np[e], d = np[e + 1] - p0;
    const int L = net_lanes(d), G = 32 / L;
    const int2 first = by_degree[d];
    const int j = q - first.x;
    const size_t base = (size_t)first.y + (size_t)(j / G) * 32 * ((d + L - 1) / L) + (j % G) * L;
    for (int k = 0; k < d; ++k) {
        const int p = p0 + k;
        const size_t slot = base + 32 * (size_t)(k / L) + (size_t)(k % L);
        const int cc = pc[p];
        if (cc < m) {
            spc[slot] = rank[cc];
            sdx[slot] = dx[p];
            sdy[slot] = dy[p];
        } else {
            spc[slot] = -1;
            sdx[slot] = __fadd_rn(fix_x[cc - m], dx[p]);
            sdy[slot] = __fadd_rn(fix_y[cc - m], dy[p]);
        }
        if (sslot) sslot[slot] = cslot[p];
    }
}

static inline unsigned nb(long long n) { return (unsigned)((n + 255) / 256); }

cudaError_t launch_label_rounds(int m, int E, const int* np, const int* pc, int* lab, int* next,
                                int* dist, int* netlab, cudaStream_t s) {
    if (m <= 0) return cudaSuccess;
    k_lp_init<<<nb(m), 256, 0, s>>>(m, kSeedStride, lab, next, dist);
    // no nets: every cell keeps its seed label (or none) at distance 0 / unset
    for (int r = 0; r < (E > 0 ? kLabelRounds : 0); ++r) {
        k_lp_net<<<nb(E), 256, 0, s>>>(E, np, pc, m, kRankMaxDegree, lab, netlab);
        k_lp_cell<<<nb(E), 256, 0, s>>>(E, np, pc, m, netlab, next);
        k_lp_step<<<nb(m), 256, 0, s>>>(m, r, lab, next, dist);
    }
    return cudaGetLastError();
}

size_t sort_counts(int n) { return 256 * (size_t)((n + kSortTile - 1) / kSortTile); }

// Sorts the pairs in buf.key[0], buf.val[0] by the keys' low bits; the result
// is in buf.key[0], buf.val[0].
static cudaError_t sort_pairs(SortBuf& buf, int n, int bits, cudaStream_t s) {
    const int tiles = (n + kSortTile - 1) / kSortTile;
    for (int shift = 0; shift < bits; shift += 8) {
        k_sort_count<<<tiles, kSortThreads, 0, s>>>(n, shift, buf.key[0], buf.counts);
        k_sort_scan<<<1, 1024, 0, s>>>(256 * tiles, buf.counts);
        k_sort_scatter<<<tiles, kSortThreads, 0, s>>>(n, shift, buf.key[0], buf.val[0], buf.counts,
                                                      buf.key[1], buf.val[1]);
        std::swap(buf.key[0], buf.key[1]);
        std::swap(buf.val[0], buf.val[1]);
    }
    return cudaGetLastError();
}

static int bits_of(unsigned v) {
    int b = 0;
    while (v) {
        ++b;
        v >>= 1;
    }
    return b;
}

cudaError_t launch_cell_rank(int m, const int* lab, const int* dist, SortBuf& buf, int* rank,
                             cudaStream_t s) {
    if (m <= 0) return cudaSuccess;
    k_cell_key<<<nb(m), 256, 0, s>>>(m, lab, dist, buf.key[0], buf.val[0]);
    const unsigned top = ((unsigned)(m + kSeedStride - 1) / kSeedStride + 1) * (kLabelRounds + 2);
    cudaError_t e = sort_pairs(buf, m, bits_of(top), s);
    if (e != cudaSuccess) return e;
    k_cell_rank<<<nb(m), 256, 0, s>>>(m, buf.val[0], rank);
    return cudaGetLastError();
}

cudaError_t launch_net_order(int m, int E, int maxd, const int* np, const int* pc, const int* rank,
                             SortBuf& buf, cudaStream_t s) {
    if (E <= 0) return cudaSuccess;
    k_net_key<<<nb(E), 256, 0, s>>>(E, np, pc, m, rank, buf.key[0], buf.val[0]);
    cudaError_t e = sort_pairs(buf, E, bits_of((unsigned)m), s);
    if (e != cudaSuccess) return e;
    k_net_degree_key<<<nb(E), 256, 0, s>>>(E, maxd, np, buf.val[0], buf.key[0]);
    return sort_pairs(buf, E, bits_of((unsigned)maxd), s);
}

cudaError_t launch_fill_slabs(int m, int nets, const int* order, const int2* by_degree,
                              const int* np, const int* pc, const float* dx, const float* dy,
                              const int* rank, const float* fix_x, const float* fix_y,
                              const int* cslot, int* spc, float* sdx, float* sdy, int* sslot,
                              cudaStream_t s) {
    if (nets <= 0) return cudaSuccess;
    k_fill_slabs<<<nb(nets), 256, 0, s>>>(nets, order, by_degree, np, pc, dx, dy, m, rank, fix_x,
                                          fix_y, cslot, spc, sdx, sdy, sslot);
    return cudaGetLastError();
}

}  // namespace fftpl
