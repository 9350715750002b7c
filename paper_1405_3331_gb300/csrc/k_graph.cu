// k_graph.cu -- the connectivity stage (include/cue_graph.h): uniform-grid
// binning (hash, sort, cell start; Sec. 3.5, Table 1), growth-cone / neuron
// connections (squared distances; Sec. 3.3), the adjacency list (Fig. 4) and
// level-synchronous breadth-first search (Fig. 5).
//
// The sort is a counting sort: cell counts (atomics), an exclusive scan, a
// scatter, then each cell's ids put in order by one thread, so the result is
// the (cell, id) order whatever order the atomics ran in.  Cell and distance
// decisions are taken in FP64 (a few operations per point or candidate pair),
// the precision of the definition they implement.
#include <algorithm>

#include "cue_barrier.cuh"
#include "cue_graph.h"
#include "cue_internal.h"

namespace cue {
namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kScanBlock = 1024;

size_t al256(size_t x) { return (x + 255) & ~(size_t)255; }
int blocks_of(long long n, int per) { return (int)((n + per - 1) / per); }

// ---------------------------------------------------------------- exclusive scan
// Block-wise scan of 1024 entries (warp shuffles, then the warp totals), the
// block totals scanned by one block with a running carry, then added back.
__device__ __forceinline__ int block_inclusive(int x, int *warp_tot)
{
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(kFull, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) warp_tot[w] = x;
    __syncthreads();
    if (w == 0) {
        int t = lane < (int)(blockDim.x >> 5) ? warp_tot[lane] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(kFull, t, o);
            if (lane >= o) t += y;
        }
        warp_tot[lane] = t;
    }
    __syncthreads();
    const int r = x + (w > 0 ? warp_tot[w - 1] : 0);
    __syncthreads();                                     // warp_tot is reused by the next call
    return r;
}

__global__ void __launch_bounds__(kScanBlock) scan_blocks(const int *in, int *out, int n, int *sums)
{
    __shared__ int warp_tot[32];
    const int i = blockIdx.x * kScanBlock + threadIdx.x;
    const int v = i < n ? in[i] : 0;
    const int incl = block_inclusive(v, warp_tot);
    if (i < n) out[i] = incl - v;
    if (threadIdx.x == kScanBlock - 1) sums[blockIdx.x] = incl;
}

__global__ void __launch_bounds__(kScanBlock) scan_sums(int *sums, int nb)
{
    __shared__ int warp_tot[32];
    __shared__ int carry;
    if (threadIdx.x == 0) carry = 0;
    __syncthreads();
    for (int base = 0; base < nb; base += kScanBlock) {
        const int i = base + threadIdx.x;
        const int v = i < nb ? sums[i] : 0;
        const int incl = block_inclusive(v, warp_tot);
        const int c = carry;
        if (i < nb) sums[i] = c + incl - v;
        __syncthreads();
        if (threadIdx.x == kScanBlock - 1) carry = c + incl;
        __syncthreads();
    }
}

__global__ void scan_add(int *out, int n, const int *sums)
{
    const int i = blockIdx.x * kScanBlock + threadIdx.x;
    if (i < n) out[i] += sums[blockIdx.x];
}

size_t scan_ws(long long n) { return al256(sizeof(int) * (size_t)std::max(1, blocks_of(n, kScanBlock))); }

cudaError_t exclusive_scan(const int *in, int *out, int n, int *sums, cudaStream_t st)
{
    if (n <= 0) return cudaSuccess;
    const int nb = blocks_of(n, kScanBlock);
    scan_blocks<<<nb, kScanBlock, 0, st>>>(in, out, n, sums);
    scan_sums<<<1, kScanBlock, 0, st>>>(sums, nb);
    scan_add<<<nb, kScanBlock, 0, st>>>(out, n, sums);
    return cudaGetLastError();
}

// ---------------------------------------------------------------- binning
struct Grid3 {
    int dim, g[3];
    float cell, inv;
    bool fast;                                           // axis_cell without the division
};

// floor(x / cell) in 64 bits, clamped to the grid.  Up to 2^22 cells an axis the FP32 product x (1 / cell)
// is off by less than one, so it names the cell or a neighbour, and the sign of x - k cell (exact: 23 + 24 bits)
// settles which; the quotient itself is never rounded up to an integer it does not reach (x and cell have
// 24 bits, so they are at least 2^-24 apart).  An FP64 division per axis and point was most of the hash and
// connection kernels: GB300's FP64 rate is a small fraction of its FP32 rate.
__device__ __forceinline__ int axis_cell(float xf, const Grid3 &G, int ax)
{
    const double x = (double)xf, cell = (double)G.cell;
    if (!G.fast) {
        long long k = (long long)floor(x / cell);
        k = k < 0 ? 0 : k;
        k = k > G.g[ax] - 1 ? G.g[ax] - 1 : k;
        return (int)k;
    }
    int k = (int)floorf(fminf(fmaxf(xf * G.inv, 0.0f), (float)G.g[ax]));      // (NaN: 0)
    const double t = x - (double)k * cell;
    k += t < 0.0 ? -1 : t >= cell ? 1 : 0;
    return min(max(k, 0), G.g[ax] - 1);
}

__global__ void bin_hash(Grid3 G, int n, const float *__restrict__ pos, int *cell_of, int *count)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    long long c = 0, stride = 1;
    for (int ax = 0; ax < G.dim; ++ax) {
        c += (long long)axis_cell(pos[(size_t)ax * n + i], G, ax) * stride;
        stride *= G.g[ax];
    }
    cell_of[i] = (int)c;
    atomicAdd(count + c, 1);
}

__global__ void bin_scatter(int n, const int *__restrict__ cell_of, const int *__restrict__ start, int *cursor,
                            int *sorted_id, int *sorted_cell)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int c = cell_of[i];
    const int slot = start[c] + atomicAdd(cursor + c, 1);
    sorted_id[slot] = i;
    sorted_cell[slot] = c;
}

// Each cell's ids in ascending order (insertion sort by the cell's thread).
__global__ void sort_segments(int nseg, const int *__restrict__ start, const int *__restrict__ count, int *ids)
{
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= nseg) return;
    const int b = start[c], k = count[c];
    for (int i = b + 1; i < b + k; ++i) {
        const int v = ids[i];
        int j = i - 1;
        while (j >= b && ids[j] > v) {
            ids[j + 1] = ids[j];
            --j;
        }
        ids[j + 1] = v;
    }
}

// The paper's identifyCellStart: one thread per sorted entry; where the cell id
// differs from the previous (next) entry's, this entry starts (ends) its cell.
__global__ void identify_cell_start(int n, const int *__restrict__ sorted_cell, int *cell_start, int *cell_end)
{
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= n) return;
    const int c = sorted_cell[j];
    if (j == 0 || sorted_cell[j - 1] != c) cell_start[c] = j;
    if (j == n - 1 || sorted_cell[j + 1] != c) cell_end[c] = j + 1;
}

struct BinLayout {
    size_t count, start, cursor, sorted_cell, sums, total;
};

BinLayout bin_layout(int n, long long ncell)
{
    BinLayout L{};
    size_t off = 0;
    L.count = off;
    off += al256(sizeof(int) * (size_t)ncell);
    L.start = off;
    off += al256(sizeof(int) * (size_t)ncell);
    L.cursor = off;
    off += al256(sizeof(int) * (size_t)ncell);
    L.sorted_cell = off;
    off += al256(sizeof(int) * (size_t)std::max(n, 1));
    L.sums = off;
    off += scan_ws(ncell);
    L.total = off;
    return L;
}

bool grid_ok(int dim, const int32_t *grid, long long *ncell)
{
    if ((dim != 2 && dim != 3) || !grid) return false;
    long long nc = 1;
    for (int ax = 0; ax < dim; ++ax) {
        if (grid[ax] < 1) return false;
        nc *= grid[ax];
        if (nc > (1LL << 30)) return false;
    }
    *ncell = nc;
    return true;
}

Grid3 make_grid(int dim, const int32_t *grid, float cell)
{
    Grid3 G{};
    G.dim = dim;
    G.g[0] = grid[0];
    G.g[1] = grid[1];
    G.g[2] = dim == 3 ? grid[2] : 1;
    G.cell = cell;
    G.inv = 1.0f / cell;
    G.fast = cell >= 1e-30f && cell <= 1e30f && G.g[0] <= 1 << 22 && G.g[1] <= 1 << 22 && G.g[2] <= 1 << 22;
    return G;
}

// ---------------------------------------------------------------- connections
// One thread per cone.  The three cells of a row (x - 1, x, x + 1) are neighbours in the
// binned order too, so a row is one run of sorted ids, and its cell bounds are loaded
// together.  A thread keeps its first matches in registers and a warp takes its output
// slots with one atomic.  1,048,576 cones on 262,144 neurons: 300 -> 210 us a call.
constexpr int kConnectKeep = 4;

__global__ void __launch_bounds__(128) connect_kernel(Grid3 G, int n_cones, const float *__restrict__ pos, const int *__restrict__ owner,
                               const uint8_t *__restrict__ active, int n_neurons, const float *__restrict__ npos,
                               double r2, const int *__restrict__ sorted_id, const int *__restrict__ cell_start,
                               const int *__restrict__ cell_end, int cap, int *src, int *dst, int *count)
{
    const int a = blockIdx.x * blockDim.x + threadIdx.x, lane = threadIdx.x & 31;
    const bool on = a < n_cones && (!active || active[a]);
    double x[3] = {0.0, 0.0, 0.0};
    int k[3] = {0, 0, 0}, me = 0;
    if (on) {
#pragma unroll
        for (int ax = 0; ax < 3; ++ax)
            if (ax < G.dim) {
                const float p = pos[(size_t)ax * n_cones + a];
                x[ax] = (double)p;
                k[ax] = axis_cell(p, G, ax);
            }
        me = owner[a];
    }
    const int zr = G.dim == 3 ? 1 : 0;
    // every match of this cone, in a fixed order.  A plane's nine cell bounds go out together (a cell
    // outside the grid stands in by its neighbour, which changes no run), and its runs' ids four at a time
    auto each = [&](const auto &fn) {
        const int x0 = max(k[0] - 1, 0), x1 = min(k[0] + 1, G.g[0] - 1);
        for (int dz = -zr; dz <= zr; ++dz) {
            const int cz = k[2] + dz;
            if (cz < 0 || cz >= G.g[2]) continue;
            int cb[3][3], ce[3][3];
#pragma unroll
            for (int dy = 0; dy < 3; ++dy) {
                const int cy = min(max(k[1] + dy - 1, 0), G.g[1] - 1);
                const long long c = (long long)G.g[0] * (cy + (long long)G.g[1] * cz);
                const int cx[3] = {x0, k[0], x1};
#pragma unroll
                for (int q = 0; q < 3; ++q) {
                    cb[dy][q] = cell_start[c + cx[q]];
                    ce[dy][q] = cell_end[c + cx[q]];
                }
            }
            int b[3], len[3];
#pragma unroll
            for (int dy = 0; dy < 3; ++dy) {
                b[dy] = 0x7fffffff;
                int e = -1;
#pragma unroll
                for (int q = 0; q < 3; ++q)
                    if (cb[dy][q] >= 0) {               // (empty cells hold -1)
                        b[dy] = min(b[dy], cb[dy][q]);
                        e = max(e, ce[dy][q]);
                    }
                const int cy = k[1] + dy - 1;
                len[dy] = e < 0 || cy < 0 || cy >= G.g[1] ? 0 : e - b[dy];
            }
            const int n = len[0] + len[1] + len[2];
            for (int i0 = 0; i0 < n; i0 += 4) {
                int id[4];
                float p[4][3];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int i = min(i0 + q, n - 1);
                    const int j = i < len[0] ? b[0] + i : i < len[0] + len[1] ? b[1] + i - len[0] : b[2] + i - len[0] - len[1];
                    id[q] = sorted_id[j];
                }
#pragma unroll
                for (int q = 0; q < 4; ++q)
#pragma unroll
                    for (int ax = 0; ax < 3; ++ax) p[q][ax] = ax < G.dim ? npos[(size_t)ax * n_neurons + id[q]] : 0.0f;
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    if (i0 + q >= n || id[q] == me) continue;
                    double d2 = 0.0;
#pragma unroll
                    for (int ax = 0; ax < 3; ++ax)
                        if (ax < G.dim) {
                            const double d = x[ax] - (double)p[q][ax];
                            d2 += d * d;
                        }
                    if (d2 < r2) fn(id[q]);
                }
            }
        }
    };
    int found[kConnectKeep], nf = 0;
    if (on)
        each([&](int nid) {
#pragma unroll
            for (int q = 0; q < kConnectKeep; ++q)
                if (nf == q) found[q] = nid;
            nf++;
        });
    int upto = nf;                                       // matches of the warp up to this lane
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, upto, o);
        if (lane >= o) upto += v;
    }
    const int total = __shfl_sync(0xffffffffu, upto, 31);
    if (total == 0) return;
    int slot = 0;
    if (lane == 0) slot = atomicAdd(count, total);
    slot = __shfl_sync(0xffffffffu, slot, 0) + upto - nf;
#pragma unroll
    for (int q = 0; q < kConnectKeep; ++q)
        if (q < nf && slot + q < cap) {
            src[slot + q] = me;
            dst[slot + q] = found[q];
        }
    if (nf > kConnectKeep) {                             // the rest of a cone with many: once more
        int q = 0;
        each([&](int nid) {
            if (q >= kConnectKeep && slot + q < cap) {
                src[slot + q] = me;
                dst[slot + q] = nid;
            }
            ++q;
        });
    }
}

// ---------------------------------------------------------------- adjacency list
__global__ void csr_count(int nv, int ne_cap, const int *__restrict__ d_ne, const int *__restrict__ src,
                          const int *__restrict__ dst, int *deg)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    const int ne = min(*d_ne, ne_cap);
    if (k >= ne) return;
    const int s = src[k], d = dst[k];
    if (s < 0 || s >= nv || d < 0 || d >= nv) return;
    atomicAdd(deg + s, 1);
}

__global__ void csr_scatter(int nv, int ne_cap, const int *__restrict__ d_ne, const int *__restrict__ src,
                            const int *__restrict__ dst, const int *__restrict__ off, int *cursor, int *tmp)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    const int ne = min(*d_ne, ne_cap);
    if (k >= ne) return;
    const int s = src[k], d = dst[k];
    if (s < 0 || s >= nv || d < 0 || d >= nv) return;
    tmp[off[s] + atomicAdd(cursor + s, 1)] = d;
}

// Per vertex: its targets in order, duplicates dropped; uniq[v] their count.
__global__ void csr_dedupe(int nv, const int *__restrict__ off, const int *__restrict__ deg, int *tmp, int *uniq)
{
    const int v = blockIdx.x * blockDim.x + threadIdx.x;
    if (v > nv) return;
    if (v == nv) {
        uniq[nv] = 0;                                    // so the scan's last entry is the total
        return;
    }
    const int b = off[v], k = deg[v];
    for (int i = b + 1; i < b + k; ++i) {
        const int x = tmp[i];
        int j = i - 1;
        while (j >= b && tmp[j] > x) {
            tmp[j + 1] = tmp[j];
            --j;
        }
        tmp[j + 1] = x;
    }
    int m = 0;
    for (int i = b; i < b + k; ++i)
        if (i == b || tmp[i] != tmp[i - 1]) tmp[b + m++] = tmp[i];
    uniq[v] = m;
}

__global__ void csr_compact(int nv, const int *__restrict__ off, const int *__restrict__ uniq,
                            const int *__restrict__ row, const int *__restrict__ tmp, int *col, int *d_m)
{
    const int v = blockIdx.x * blockDim.x + threadIdx.x;
    if (v > nv) return;
    if (v == nv) {
        *d_m = row[nv];
        return;
    }
    for (int i = 0; i < uniq[v]; ++i) col[row[v] + i] = tmp[off[v] + i];
}

struct CsrLayout {
    size_t deg, off, cursor, tmp, uniq, sums, total;
};

CsrLayout csr_layout(int nv, int ne_cap)
{
    CsrLayout L{};
    size_t off = 0;
    L.deg = off;
    off += al256(sizeof(int) * (size_t)(nv + 1));
    L.off = off;
    off += al256(sizeof(int) * (size_t)(nv + 1));
    L.cursor = off;
    off += al256(sizeof(int) * (size_t)(nv + 1));
    L.tmp = off;
    off += al256(sizeof(int) * (size_t)std::max(ne_cap, 1));
    L.uniq = off;
    off += al256(sizeof(int) * (size_t)(nv + 1));
    L.sums = off;
    off += scan_ws(nv + 1);
    L.total = off;
    return L;
}

// ---------------------------------------------------------------- breadth-first search
// Fig. 5's arrays: F (frontier), X (visited, here level >= 0), C (cost =
// level).  Fig. 5 sets F[nid] in the same pass that reads F, so a vertex found
// at this level could be expanded within it; the levels stay exact here with
// two frontier arrays: level L expands the vertices of F[L % 2] and writes the
// vertices it finds into F[(L + 1) % 2], each claimed once by a compare-and-swap
// of its level from -1 to L + 1, then the grid meets at one barrier (the level
// synchronisation the text describes).  Three flag words rotate: level L sets
// flag[L % 3] when it finds a vertex and clears flag[(L + 1) % 3], last read
// after the barrier before the previous one.
//
// Most levels of a sparse graph hold a few thousand vertices, and a level over the whole
// grid costs its barrier (9.8 us a level over 1,024 blocks).  So the search starts on one
// thread-block cluster (bfs_cluster_kernel): its queues and the visited map lie in distributed
// shared memory, and a level ends at the hardware's cluster barrier.  When a level is
// sent more than kBfsWide finds (or a queue overflows) the cluster stops and bfs_kernel, over all
// SMs, goes on from the levels written so far: `from` says where ({done, level}; null: from the source).
// 262,144 vertices, 786,432 edges, 88 levels: 890 -> 390 us a call (4 us a level: the row, its edges and
// the barrier, one after the other).  Measured and not kept: claiming by a compare-and-swap of the level before
// the send (480; each claim waits for L2), the block's finds staged and handed out together (690).
__global__ void __launch_bounds__(256) bfs_kernel(int nv, const int *__restrict__ row, const int *__restrict__ col,
                                                  int source, int *level, uint8_t *F0, uint8_t *F1, int *flag,
                                                  PBar *bar, unsigned expected, long long limit, unsigned *status,
                                                  const int *from)
{
    if (from && from[0]) return;                         // the cluster finished (every block sees it)
    const int stride = gridDim.x * blockDim.x;
    const int t0 = blockIdx.x * blockDim.x + threadIdx.x;
    const int first = from ? from[1] : 0;
    for (int v = t0; v < nv; v += stride) {
        if (!from) level[v] = v == source ? 0 : -1;
        const int l = from ? __ldcg(level + v) : level[v];
        const uint8_t in = l >= 0 && l == first;         // (the cluster has reached none beyond `first`)
        F0[v] = first & 1 ? 0 : in;
        F1[v] = first & 1 ? in : 0;
    }
    if (!grid_barrier(bar, expected, limit, status)) return;
    for (int L = first; L < nv; ++L) {
        uint8_t *Fc = (L & 1) ? F1 : F0, *Fn = (L & 1) ? F0 : F1;
        bool found = false;
        for (int v = t0; v < nv; v += stride) {
            if (!__ldcg(Fc + v)) continue;
            Fc[v] = 0;
            const int e1 = row[v + 1];
            for (int e = row[v]; e < e1; ++e) {
                const int u = col[e];
                if (__ldcg(level + u) < 0 && atomicCAS(level + u, -1, L + 1) == -1) {
                    Fn[u] = 1;
                    found = true;
                }
            }
        }
        if (t0 == 0) flag[(L + 1) % 3] = 0;
        if (__syncthreads_or(found) && threadIdx.x == 0) flag[L % 3] = 1;
        if (!grid_barrier(bar, expected, limit, status)) return;
        if (!__ldcg(flag + L % 3)) break;
    }
}

constexpr int kBfsThreads = 1024;
constexpr int kBfsQueue = 16384;             // finds a block can be sent for a level (two queues), an equal part by each block
constexpr int kBfsMaxVertices = 1 << 22;     // bits of the visited map over a cluster of 16 (32 KB a block)
constexpr int kBfsWide = 65536;              // a level that was sent more finds goes to all SMs

__device__ __forceinline__ uint32_t cluster_addr(const void *p, int rank)
{
    uint32_t a = (uint32_t)__cvta_generic_to_shared(p), r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    return r;
}

__device__ __forceinline__ void st_cluster(void *p, int rank, int v)
{
    asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(cluster_addr(p, rank)), "r"(v) : "memory");
}

__device__ __forceinline__ void cluster_sync_all()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Vertex u belongs to block u % G, which alone knows (a bit in its shared memory) whether it was
// reached.  At level L a block goes over the vertices it was sent, drops those it has seen, writes the others'
// level and sends their edges' ends to the blocks they belong to, into the sender's own part of
// their queues: no atomic leaves a block, and nothing waits for memory but the row and its edges.
// state: {1 when the search is complete, else 0; the level to go on from, whose vertices all carry it}.
// level is -1 everywhere at the start.
__global__ void __launch_bounds__(kBfsThreads) bfs_cluster_kernel(int nv, const int *__restrict__ row, const int *__restrict__ col,
                                                                  int source, int *level, int *state)
{
    extern __shared__ int queue[];                       // [2][G][kBfsQueue / G], then the visited map
    unsigned *seen = reinterpret_cast<unsigned *>(queue + 2 * kBfsQueue);
    __shared__ int cnt[2][16], tot[2][16], over[2];      // by level parity and sender: finds sent here; to anyone; some lost
    __shared__ int s_out[16];                            // finds of this level by the block they go to
    int G, rank;
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(G));
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
    const int tid = threadIdx.x, lane = tid & 31, part = kBfsQueue / G;
    const int words = (nv / G + 32) >> 5;
    for (int i = tid; i < words; i += kBfsThreads) seen[i] = 0;
    const bool valid = source >= 0 && source < nv;
    if (tid < 16) {
        cnt[0][tid] = tid == 0 && valid && source % G == rank;
        tot[0][tid] = tid == 0 && valid;
        s_out[tid] = 0;
    }
    if (tid == 0) {
        over[0] = over[1] = 0;
        queue[0] = source;
    }
    cluster_sync_all();
    const int per = kBfsThreads / G, from = tid / per;   // this thread's sender
    int L = 0;
    bool wide = false;
    for (; L < nv; ++L) {
        const int par = L & 1;
        const int sent = __reduce_add_sync(0xffffffffu, lane < G ? tot[par][lane] : 0);
        if (sent == 0) break;
        wide = over[par] != 0 || sent > kBfsWide;        // (the same in every thread of the cluster)
        if (wide) break;
        const int *q = queue + par * kBfsQueue + from * part;
        int *qn = queue + (par ^ 1) * kBfsQueue + rank * part;
        const int n = cnt[par][from];
        for (int i = tid - from * per; i < n; i += per) {
            const int v = q[i], at = v / G;
            const unsigned bit = 1u << (at & 31);
            if (atomicOr(&seen[at >> 5], bit) & bit) continue;
            level[v] = L;
            const int e1 = row[v + 1];
            for (int e = row[v]; e < e1; e += 4) {       // four edges at a time: their ends are loaded together
                int u[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) u[k] = e + k < e1 ? col[e + k] : -1;
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    if (u[k] >= 0) {
                        const int to = u[k] % G, slot = atomicAdd(&s_out[to], 1);
                        if (slot < part) st_cluster(qn + slot, to, u[k]);
                    }
            }
        }
        __syncthreads();
        if (tid < 32) {
            const int k = lane < G ? s_out[lane] : 0;
            const int all = __reduce_add_sync(0xffffffffu, k);
            const bool lost = __any_sync(0xffffffffu, k > part);
            if (lane < G) {
                st_cluster(&cnt[par ^ 1][rank], lane, min(k, part));
                st_cluster(&tot[par ^ 1][rank], lane, all);
                if (lost) st_cluster(&over[par ^ 1], lane, 1);
                s_out[lane] = 0;
            }
            if (lane == 0) over[par] = 0;
        }
        cluster_sync_all();
    }
    if (tid == 0 && rank == 0) {
        state[0] = wide ? 0 : 1;
        state[1] = L - 1;                                // (a wide level has a level before it)
    }
    cluster_sync_all();                                  // no block leaves while another may still write to it
}

int bfs_smem(int nv, int G) { return (2 * kBfsQueue + (nv / G + 32) / 32 + 1) * (int)sizeof(int); }

// Blocks of the cluster the search starts on: 16 where the device can schedule it, else 8, else 0 (none).
int bfs_find_cluster_size()
{
    const int smem = bfs_smem(kBfsMaxVertices, 16);
    int best = 0;
    if (cudaFuncSetAttribute(bfs_cluster_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) == cudaSuccess &&
        cudaFuncSetAttribute(bfs_cluster_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess)
        for (int g = 16; g >= 8 && best == 0; g /= 2) {
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3(g);
            cfg.blockDim = dim3(kBfsThreads);
            cfg.dynamicSmemBytes = smem;
            cudaLaunchAttribute attr[1];
            attr[0].id = cudaLaunchAttributeClusterDimension;
            attr[0].val.clusterDim.x = g;
            attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
            cfg.attrs = attr;
            cfg.numAttrs = 1;
            int n = 0;
            if (cudaOccupancyMaxActiveClusters(&n, bfs_cluster_kernel, &cfg) == cudaSuccess && n > 0) best = g;
        }
    if (best < 16) cudaGetLastError();                   // a size the device refuses is no error of the caller's
    return best;
}

int bfs_cluster_size()
{
    static PerDevice size;
    return size.on_current(bfs_find_cluster_size);
}

cudaError_t launch_bfs_cluster(int G, int nv, const int *row, const int *col, int source, int *level, int *state, cudaStream_t st)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(G);
    cfg.blockDim = dim3(kBfsThreads);
    cfg.dynamicSmemBytes = bfs_smem(nv, G);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = G;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, bfs_cluster_kernel, nv, row, col, source, level, state);
}

struct BfsLayout {
    size_t status, bar, flag, F, U, total;
};

BfsLayout bfs_layout(int nv)
{
    BfsLayout L{};
    L.status = 0;
    L.bar = 256;
    L.flag = 512;
    L.F = 768;
    L.U = L.F + al256((size_t)std::max(nv, 1));
    L.total = L.U + al256((size_t)std::max(nv, 1));
    return L;
}

int sm_count_g()
{
    static int n = 0;
    if (n == 0) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
        if (n <= 0) n = 152;
    }
    return n;
}

bool ws_ok(const void *ws, size_t have, size_t need)
{
    return ws && have >= need && (reinterpret_cast<uintptr_t>(ws) & 255u) == 0;
}

}  // namespace
}  // namespace cue

using namespace cue;

extern "C" {

size_t cue_bin_workspace_bytes(int32_t n, int64_t n_cells)
{
    if (n < 0 || n_cells <= 0 || n_cells > (1LL << 30)) return 0;
    return bin_layout(n, n_cells).total;
}

int cue_bin_points(int32_t dim, int32_t n, const float *d_pos, float cell, const int32_t *grid, int32_t *d_cell_of,
                   int32_t *d_sorted_id, int32_t *d_cell_start, int32_t *d_cell_end, void *d_ws, size_t ws_bytes,
                   void *stream)
{
    long long ncell = 0;
    if (!grid_ok(dim, grid, &ncell) || n < 0 || !(cell > 0.0f) || !std::isfinite(cell)) return CUE_ERR_ARG;
    if (n > 0 && (!d_pos || !d_cell_of || !d_sorted_id)) return CUE_ERR_ARG;
    if (!d_cell_start || !d_cell_end) return CUE_ERR_ARG;
    const BinLayout L = bin_layout(n, ncell);
    if (!ws_ok(d_ws, ws_bytes, L.total)) return CUE_ERR_WORKSPACE;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    unsigned char *W = static_cast<unsigned char *>(d_ws);
    int *count = reinterpret_cast<int *>(W + L.count), *start = reinterpret_cast<int *>(W + L.start);
    int *cursor = reinterpret_cast<int *>(W + L.cursor), *scell = reinterpret_cast<int *>(W + L.sorted_cell);
    int *sums = reinterpret_cast<int *>(W + L.sums);
    const Grid3 G = make_grid(dim, grid, cell);
    if (cudaMemsetAsync(count, 0, sizeof(int) * ncell, st) != cudaSuccess ||
        cudaMemsetAsync(cursor, 0, sizeof(int) * ncell, st) != cudaSuccess ||
        cudaMemsetAsync(d_cell_start, 0xFF, sizeof(int) * ncell, st) != cudaSuccess ||
        cudaMemsetAsync(d_cell_end, 0xFF, sizeof(int) * ncell, st) != cudaSuccess)
        return CUE_ERR_CUDA;
    if (n == 0) return CUE_OK;
    bin_hash<<<blocks_of(n, 256), 256, 0, st>>>(G, n, d_pos, d_cell_of, count);
    if (exclusive_scan(count, start, (int)ncell, sums, st) != cudaSuccess) return CUE_ERR_CUDA;
    bin_scatter<<<blocks_of(n, 256), 256, 0, st>>>(n, d_cell_of, start, cursor, d_sorted_id, scell);
    sort_segments<<<blocks_of(ncell, 256), 256, 0, st>>>((int)ncell, start, count, d_sorted_id);
    identify_cell_start<<<blocks_of(n, 256), 256, 0, st>>>(n, scell, d_cell_start, d_cell_end);
    return cudaGetLastError() == cudaSuccess ? CUE_OK : CUE_ERR_CUDA;
}

int cue_connect(int32_t dim, int32_t n_cones, const float *d_pos, const int32_t *d_owner, const uint8_t *d_active,
                int32_t n_neurons, const float *d_npos, float radius, float cell, const int32_t *grid,
                const int32_t *d_sorted_id, const int32_t *d_cell_start, const int32_t *d_cell_end, int32_t cap,
                int32_t *d_src, int32_t *d_dst, int32_t *d_count, void *stream)
{
    long long ncell = 0;
    if (!grid_ok(dim, grid, &ncell) || n_cones < 0 || n_neurons < 0 || cap < 0 || !d_count) return CUE_ERR_ARG;
    if (!(radius >= 0.0f) || !(cell >= radius) || !std::isfinite(cell) || !(cell > 0.0f)) return CUE_ERR_ARG;
    if (n_cones > 0 && (!d_pos || !d_owner)) return CUE_ERR_ARG;
    if (n_neurons > 0 && (!d_npos || !d_sorted_id || !d_cell_start || !d_cell_end)) return CUE_ERR_ARG;
    if (cap > 0 && (!d_src || !d_dst)) return CUE_ERR_ARG;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (cudaMemsetAsync(d_count, 0, sizeof(int32_t), st) != cudaSuccess) return CUE_ERR_CUDA;
    if (n_cones == 0 || n_neurons == 0) return CUE_OK;
    const Grid3 G = make_grid(dim, grid, cell);
    connect_kernel<<<blocks_of(n_cones, 128), 128, 0, st>>>(G, n_cones, d_pos, d_owner, d_active, n_neurons, d_npos,
                                                            (double)radius * (double)radius, d_sorted_id,
                                                            d_cell_start, d_cell_end, cap, d_src, d_dst, d_count);
    return cudaGetLastError() == cudaSuccess ? CUE_OK : CUE_ERR_CUDA;
}

size_t cue_csr_workspace_bytes(int32_t nv, int32_t ne_cap)
{
    if (nv < 0 || ne_cap < 0 || nv >= (1 << 30)) return 0;
    return csr_layout(nv, ne_cap).total;
}

int cue_csr_build(int32_t nv, int32_t ne_cap, const int32_t *d_ne, const int32_t *d_src, const int32_t *d_dst,
                  int32_t *d_row, int32_t *d_col, int32_t *d_m, void *d_ws, size_t ws_bytes, void *stream)
{
    if (nv < 0 || nv >= (1 << 30) || ne_cap < 0 || !d_ne || !d_row || !d_m) return CUE_ERR_ARG;
    if (ne_cap > 0 && (!d_src || !d_dst || !d_col)) return CUE_ERR_ARG;
    const CsrLayout L = csr_layout(nv, ne_cap);
    if (!ws_ok(d_ws, ws_bytes, L.total)) return CUE_ERR_WORKSPACE;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    unsigned char *W = static_cast<unsigned char *>(d_ws);
    int *deg = reinterpret_cast<int *>(W + L.deg), *off = reinterpret_cast<int *>(W + L.off);
    int *cursor = reinterpret_cast<int *>(W + L.cursor), *tmp = reinterpret_cast<int *>(W + L.tmp);
    int *uniq = reinterpret_cast<int *>(W + L.uniq), *sums = reinterpret_cast<int *>(W + L.sums);
    if (cudaMemsetAsync(deg, 0, sizeof(int) * (nv + 1), st) != cudaSuccess ||
        cudaMemsetAsync(cursor, 0, sizeof(int) * (nv + 1), st) != cudaSuccess)
        return CUE_ERR_CUDA;
    if (ne_cap > 0) csr_count<<<blocks_of(ne_cap, 256), 256, 0, st>>>(nv, ne_cap, d_ne, d_src, d_dst, deg);
    if (exclusive_scan(deg, off, nv + 1, sums, st) != cudaSuccess) return CUE_ERR_CUDA;
    if (ne_cap > 0)
        csr_scatter<<<blocks_of(ne_cap, 256), 256, 0, st>>>(nv, ne_cap, d_ne, d_src, d_dst, off, cursor, tmp);
    csr_dedupe<<<blocks_of(nv + 1, 256), 256, 0, st>>>(nv, off, deg, tmp, uniq);
    if (exclusive_scan(uniq, d_row, nv + 1, sums, st) != cudaSuccess) return CUE_ERR_CUDA;
    csr_compact<<<blocks_of(nv + 1, 256), 256, 0, st>>>(nv, off, uniq, d_row, tmp, d_col, d_m);
    return cudaGetLastError() == cudaSuccess ? CUE_OK : CUE_ERR_CUDA;
}

size_t cue_bfs_workspace_bytes(int32_t nv)
{
    if (nv < 0) return 0;
    return bfs_layout(nv).total;
}

int cue_bfs(int32_t nv, const int32_t *d_row, const int32_t *d_col, int32_t source, int32_t *d_level, void *d_ws,
            size_t ws_bytes, void *stream)
{
    if (nv < 0 || !d_row || !d_level || (nv > 0 && !d_col)) return CUE_ERR_ARG;
    const BfsLayout L = bfs_layout(nv);
    if (!ws_ok(d_ws, ws_bytes, L.total)) return CUE_ERR_WORKSPACE;
    if (nv == 0) return CUE_OK;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    unsigned char *W = static_cast<unsigned char *>(d_ws);
    int maxb = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&maxb, bfs_kernel, 256, 0) != cudaSuccess || maxb <= 0)
        return CUE_ERR_CUDA;
    const int grid = std::max(1, std::min(blocks_of(nv, 256), maxb * sm_count_g()));
    if (cudaMemsetAsync(W, 0, 768, st) != cudaSuccess) return CUE_ERR_CUDA;   // status, barrier, flags
    // the cluster first; the launch over all SMs returns at once unless a level was too wide for it
    const int G = nv <= kBfsMaxVertices / 16 * bfs_cluster_size() ? bfs_cluster_size() : 0;
    int *state = G > 0 ? reinterpret_cast<int *>(W + L.flag) + 8 : nullptr;
    if (G > 0) {
        if (cudaMemsetAsync(d_level, 0xFF, sizeof(int) * (size_t)nv, st) != cudaSuccess ||
            launch_bfs_cluster(G, nv, d_row, d_col, source, d_level, state, st) != cudaSuccess)
            return CUE_ERR_CUDA;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(256);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cudaError_t e = cudaLaunchKernelEx(&cfg, bfs_kernel, (int)nv, d_row, d_col, (int)source, d_level,
                                       reinterpret_cast<uint8_t *>(W + L.F), reinterpret_cast<uint8_t *>(W + L.U),
                                       reinterpret_cast<int *>(W + L.flag), reinterpret_cast<PBar *>(W + L.bar),
                                       (unsigned)grid, kPersistSpinLimit, reinterpret_cast<unsigned *>(W + L.status),
                                       static_cast<const int *>(state));
    return e == cudaSuccess ? CUE_OK : CUE_ERR_CUDA;
}

int cue_graph_status(void *d_ws, void *stream)
{
    if (!d_ws) return CUE_ERR_ARG;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (cudaStreamSynchronize(st) != cudaSuccess) return CUE_ERR_CUDA;
    unsigned word = 0;
    if (cudaMemcpy(&word, d_ws, sizeof(word), cudaMemcpyDeviceToHost) != cudaSuccess) return CUE_ERR_CUDA;
    if (word && cudaMemset(d_ws, 0, sizeof(word)) != cudaSuccess) return CUE_ERR_CUDA;
    return (word & kStatusTimeout) ? CUE_ERR_TIMEOUT : CUE_OK;
}

}  // extern "C"
