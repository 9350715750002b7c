// k_field.cu -- one explicit field step (rows a1, a2): the no-flux
// neighbour-difference stencil with decay, the optional dense rate map, and
// point-source emission.  These are the unfused kernels: one HBM/L2 round
// trip per step (8 B per node update, 12 B with a rate map).
//
// Update (Sec. 5.2 Eulerian grid, Sec. 4.3 sources with their own rates):
//   C'_i = C_i + alpha * sum_{existing axis nbrs j} (C_j - C_i) - decay * C_i
//          [+ dt * M_i] [+ e_k at source nodes]
// evaluated as beta C_i + alpha sum_j C_j with a missing neighbour (wall)
// replaced by the node itself (node_update2/3).
#include <algorithm>

#include "cue_internal.h"

namespace cue {
namespace {

constexpr unsigned kFull = 0xffffffffu;

__device__ __forceinline__ bool finite4(const float4 &v)
{
    const float big = 3.402823466e38f;
    return fabsf(v.x) <= big && fabsf(v.y) <= big && fabsf(v.z) <= big && fabsf(v.w) <= big;
}

// ---------------------------------------------------------------- 2D, float4
// Block = 32 lanes (x, 4 nodes each) x BY warps (y segments of `rows` rows).
// Each thread streams its 4-wide column strip down its rows, keeping the
// rows above/at/below in registers; x neighbours come from the adjacent lane
// by shuffle, and from global memory at the warp edges.
//
// Point sources are added by the block that owns their node, after the
// update of that node and in source order (the same rounding as a separate
// pass): the block first lists the sources inside its rectangle in shared
// memory, so a block without sources pays one pass over the source table.
constexpr int kBlockSources = 64;

template <bool MAP>
__global__ void __launch_bounds__(256) field2d_vec4(FieldDesc f, const float *__restrict__ Cin,
                                                    float *__restrict__ Cout,
                                                    const float *__restrict__ M, int rows,
                                                    const int32_t *__restrict__ src_cell,
                                                    const float *__restrict__ src_emit, int n_src,
                                                    unsigned *status)
{
    __shared__ int s_n;
    __shared__ int s_cell[kBlockSources];
    __shared__ float s_emit[kBlockSources];
    const int lane = threadIdx.x;
    const int nx4 = f.nx >> 2;
    const int x4 = blockIdx.x * 32 + lane;
    const bool xin = x4 < nx4;
    const int bx0 = blockIdx.x * 128, bx1 = min(bx0 + 128, f.nx);
    const int by0 = blockIdx.y * blockDim.y * rows, by1 = min(by0 + (int)blockDim.y * rows, f.ny);
    const int tid = threadIdx.y * 32 + lane;
    if (tid == 0) s_n = 0;
    __syncthreads();
    for (int k = tid; k < n_src; k += blockDim.x * blockDim.y) {
        const int c = src_cell[k];
        if (c < 0 || (long long)c >= (long long)f.nx * f.ny) {
            if (blockIdx.x == 0 && blockIdx.y == 0) flag_status(status, kStatusBounds);
            continue;
        }
        const int cx = c % f.nx, cy = c / f.nx;
        if (cx >= bx0 && cx < bx1 && cy >= by0 && cy < by1) {
            const int slot = atomicAdd(&s_n, 1);
            if (slot < kBlockSources) {
                s_cell[slot] = k;          // source index first: sorted below
            } else {
                flag_status(status, kStatusBounds);
            }
        }
    }
    __syncthreads();
    const int nb = min(s_n, kBlockSources);
    if (tid == 0 && nb > 1) {          // keep the table's order (ties add as a separate pass would)
        for (int i = 1; i < nb; ++i)
            for (int j = i; j > 0 && s_cell[j - 1] > s_cell[j]; --j) {
                const int t = s_cell[j];
                s_cell[j] = s_cell[j - 1];
                s_cell[j - 1] = t;
            }
    }
    __syncthreads();
    if (tid < nb) {
        const int k = s_cell[tid];
        s_emit[tid] = src_emit[k];
        s_cell[tid] = src_cell[k];
    }
    __syncthreads();
    const int y0 = (blockIdx.y * blockDim.y + threadIdx.y) * rows;
    if (y0 >= f.ny) return;                       // warp-uniform
    const int y1 = min(y0 + rows, f.ny);
    const int x = x4 * 4;
    const bool has_l = x > 0, has_r = x + 4 < f.nx;
    const float4 *in4 = reinterpret_cast<const float4 *>(Cin);
    float4 *out4 = reinterpret_cast<float4 *>(Cout);
    const float4 *m4 = reinterpret_cast<const float4 *>(M);
    const float4 z4 = make_float4(0.f, 0.f, 0.f, 0.f);

    float4 cur = xin ? __ldg(in4 + (size_t)y0 * nx4 + x4) : z4;
    float4 up = (xin && y0 > 0) ? __ldg(in4 + (size_t)(y0 - 1) * nx4 + x4) : cur;
    bool bad = false;
    for (int y = y0; y < y1; ++y) {
        float4 dn = (xin && y + 1 < f.ny) ? __ldg(in4 + (size_t)(y + 1) * nx4 + x4) : cur;
        float l = __shfl_up_sync(kFull, cur.w, 1);
        float r = __shfl_down_sync(kFull, cur.x, 1);
        if (lane == 0) l = (xin && has_l) ? __ldg(Cin + (size_t)y * f.nx + x - 1) : cur.x;
        if (lane == 31) r = (xin && has_r) ? __ldg(Cin + (size_t)y * f.nx + x + 4) : cur.w;
        if (!has_l) l = cur.x;
        if (!has_r) r = cur.w;
        if (xin) {
            float4 o;
            o.x = node_update2(cur.x, l, cur.y, up.x, dn.x, f.alpha, f.beta);
            o.y = node_update2(cur.y, cur.x, cur.z, up.y, dn.y, f.alpha, f.beta);
            o.z = node_update2(cur.z, cur.y, cur.w, up.z, dn.z, f.alpha, f.beta);
            o.w = node_update2(cur.w, cur.z, r, up.w, dn.w, f.alpha, f.beta);
            if constexpr (MAP) {
                float4 m = __ldg(m4 + (size_t)y * nx4 + x4);
                o.x = fmaf(f.dt, m.x, o.x);
                o.y = fmaf(f.dt, m.y, o.y);
                o.z = fmaf(f.dt, m.z, o.z);
                o.w = fmaf(f.dt, m.w, o.w);
            }
            for (int i = 0; i < nb; ++i) {
                const int c = s_cell[i] - y * f.nx - x;
                if (c == 0) o.x += s_emit[i];
                else if (c == 1) o.y += s_emit[i];
                else if (c == 2) o.z += s_emit[i];
                else if (c == 3) o.w += s_emit[i];
            }
            bad |= !finite4(o);
            out4[(size_t)y * nx4 + x4] = o;
        }
        up = cur;
        cur = dn;
    }
    if (__any_sync(kFull, bad) && lane == 0) flag_status(status, kStatusNonFinite);
}

// ---------------------------------------------------------------- 3D, float4
// Block = 32 lanes (x, 4 nodes each) x BY rows (y); each thread streams a
// chunk of z planes keeping z-1, z, z+1 in registers.  y neighbours come from
// a shared-memory copy of the block's plane row set (+1 halo row each side).
template <bool MAP, int BY>
__global__ void __launch_bounds__(32 * BY) field3d_vec4(FieldDesc f, const float *__restrict__ Cin,
                                                         float *__restrict__ Cout,
                                                         const float *__restrict__ M, int zchunk,
                                                         unsigned *status)
{
    __shared__ float4 tile[BY + 2][32];
    const int lane = threadIdx.x, ty = threadIdx.y;
    const int nx4 = f.nx >> 2;
    const int x4 = blockIdx.x * 32 + lane;
    const bool xin = x4 < nx4;
    const int y = blockIdx.y * BY + ty;
    const bool act = xin && y < f.ny;
    const int z0 = blockIdx.z * zchunk;
    const int z1 = min(z0 + zchunk, f.nz);
    const int x = x4 * 4;
    const bool has_l = x > 0, has_r = x + 4 < f.nx;
    const size_t plane4 = (size_t)f.ny * nx4;
    const float4 *in4 = reinterpret_cast<const float4 *>(Cin);
    float4 *out4 = reinterpret_cast<float4 *>(Cout);
    const float4 *m4 = reinterpret_cast<const float4 *>(M);
    const float4 z4 = make_float4(0.f, 0.f, 0.f, 0.f);
    auto at = [&](int yy, int zz) { return (size_t)zz * plane4 + (size_t)yy * nx4 + x4; };

    float4 cur = act ? __ldg(in4 + at(y, z0)) : z4;
    float4 below = (act && z0 > 0) ? __ldg(in4 + at(y, z0 - 1)) : cur;
    bool bad = false;
    for (int z = z0; z < z1; ++z) {
        float4 above = (act && z + 1 < f.nz) ? __ldg(in4 + at(y, z + 1)) : cur;
        tile[ty + 1][lane] = cur;
        if (ty == 0) tile[0][lane] = (xin && y > 0) ? __ldg(in4 + at(y - 1, z)) : z4;
        if (ty == BY - 1) tile[BY + 1][lane] = (xin && y + 1 < f.ny) ? __ldg(in4 + at(y + 1, z)) : z4;
        __syncthreads();
        float4 s = (y > 0) ? tile[ty][lane] : cur;
        float4 n = (y + 1 < f.ny) ? tile[ty + 2][lane] : cur;
        float l = __shfl_up_sync(kFull, cur.w, 1);
        float r = __shfl_down_sync(kFull, cur.x, 1);
        const size_t row = (size_t)z * f.ny * f.nx + (size_t)y * f.nx;
        if (lane == 0) l = (act && has_l) ? __ldg(Cin + row + x - 1) : cur.x;
        if (lane == 31) r = (act && has_r) ? __ldg(Cin + row + x + 4) : cur.w;
        if (!has_l) l = cur.x;
        if (!has_r) r = cur.w;
        if (act) {
            float4 o;
            o.x = node_update3(cur.x, l, cur.y, s.x, n.x, below.x, above.x, f.alpha, f.beta);
            o.y = node_update3(cur.y, cur.x, cur.z, s.y, n.y, below.y, above.y, f.alpha, f.beta);
            o.z = node_update3(cur.z, cur.y, cur.w, s.z, n.z, below.z, above.z, f.alpha, f.beta);
            o.w = node_update3(cur.w, cur.z, r, s.w, n.w, below.w, above.w, f.alpha, f.beta);
            if constexpr (MAP) {
                float4 m = __ldg(m4 + at(y, z));
                o.x = fmaf(f.dt, m.x, o.x);
                o.y = fmaf(f.dt, m.y, o.y);
                o.z = fmaf(f.dt, m.z, o.z);
                o.w = fmaf(f.dt, m.w, o.w);
            }
            bad |= !finite4(o);
            out4[at(y, z)] = o;
        }
        __syncthreads();
        below = cur;
        cur = above;
    }
    if (__any_sync(kFull, bad) && lane == 0) flag_status(status, kStatusNonFinite);
}

// ---------------------------------------------------------------- any size
// Any row length and alignment (nx not a multiple of 4, or a buffer that is not 16-byte aligned): one
// thread per column of the march (y in 2D, z in 3D), so a node's index is worked out once
// per thread and its neighbours along the march stay in registers; the others come from L1.  A launch
// can carry the step's cones (blocks at the start of the grid, kAnyCones each: their chain of dependent loads is the
// longest) and the point sources of its nodes (added once the block's nodes are stored), so a
// coupled step is one launch, and a programmatic dependent one: its blocks are set up while the previous step's
// end.  129 x 97 x 65 with 5,000 cones: 17.3 us a step as three launches with two 64-bit divisions per node
// -> 5.4 (5.3 of it the field's); 255^3 86 -> 69; 2D 2049^2 with 16,384 cones 31 -> 9.3, 4095^2 89 -> 37.
// What bounds it: rows that start anywhere in a sector, so every warp's load and store touches one
// more, and the loads of a step behind the stores of the one before.  Measured and not kept: tiles of 32 x 8
// columns in 3D (6.0), four march steps loaded ahead of their stores (5.6; 4095^2 60).
constexpr int kAnyCones = 128;
constexpr int kAnySources = 1024;             // point sources a block looks through

struct AnyArgs {
    FieldDesc f;
    ConeDesc c;
    const float *Cin;
    float *Cout;
    const float *M;
    int chunk;                                // march steps per block
    unsigned plane_blocks, cone_blocks;
    // cones
    uint32_t step;
    int n;
    float *pos, *dir;
    uint8_t *active;
    const float *src_xyz;
    int n_stop;
    unsigned long long *counter;
    // point sources
    const int32_t *src_cell;
    const float *src_emit;
    int n_add;
    unsigned *status;
};

// A weak load that the compiler may move past this kernel's stores (they go to another buffer), but
// not before the dependency wait: the pointer carries the wait's result.
__device__ __forceinline__ float ld_in(const float *p)
{
    float v;
    asm("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(p));
    return v;
}

template <int DIM, bool MAP>
__global__ void __launch_bounds__(256) step_any(const __grid_constant__ AnyArgs A)
{
    const FieldDesc &f = A.f;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const size_t plane = DIM == 3 ? (size_t)f.nx * f.ny : (size_t)f.nx;
    const int tid = threadIdx.x;
    long long after;                          // 0, once the previous launch's writes are visible
    if (blockIdx.x < A.cone_blocks) {
        asm volatile("griddepcontrol.wait;\n mov.u64 %0, 0;" : "=l"(after)::"memory");
        if (tid >= kAnyCones) return;
        const float *C = A.Cin + after;
        const int a = blockIdx.x * kAnyCones + tid, n = A.n;
        const bool inr = a < n;
        const uint8_t act = inr ? A.active[a] : 0;
        float p[DIM], d[DIM], xi[DIM];
#pragma unroll
        for (int i = 0; i < DIM; ++i) {
            p[i] = inr ? A.pos[(size_t)i * n + a] : 0.0f;
            d[i] = inr ? A.dir[(size_t)i * n + a] : 0.0f;
        }
        cone_noise<DIM>(A.c.key0, A.c.key1, (uint32_t)a, A.step, xi);
        const bool live = inr && act;
        count_active(A.counter, live);
        if (!live) return;
        auto ld = [&](int i, int j, int k) { return ld_in(C + (size_t)i + (size_t)f.nx * j + (DIM == 3 ? plane * k : 0)); };
        const bool alive = cone_step_rule<DIM>(f, A.c, ld, xi, p, d, A.src_xyz, A.n_stop, A.n_stop);
        bool bad = false;
#pragma unroll
        for (int i = 0; i < DIM; ++i) {
            A.pos[(size_t)i * n + a] = p[i];
            A.dir[(size_t)i * n + a] = d[i];
            bad |= !(fabsf(p[i]) <= 3.402823466e38f) || !(fabsf(d[i]) <= 3.402823466e38f);
        }
        if (!alive) A.active[a] = 0;
        if (bad) flag_status(A.status, kStatusNonFinite);
        return;
    }
    const unsigned fb = blockIdx.x - A.cone_blocks, pb = fb % A.plane_blocks, cb = fb / A.plane_blocks;
    const size_t i0 = (size_t)pb * 256, i = i0 + tid;
    const int N = DIM == 3 ? f.nz : f.ny;
    const int z0 = (int)cb * A.chunk, z1 = min(z0 + A.chunk, N);
    const bool in = i < plane;
    const unsigned y = DIM == 3 ? (unsigned)i / (unsigned)f.nx : 0u, x = (unsigned)i - y * (unsigned)f.nx;
    const ptrdiff_t xm = x > 0 ? -1 : 0, xp = x + 1 < (unsigned)f.nx ? 1 : 0;
    const ptrdiff_t ym = DIM == 3 && y > 0 ? -(ptrdiff_t)f.nx : 0, yp = DIM == 3 && y + 1 < (unsigned)f.ny ? (ptrdiff_t)f.nx : 0;
    asm volatile("griddepcontrol.wait;\n mov.u64 %0, 0;" : "=l"(after)::"memory");
    bool bad = false;
    if (in) {
        const float *C = A.Cin + after + plane * z0 + i;
        float *O = A.Cout + plane * z0 + i;
        const float *M = MAP ? A.M + plane * z0 + i : nullptr;
        float c = ld_in(C), m = z0 > 0 ? ld_in(C - plane) : c;
#pragma unroll 4
        for (int z = z0; z < z1; ++z, C += plane, O += plane) {
            const float p = z + 1 < N ? ld_in(C + plane) : c;
            const float l = ld_in(C + xm), r = ld_in(C + xp);
            float o;
            if constexpr (DIM == 3) o = node_update3(c, l, r, ld_in(C + ym), ld_in(C + yp), m, p, f.alpha, f.beta);
            else o = node_update2(c, l, r, m, p, f.alpha, f.beta);
            if constexpr (MAP) {
                o = fmaf(f.dt, __ldg(M), o);
                M += plane;
            }
            bad |= !(fabsf(o) <= 3.402823466e38f);
            *O = o;
            m = c;
            c = p;
        }
    }
    if (__any_sync(0xffffffffu, bad) && (tid & 31) == 0) flag_status(A.status, kStatusNonFinite);
    if (A.n_add > 0) {
        __syncthreads();                      // the block's nodes are stored: their sources (atomic: duplicates add up)
        const long long n_cells = (long long)plane * N;
        for (int k = tid; k < A.n_add; k += 256) {
            const long long cell = __ldg(A.src_cell + k);
            if (cell < 0 || cell >= n_cells) {
                if (fb == 0) flag_status(A.status, kStatusBounds);
                continue;
            }
            const unsigned z = (unsigned)cell / (unsigned)plane, at = (unsigned)cell - z * (unsigned)plane;
            if (at >= i0 && at < i0 + 256 && (int)z >= z0 && (int)z < z1) atomicAdd(A.Cout + cell, __ldg(A.src_emit + k));
        }
    }
}

// Point sources: C'[cell_k] += e_k (atomic, so duplicate cells accumulate).
__global__ void add_sources(float *C, size_t n_cells, const int32_t *__restrict__ cell,
                            const float *__restrict__ emit, int n_src, unsigned *status)
{
    int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= n_src) return;
    int c = cell[s];
    if (c < 0 || (size_t)c >= n_cells) {
        flag_status(status, kStatusBounds);
        return;
    }
    atomicAdd(C + c, emit[s]);
}

// Source node coordinates [3][n_src] for the cones' squared-distance stop test.
__global__ void source_coords(FieldDesc f, const int32_t *__restrict__ cell, int n_src,
                              float *xyz, unsigned *status)
{
    int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= n_src) return;
    long long c = cell[s];
    long long n = (long long)f.nx * f.ny * f.nz;
    if (c < 0 || c >= n) {
        flag_status(status, kStatusBounds);     // far away: never triggers the stop test
        xyz[s] = xyz[n_src + s] = xyz[2 * n_src + s] = 3.0e38f;
        return;
    }
    xyz[s] = (float)(c % f.nx) * f.h;
    xyz[n_src + s] = (float)((c / f.nx) % f.ny) * f.h;
    xyz[2 * n_src + s] = (float)(c / ((long long)f.nx * f.ny)) * f.h;
}

int sm_count()
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

}  // namespace

// One launch of step_any: the field, the cones with `cones`, and the sources where the caller can be told.
static cudaError_t launch_any(Sim &s, const float *Cin, float *Cout, bool cones, bool *sources_done)
{
    const FieldDesc &f = s.fd;
    AnyArgs A{};
    A.f = f;
    A.c = s.cd;
    A.Cin = Cin;
    A.Cout = Cout;
    A.M = s.src_map;
    const size_t plane = f.dim == 3 ? (size_t)f.nx * f.ny : (size_t)f.nx;
    const int N = f.dim == 3 ? f.nz : f.ny;
    A.plane_blocks = (unsigned)((plane + 255) / 256);
    // as many blocks as the SMs hold (8 each) when the march is long enough to be cut
    long long chunks = std::max(1LL, std::min<long long>(N, 8LL * sm_count() / A.plane_blocks));
    A.chunk = (int)((N + chunks - 1) / chunks);
    chunks = (N + A.chunk - 1) / A.chunk;
    A.step = (uint32_t)s.cone_step;
    A.n = cones ? s.n_axons : 0;
    A.cone_blocks = (unsigned)((A.n + kAnyCones - 1) / kAnyCones);
    A.pos = s.pos;
    A.dir = s.dir;
    A.active = s.active;
    A.src_xyz = s.src_xyz();
    A.n_stop = s.cd.stop_r2 >= 0.0f ? s.n_src : 0;
    A.counter = s.cone_counter();
    A.src_cell = s.src_cell;
    A.src_emit = s.src_emit;
    A.n_add = sources_done && s.n_src <= kAnySources ? s.n_src : 0;
    if (sources_done) *sources_done = A.n_add == s.n_src;
    A.status = s.status();
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(A.cone_blocks + A.plane_blocks * chunks));
    cfg.blockDim = dim3(256);
    cfg.stream = s.stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const bool map = s.src_map != nullptr;
    if (f.dim == 3) return map ? cudaLaunchKernelEx(&cfg, step_any<3, true>, A) : cudaLaunchKernelEx(&cfg, step_any<3, false>, A);
    return map ? cudaLaunchKernelEx(&cfg, step_any<2, true>, A) : cudaLaunchKernelEx(&cfg, step_any<2, false>, A);
}

cudaError_t launch_step_any(Sim &s, const float *Cin, float *Cout, bool *sources_done)
{
    timing_begin(s);
    const cudaError_t e = launch_any(s, Cin, Cout, true, sources_done);
    timing_end(s);
    s.launches++;
    return e;
}

cudaError_t launch_field_step(Sim &s, const float *Cin, float *Cout, bool *sources_done)
{
    const FieldDesc &f = s.fd;
    const bool map = s.src_map != nullptr;
    if (sources_done) *sources_done = false;
    timing_begin(s);
    if (s.vec4 && f.dim == 2) {
        const int nx4 = f.nx / 4;
        const int BY = 8;
        const int xb = (nx4 + 31) / 32;
        // rows per thread: the most register reuse that still leaves >= 4 blocks per SM
        int rows = s.rows_per_thread;
        if (rows <= 0) {
            rows = 8;
            while (rows > 1 && (long long)xb * ((f.ny + BY * rows - 1) / (BY * rows)) < 4LL * sm_count())
                rows /= 2;
        }
        dim3 grid(xb, (f.ny + BY * rows - 1) / (BY * rows));
        dim3 block(32, BY);
        const int ns = (sources_done && s.n_src <= kBlockSources) ? s.n_src : 0;
        if (map)
            field2d_vec4<true><<<grid, block, 0, s.stream>>>(f, Cin, Cout, s.src_map, rows, s.src_cell, s.src_emit,
                                                             ns, s.status());
        else
            field2d_vec4<false><<<grid, block, 0, s.stream>>>(f, Cin, Cout, nullptr, rows, s.src_cell, s.src_emit,
                                                              ns, s.status());
        if (sources_done) *sources_done = ns == s.n_src;
    } else if (s.vec4 && f.dim == 3 && (Cin == s.field[0] || Cin == s.field[1]) && field3d_tma_prepare(s)) {
        cudaError_t e = launch_field3d_tma(s, Cin == s.field[0] ? 0 : 1, Cout, nullptr, sources_done);
        timing_end(s);
        s.launches++;
        return e;
    } else if (s.vec4 && f.dim == 3) {
        constexpr int BY = 8;
        const int nx4 = f.nx / 4;
        const int xb = (nx4 + 31) / 32, yb = (f.ny + BY - 1) / BY;
        const long long target = 8LL * sm_count();
        int zchunk = f.nz;
        while (zchunk > 8 && (long long)xb * yb * ((f.nz + zchunk - 1) / zchunk) < target) zchunk /= 2;
        dim3 grid(xb, yb, (f.nz + zchunk - 1) / zchunk);
        dim3 block(32, BY);
        if (map) field3d_vec4<true, BY><<<grid, block, 0, s.stream>>>(f, Cin, Cout, s.src_map, zchunk, s.status());
        else field3d_vec4<false, BY><<<grid, block, 0, s.stream>>>(f, Cin, Cout, nullptr, zchunk, s.status());
    } else {
        const cudaError_t e = launch_any(s, Cin, Cout, false, nullptr);
        if (e != cudaSuccess) return e;
    }
    timing_end(s);
    s.launches++;
    return cudaGetLastError();
}

cudaError_t launch_field_and_sources(Sim &s, const float *Cin, float *Cout)
{
    bool done = false;
    cudaError_t e = launch_field_step(s, Cin, Cout, &done);
    if (e == cudaSuccess && !done) e = launch_sources(s, Cout);
    return e;
}

cudaError_t launch_sources(Sim &s, float *Cout)
{
    if (s.n_src == 0) return cudaSuccess;
    const size_t n = (size_t)s.fd.nx * s.fd.ny * s.fd.nz;
    add_sources<<<(s.n_src + 127) / 128, 128, 0, s.stream>>>(Cout, n, s.src_cell, s.src_emit, s.n_src,
                                                             s.status());
    s.launches++;
    return cudaGetLastError();
}

cudaError_t launch_src_xyz(Sim &s)
{
    if (s.n_src == 0) return cudaSuccess;
    source_coords<<<(s.n_src + 127) / 128, 128, 0, s.stream>>>(s.fd, s.src_cell, s.n_src, s.src_xyz(),
                                                               s.status());
    s.launches++;
    return cudaGetLastError();
}

}  // namespace cue
