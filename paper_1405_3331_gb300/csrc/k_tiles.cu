// k_tiles.cu -- the persistent path's tile engine: one cooperative launch holds
// a whole 2D grid in the SMs' shared memory, one tile per SM, for all its steps.
//
// Each block owns an interior of the grid and loads it once with a halo of
// (HX, HY) nodes around it, in two buffers (C^n and C^{n+1}).  Time runs in
// rounds of K steps: within a round a block advances its own nodes and, one
// node less per step, its halo, without talking to anyone; then it sends the
// border of its interior to its (at most eight) neighbours and refreshes its halo
// from theirs.  So a step costs a sweep and one block barrier, and the grid-wide
// barrier plus the pass over L2 of the work-list kernel (k_persist.cu) becomes an
// exchange of borders once per K steps.
//
// Borders travel as packets: 64-bit words of a value and a tag (the round's
// number, never used again on a handle), written and read with single relaxed
// accesses, so a word that carries the tag carries its value and the receiver
// polls the data itself: no fence, no flag, no second trip to L2.  Packets lie at
// their node's place in two grids that alternate by round: a sender is at most
// one round ahead, because it needs this round's packets from the receiver too.
//
// Field warps (12) hold their rows in registers for a round and write each new
// row to shared memory too, where the cones and the warps above and below read
// it: shared-memory bandwidth, 128 bytes a cycle, bounds a sweep that loads its
// rows too.  The border goes out straight from the registers of the round's last
// step, before that step's barrier.
//
// Cone warps (4): a block steps the cones that are inside
// its interior at the start of a round.  They move at most K step_len in a round
// and read a 4-node footprint, so the halo H = K + 1 + ceil((K - 1) step_len / h)
// holds what they sense.  With two buffers the cones read C^n while C^{n+1} is
// written.  The first 128 cones of a tile ride in the cone warps' registers (with
// at most 64, two warps step them and two draw the next step's noise); of a more
// crowded tile the rest live in shared memory (up to `cap`) or are stepped from
// global memory, and all warps share them out by a ticket.  At the end of a round
// a cone that left the interior is posted to the neighbour it went to: the first
// kTlPost per neighbour with their state, more through the tile's inbox (ids;
// state through the caller's arrays).  An inbox is ordinary memory: who put
// cones into one fences before the number that tells of it, and a tile that took cones from its
// own fences before its next number and says so in it (kTlInboxUsed), on which the neighbours
// fence before they may add to that inbox again.
//
// All tiles have one shape, W = 128 columns (one float4 per lane) by R rows, always inside the
// grid (the last tile of an axis is shifted inwards), so a wall is always the
// first or last loaded column or row, whose missing neighbour is itself: walls
// need no code of their own, and rows of any length (nx not a multiple of 4)
// differ only in how global memory is read and written.
//
// What bounds it: a step's critical path is the longer of a field warp's rows (1,100 cycles for 7 rows of 12
// warps: shuffles and the shared-memory pipe, then the FP32 pipe) and one cone step (1,000 to 1,300 cycles of
// dependent code), the exchange 4,000 to 6,000 cycles a round (16 bytes a cycle out of an SM, 20 in).  Measured and not
// kept: flags instead of tags (a release and an acquire more per round, 5% slower at 1024^2, 9% at 512 x 384),
// two half-sized tiles per SM (more border: 60% slower), 6 or 8 cone warps (10% slower with few cones a tile,
// 20% faster with hundreds), the cone warps on a scheduler of their own (the field's three then bound the step).
//
// The caller's arrays are read once, at the start: a block loads its tile and looks through all
// cones for those inside its interior, then raises its flag.  Until a block knows its neighbours' flags it
// writes neither field nor cone state: a neighbour that came later would find a cone that had
// moved into its interior, take it for its own and step it again.  What goes out in the first
// round (a run of one round, cones that stop, cones past a full list) waits for them where it is written; the
// arrivals warp looks for them in the first exchange, whose last barrier frees every later round.
// The neighbours are enough: no one farther away takes a cone for its own, whatever mix of an old and a new coordinate
// it reads, because a block in its round r has had the exchanges of r rounds, so blocks within r tiles have
// loaded, and a cone it writes came from r tiles away at most and is now one tile away at most.
// (Trajectory mode reads slot 0 and writes the later ones, and its cones do not stop.)
//
// Arithmetic per node and per cone is the plain path's (update4 = node_update2,
// the map as fma(dt, M, C'), sources added after it in index order; cone_step_rule),
// bit for bit.  Every wait is bounded, as in cue_barrier.cuh: past the limit the
// block raises the timeout status and an abort word that makes the others leave.
//
// Model: the cue field on the Eulerian grid of Sec. 5.2, growth cones of Sec. 3.5.
#include <algorithm>
#include <cmath>

#include "cue_internal.h"
#include "cue_tile.cuh"

namespace cue {
namespace {

using tile::kFull;

constexpr int kTlFieldWarps = 12;
constexpr int kTlConeWarps = 4;
constexpr int kTlWarps = kTlFieldWarps + kTlConeWarps;
constexpr int kTlThreads = 32 * kTlWarps;
constexpr int kTlOwn = 32 * kTlConeWarps;    // cones whose state rides in the cone warps' registers
constexpr int kTlHelped = kTlOwn / 2;        // cones whose noise the other half of the cone warps draws
constexpr int kTlMaxSrc = 1024;
constexpr int kTlW = 128;                    // loaded columns: one float4 per lane
constexpr int kTlMaxRows = 15;               // rows of a field warp, in registers
constexpr int kTlPost = kTilesPost;          // cones posted with their state per neighbour and round
constexpr unsigned kTlInboxUsed = 1u << 31;  // beside the number of posted cones
constexpr int kTlFlagWords = 64;             // a flag's stride: a line of its own
constexpr int kTlInFlight = 4;               // rows whose packets a warp polls together

struct TileArgs {
    FieldDesc f;
    ConeDesc c;
    AxisTiles ax, ay;                        // ghost 0; loaded extents W and R
    int gx, gy;                              // tiles per axis
    int K, nsteps, cur0;
    uint32_t step0;
    float *field0, *field1;
    const float *map;
    const int32_t *src_cell;
    const float *src_emit, *src_xyz;
    int n_src, local_stop;
    float *pos, *dir;
    uint8_t *active;
    int n, cap;
    float *traj_field, *traj_cone;           // trajectory mode (see run_tiles_trajectory)
    size_t cells;
    unsigned long long *packets;             // [2][cells]: border nodes, by round parity
    ulonglong2 *post;                        // [2][tiles][9][3 kTlPost + 1]: posted cones, then their number
    int *inbox;                              // [2][tiles][n] cone ids
    int *cnt_cur, *cnt_next;                 // [2][kTilesMax]: this launch's counts (zero at its start), the next's
    unsigned *flags;                         // [tiles], kTlFlagWords apart, only growing: "tile loaded"
    unsigned base;                           // this launch's first tag and its flag; earlier ones' are below it
    unsigned *abort;                         // the aborting launch's base
    int *crowd;                              // the nanoseconds a step that a tile's crowd added (the largest tile's)
    long long limit;
    unsigned *status;
    unsigned long long *counter;
};

__device__ __forceinline__ unsigned ld_acquire_u32(const unsigned *p)
{
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void st_release_u32(unsigned *p, unsigned v)
{
    asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// Packets: {value, tag} words, read and written whole.
__device__ __forceinline__ unsigned long long packet(unsigned v, unsigned tag)
{
    return ((unsigned long long)tag << 32) | v;
}

__device__ __forceinline__ void st_packets(void *p, unsigned long long a, unsigned long long b)
{
    asm volatile("st.relaxed.gpu.global.v2.b64 [%0], {%1, %2};" ::"l"(p), "l"(a), "l"(b) : "memory");
}

__device__ __forceinline__ void ld_packets(const void *p, unsigned long long &a, unsigned long long &b)
{
    asm volatile("ld.relaxed.gpu.global.v2.b64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "l"(p) : "memory");
}

__device__ __forceinline__ void st_packet(void *p, unsigned long long a)
{
    asm volatile("st.relaxed.gpu.global.b64 [%0], %1;" ::"l"(p), "l"(a) : "memory");
}

__device__ __forceinline__ unsigned long long ld_packet(const void *p)
{
    unsigned long long a;
    asm volatile("ld.relaxed.gpu.global.b64 %0, [%1];" : "=l"(a) : "l"(p) : "memory");
    return a;
}

__device__ __forceinline__ bool tagged(unsigned long long a, unsigned tag) { return (unsigned)(a >> 32) == tag; }

// One more look at a wait: false once it has to be given up (the launch is aborting, or the
// limit is reached, which aborts it).
__device__ __forceinline__ bool keep_waiting(long long &it, long long limit, unsigned *abort, unsigned base, unsigned *status)
{
    if ((it & 15) == 15 && *(volatile unsigned *)abort == base) return false;
    if (++it > limit) {
        flag_status(status, kStatusTimeout);
        atomicExch(abort, base);
        return false;
    }
    if (it > 64) __nanosleep(32);
    return true;
}

__device__ __forceinline__ void block_sync() { asm volatile("bar.sync 0;" ::: "memory"); }

// One block's tile: its place, its shared memory and its inboxes.
struct Tile {
    int t, tx, ty;
    int sx, ex, sy, ey;                      // interior
    int ox, oy, R;                           // loaded region (kTlW x R)
    int cx0, cx1, cy0, cy1;                  // cells whose four-node footprint lies in it
    float *S;                                // [2][R][kTlW]
    const float *M;                          // [R][kTlW] or null
    int *l_id;                               // [2][cap] cone ids by list
    float *l_st;                             // [2][4][cap]: x, y, dx, dy
    const float *stop_xy;
    int n_stop;
    __device__ __forceinline__ float &st(int cap, int lb, int k, int i) const { return l_st[(lb * 4 + k) * cap + i]; }
};

__device__ __forceinline__ int *inbox_of(const TileArgs &A, int par, int tl)
{
    return A.inbox + ((size_t)par * (A.gx * A.gy) + tl) * A.n;
}

__device__ __forceinline__ ulonglong2 *post_box(const TileArgs &A, int par, int tl, int dir)
{
    return A.post + ((size_t)(par * kTilesMax + tl) * 9 + dir) * (3 * kTlPost + 1);
}

// Wait until the neighbour in direction `lane` (0..8, 4 the tile itself; none past the grid's edge or
// lane 8) has raised its flag to `want`.  Every lane of the warp; false when it is given up.
__device__ __forceinline__ bool wait_neighbours(const TileArgs &A, int tx, int ty, unsigned want)
{
    const int lane = threadIdx.x & 31;
    const int nx = tx + lane % 3 - 1, ny = ty + lane / 3 - 1;
    bool ok = true;
    if (lane < 9 && lane != 4 && nx >= 0 && nx < A.gx && ny >= 0 && ny < A.gy) {
        const unsigned *flag = A.flags + kTlFlagWords * (ny * A.gx + nx);
        long long it = 0;
        while (ok && (int)(ld_acquire_u32(flag) - want) < 0) ok = keep_waiting(it, A.limit, A.abort, A.base, A.status);
    }
    return __all_sync(kFull, ok);
}

// The same for one lane, in the rare places where a lane alone has cone state to write in the first round; a wait
// given up also ends the block's run.
__device__ __noinline__ bool neighbours_loaded(const TileArgs &A, int tx, int ty, volatile int *s_fail)
{
    bool ok = true;
    long long it = 0;
    for (int q = 0; q < 9 && ok; ++q) {
        const int nx = tx + q % 3 - 1, ny = ty + q / 3 - 1;
        if (q == 4 || nx < 0 || nx >= A.gx || ny < 0 || ny >= A.gy) continue;
        const unsigned *flag = A.flags + kTlFlagWords * (ny * A.gx + nx);
        while (ok && (int)(ld_acquire_u32(flag) - A.base) < 0) ok = keep_waiting(it, A.limit, A.abort, A.base, A.status);
    }
    if (!ok) *s_fail = 1;
    return ok;
}

// Cone state after s steps of this launch: the caller's arrays, or the trajectory's slot.
template <bool TRAJ>
__device__ __forceinline__ float *cone_pos(const TileArgs &A, int s)
{
    return TRAJ ? A.traj_cone + (size_t)s * 4 * A.n : A.pos;
}

template <bool TRAJ>
__device__ __forceinline__ float *cone_dir(const TileArgs &A, int s)
{
    return TRAJ ? A.traj_cone + (size_t)s * 4 * A.n + 2 * (size_t)A.n : A.dir;
}

// One cone step on the tile's field `in`; false when the cone stops.  The cell is kept inside the
// loaded region (a cone is always there: a status bit tells if one ever were not), so that no load
// needs a check of its own; `bits` collects status bits.
__device__ __forceinline__ bool tile_cone_step(const TileArgs &A, const Tile &T, const float *in, const float *xi, float *p,
                                               float *d, unsigned &bits)
{
    const FieldDesc &f = A.f;
    bool alive;
    if (A.c.steer == 0) {
        int lo[2];
        float fr[2], v[kPatch2], g[2];
        cell_of<2>(f, p, lo, fr);
        const int x = clampi(lo[0], T.cx0, T.cx1), y = clampi(lo[1], T.cy0, T.cy1);
        bits |= x != lo[0] || y != lo[1] ? kStatusBounds : 0u;
        lo[0] = x;
        lo[1] = y;
        gather2(f, lo, [&](int i, int j, int) { return in[(j - T.oy) * kTlW + (i - T.ox)]; }, v);
        grad2(A.c, v, fr, g);
        alive = cone_finish_xi<2>(A.c, g, xi, p, d, T.stop_xy, A.n_src, T.n_stop);
    } else {
        const unsigned top = (unsigned)(T.R * kTlW - 1);
        auto ld = [&](int i, int j, int) { return in[min((unsigned)((j - T.oy) * kTlW + (i - T.ox)), top)]; };
        alive = cone_update_snr(f, A.c, ld, xi, p, d, T.stop_xy, A.n_src, T.n_stop);
    }
    const float big = 3.402823466e38f;
    bits |= fabsf(p[0]) <= big && fabsf(p[1]) <= big && fabsf(d[0]) <= big && fabsf(d[1]) <= big ? 0u : kStatusNonFinite;
    return alive;
}

template <bool TRAJ>
__device__ __forceinline__ void put_cone(const TileArgs &A, int s, int a, const float *p, const float *d)
{
    float *gp = cone_pos<TRAJ>(A, s), *gd = cone_dir<TRAJ>(A, s);
    gp[a] = p[0];
    gp[A.n + a] = p[1];
    gd[a] = d[0];
    gd[A.n + a] = d[1];
}

// A crowded tile's cones past the cone warps' registers, a warp's 32 at a time by ticket: from the
// list in shared memory, then from global memory.  Any warp takes part; returns this thread's count.
template <bool TRAJ>
__device__ __noinline__ unsigned crowd_cones(const TileArgs &A, Tile T, const float *in, int s, int lb, int m, int n_ovf,
                                             int *ovf, int *ticket)
{
    const int lane = threadIdx.x & 31, n = A.n, cap = A.cap;
    const float *gp = cone_pos<TRAJ>(A, s), *gd = cone_dir<TRAJ>(A, s);
    unsigned live = 0, bits = 0;
    for (;;) {
        int c = 0;
        if (lane == 0) c = atomicAdd(ticket, 1);
        const int i = kTlOwn + 32 * __shfl_sync(kFull, c, 0) + lane;
        if (i - lane >= m + n_ovf) break;
        int a = -1;
        float p[2], d[2], xi[2];
        if (i < m) {
            a = T.l_id[lb * cap + i];
            p[0] = T.st(cap, lb, 0, i);
            p[1] = T.st(cap, lb, 1, i);
            d[0] = T.st(cap, lb, 2, i);
            d[1] = T.st(cap, lb, 3, i);
        } else if (i < m + n_ovf) {
            a = __ldcg(ovf + i - m);
            if (a >= 0) {
                p[0] = __ldcg(gp + a);
                p[1] = __ldcg(gp + n + a);
                d[0] = __ldcg(gd + a);
                d[1] = __ldcg(gd + n + a);
            }
        }
        if (a < 0) continue;
        live++;
        cone_noise<2>(A.c.key0, A.c.key1, (uint32_t)a, A.step0 + (uint32_t)s, xi);
        const bool alive = tile_cone_step(A, T, in, xi, p, d, bits);
        if (i < m) {
            T.st(cap, lb, 0, i) = p[0];
            T.st(cap, lb, 1, i) = p[1];
            T.st(cap, lb, 2, i) = d[0];
            T.st(cap, lb, 3, i) = d[1];
        }
        if (TRAJ || i >= m || !alive) put_cone<TRAJ>(A, s + 1, a, p, d);
        if (!alive) {                                   // out of the lists
            A.active[a] = 0;
            if (i < m) T.l_id[lb * cap + i] = -1;
            else ovf[i - m] = -1;
        }
    }
    if (bits) flag_status(A.status, bits);
    return live;
}

// What `held` cones of one tile (more than kTlOwn) add to its step, in nanoseconds: the field sweep leaves the registers,
// and the cones past the first 128 queue up.  Measured at 512 x 384, 768^2 and 1280^2 with one crowd, over the
// uncrowded step of 1.0, 1.1 and 1.7 us: 150 cones 1.6, 1.8, 1.6 us; 500: 2.0, 2.1, 2.1; 1,000: 3.2, 3.4, 3.4;
// 2,500: 8.2, 8.6, 8.8; 4,000: 12.9, 13.3, 14.1.
__device__ __forceinline__ float crowd_ns(int held)
{
    return 1300.0f + 1.5f * (float)min(held, 512) + 2.5f * (float)min(max(held - 512, 0), 512) + 3.3f * (float)max(held - 1024, 0);
}

// What a field warp's lane does with its group's four nodes: bit k is node k.
struct LaneMasks {
    int own;                                 // in the interior's columns: published in the rows near a neighbour
    int edge;                                // ... and within HX of one: published in every row
    int halo, halo_side;                     // refreshed in a halo row; in an interior row
};

// A group's new values from its row's x neighbours l and r, the rows above and below, and the map.
template <bool MAP>
__device__ __forceinline__ float4 row_update(const float4 &c, float l, float r, const float4 &u, const float4 &d, const float4 *m,
                                             float2 alpha2, float2 beta2, float dt)
{
    float4 o = tile::update4<false>(l, c, r, u, d, alpha2, beta2, 4);
    if (MAP) o = tile::fma4(dt, *m, o);
    return o;
}

// The x neighbours of a lane's group; past the tile's edge the group's own node (at a wall: no flux).
__device__ __forceinline__ void x_neighbours(const float4 &c, int lane, float &l, float &r)
{
    l = __shfl_up_sync(kFull, c.w, 1);
    r = __shfl_down_sync(kFull, c.x, 1);
    l = lane == 0 ? c.x : l;
    r = lane == 31 ? c.w : r;
}

// The nodes `mask` names of a lane's group to global memory.
template <bool VEC>
__device__ __forceinline__ void put_group(float *g, const float4 &v, int mask)
{
    if constexpr (VEC) {
        if (mask) *reinterpret_cast<float4 *>(g) = v;
    } else {
        if (mask & 1) g[0] = v.x;
        if (mask & 2) g[1] = v.y;
        if (mask & 4) g[2] = v.z;
        if (mask & 8) g[3] = v.w;
    }
}

// The same as packets.
template <bool VEC>
__device__ __forceinline__ void send_group(unsigned long long *g, const float4 &v, int mask, unsigned tag)
{
    if constexpr (VEC) {
        if (!mask) return;
        st_packets(g, packet(__float_as_uint(v.x), tag), packet(__float_as_uint(v.y), tag));
        st_packets(g + 2, packet(__float_as_uint(v.z), tag), packet(__float_as_uint(v.w), tag));
    } else {
        if (mask & 1) st_packet(g, packet(__float_as_uint(v.x), tag));
        if (mask & 2) st_packet(g + 1, packet(__float_as_uint(v.y), tag));
        if (mask & 4) st_packet(g + 2, packet(__float_as_uint(v.z), tag));
        if (mask & 8) st_packet(g + 3, packet(__float_as_uint(v.w), tag));
    }
}

// What of row gy a tile sends at the end of a round.
__device__ __forceinline__ int border_mask(const TileArgs &A, const Tile &T, const LaneMasks &L, int gy)
{
    const bool full = (T.ty > 0 && gy < T.sy + A.ay.H) || (T.ty + 1 < A.gy && gy >= T.ey - A.ay.H);
    return gy < T.sy || gy >= T.ey ? 0 : full ? L.own : L.edge;
}

// One warp's sources in shared memory: [b, e) of the offsets and emissions.
struct WarpSources {
    const int *off;
    const float *e;
    int b, end;
};

// The steps [s0, s0 + kr) of a round on a warp's N rows, held in registers; every new row also goes
// to shared memory, where the cones and the neighbouring warps read it.  One block barrier after each
// step but the last.
template <int N, bool MAP, bool TRAJ, bool VEC>
__device__ __forceinline__ void field_steps(const TileArgs &A, const Tile &T, int r0, int s0, int kr, const LaneMasks &L, const WarpSources &src)
{
    constexpr int W4 = kTlW / 4;
    const FieldDesc &f = A.f;
    const int lane = threadIdx.x & 31, R = T.R, half = R * W4;
    const float2 alpha2 = make_float2(f.alpha, f.alpha), beta2 = make_float2(f.beta, f.beta);
    float4 *S4 = reinterpret_cast<float4 *>(T.S) + r0 * W4 + lane;
    const float4 *M4 = reinterpret_cast<const float4 *>(T.M) + r0 * W4 + lane;
    const int up_off = r0 > 0 ? -W4 : 0, last_off = (r0 + N < R ? N : N - 1) * W4;
    const int gy0 = T.oy + r0;
    float *tout = TRAJ ? A.traj_field + (size_t)(s0 + 1) * A.cells + (size_t)gy0 * f.nx + T.ox + 4 * lane : nullptr;
    int b = s0 & 1;
    float4 v[N];
#pragma unroll
    for (int k = 0; k < N; ++k) v[k] = S4[(b ? half : 0) + k * W4];
    for (int j = 0; j < kr; ++j) {
        const float4 *in4 = S4 + (b ? half : 0);
        float4 *out4 = S4 + (b ? 0 : half);
        const float4 up = in4[up_off], last = in4[last_off];
        // the shuffles run some rows ahead (all of them where registers allow): they hide one another's latency
        constexpr int kAhead = N <= 9 ? N : 4;
        float l[N], r[N];
#pragma unroll
        for (int k = 0; k < kAhead; ++k) x_neighbours(v[k], lane, l[k], r[k]);
        // rows 1 .. N - 1, then row 0: the rows above and below the warp's, just read, come last
        float4 first = last, above = v[0];
        if constexpr (N > 1) {
            first = v[1];
#pragma unroll
            for (int k = 1; k < N; ++k) {
                const float4 old = v[k];
                v[k] = row_update<MAP>(old, l[k], r[k], above, k + 1 < N ? v[k + 1 < N ? k + 1 : k] : last, M4 + k * W4, alpha2, beta2, f.dt);
                out4[k * W4] = v[k];
                above = old;
                if (k + kAhead - 1 < N && k + kAhead - 1 >= kAhead) x_neighbours(v[k + kAhead - 1 < N ? k + kAhead - 1 : 0], lane, l[k + kAhead - 1 < N ? k + kAhead - 1 : 0], r[k + kAhead - 1 < N ? k + kAhead - 1 : 0]);
            }
        }
        v[0] = row_update<MAP>(v[0], l[0], r[0], up, first, M4, alpha2, beta2, f.dt);
        out4[0] = v[0];
        for (int k = src.b; k < src.end; ++k) {         // this warp's sources, in index order
            const int off = src.off[k];
            if (((off & (kTlW - 1)) >> 2) != lane) continue;
            const float e = src.e[k];
            const int rr = (off >> 7) - r0, q = off & 3;
#pragma unroll
            for (int i = 0; i < N; ++i)
                if (rr == i) {
                    if (q == 0) v[i].x += e;
                    else if (q == 1) v[i].y += e;
                    else if (q == 2) v[i].z += e;
                    else v[i].w += e;
                    out4[i * W4] = v[i];
                }
        }
        if constexpr (TRAJ) {
#pragma unroll
            for (int k = 0; k < N; ++k)
                if (gy0 + k >= T.sy && gy0 + k < T.ey) put_group<VEC>(tout + (size_t)k * f.nx, v[k], L.own);
            tout += A.cells;
        }
        if (j + 1 < kr) block_sync();
        b ^= 1;
    }
}

// One step of any number of rows, from shared memory, four rows in flight: the field part of a crowded tile's step.
template <bool MAP, bool TRAJ, bool VEC>
__device__ __noinline__ void field_step_any(const TileArgs &A, Tile T, int r0, int r1, int s, int own, WarpSources src)
{
    constexpr int W4 = kTlW / 4, kB = 4;
    const FieldDesc &f = A.f;
    const int lane = threadIdx.x & 31, R = T.R;
    const float2 alpha2 = make_float2(f.alpha, f.alpha), beta2 = make_float2(f.beta, f.beta);
    const float4 *in4 = reinterpret_cast<const float4 *>(T.S) + (s & 1 ? R * W4 : 0) + lane;
    float4 *out4 = reinterpret_cast<float4 *>(T.S) + (s & 1 ? 0 : R * W4) + lane;
    float *tout = TRAJ ? A.traj_field + (size_t)(s + 1) * A.cells + T.ox + 4 * lane : nullptr;
    for (int q0 = r0; q0 < r1; q0 += kB) {
        float4 v[kB + 2];
#pragma unroll
        for (int u = 0; u < kB + 2; ++u) v[u] = in4[min(max(q0 + u - 1, 0), R - 1) * W4];
        float l[kB], r[kB];
#pragma unroll
        for (int u = 0; u < kB; ++u) x_neighbours(v[u + 1], lane, l[u], r[u]);
#pragma unroll
        for (int u = 0; u < kB; ++u) {
            const int row = q0 + u;
            if (row >= r1) break;
            float4 o = row_update<MAP>(v[u + 1], l[u], r[u], v[u], v[u + 2],
                                       reinterpret_cast<const float4 *>(T.M) + row * W4 + lane, alpha2, beta2, f.dt);
            for (int k = src.b; k < src.end; ++k) {     // (in index order, not by row)
                const int off = src.off[k], q = off & 3;
                if ((off >> 7) != row || ((off & (kTlW - 1)) >> 2) != lane) continue;
                if (q == 0) o.x += src.e[k];
                else if (q == 1) o.y += src.e[k];
                else if (q == 2) o.z += src.e[k];
                else o.w += src.e[k];
            }
            out4[row * W4] = o;
            const int gy = T.oy + row;
            if (TRAJ && gy >= T.sy && gy < T.ey) put_group<VEC>(tout + (size_t)gy * f.nx, o, own);
        }
    }
}

// The border of a field warp's rows (its lanes' own groups in shared memory) to the neighbours.
template <bool VEC>
__device__ __forceinline__ void send_border(const TileArgs &A, const Tile &T, int r0, int r1, int b, const LaneMasks &L,
                                            unsigned long long *packets, unsigned tag)
{
    const int lane = threadIdx.x & 31;
    const float4 *C4 = reinterpret_cast<const float4 *>(T.S) + (b ? T.R * (kTlW / 4) : 0) + lane;
    unsigned long long *pk = packets + T.ox + 4 * lane;
#pragma unroll 4
    for (int r = r0; r < r1; ++r) {
        const int gy = T.oy + r, mask = border_mask(A, T, L, gy);
        if (mask) send_group<VEC>(pk + (size_t)gy * A.f.nx, C4[r * (kTlW / 4)], mask, tag);
    }
}

// The halo of a field warp's rows from the neighbours' packets.  False when the wait was given up.
template <bool VEC>
__device__ __forceinline__ bool receive_halo(const TileArgs &A, const Tile &T, int r0, int r1, int b, const LaneMasks &L,
                                             const unsigned long long *packets, unsigned tag)
{
    constexpr int W4 = kTlW / 4, kB = kTlInFlight;
    const FieldDesc &f = A.f;
    const int lane = threadIdx.x & 31;
    float4 *C4 = reinterpret_cast<float4 *>(T.S) + (b ? T.R * W4 : 0) + lane;
    const unsigned long long *pk = packets + T.ox + 4 * lane;
    bool ok = true;
    long long it = 0;
    for (int k0 = r0; k0 < r1; k0 += kB) {
        int need[kB];
#pragma unroll
        for (int u = 0; u < kB; ++u) {
            const int gy = T.oy + k0 + u;
            need[u] = k0 + u >= r1 || gy < T.sy - A.ay.H || gy >= T.ey + A.ay.H ? 0 : gy < T.sy || gy >= T.ey ? L.halo : L.halo_side;
        }
        bool more;
        do {
            unsigned long long w[kB][4];
#pragma unroll
            for (int u = 0; u < kB; ++u) {
                const unsigned long long *g = pk + (size_t)(T.oy + k0 + u) * f.nx;
                if constexpr (VEC) {
                    if (need[u]) {
                        ld_packets(g, w[u][0], w[u][1]);
                        ld_packets(g + 2, w[u][2], w[u][3]);
                    }
                } else {
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        if (need[u] >> q & 1) w[u][q] = ld_packet(g + q);
                }
            }
            more = false;
#pragma unroll
            for (int u = 0; u < kB; ++u) {
                if (!need[u]) continue;
                float *x = reinterpret_cast<float *>(C4 + (k0 + u) * W4);
                if constexpr (VEC) {
                    if (tagged(w[u][0], tag) && tagged(w[u][1], tag) && tagged(w[u][2], tag) && tagged(w[u][3], tag)) {
                        *reinterpret_cast<float4 *>(x) =
                            make_float4(__uint_as_float((unsigned)w[u][0]), __uint_as_float((unsigned)w[u][1]),
                                        __uint_as_float((unsigned)w[u][2]), __uint_as_float((unsigned)w[u][3]));
                        need[u] = 0;
                    }
                } else {
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        if ((need[u] >> q & 1) && tagged(w[u][q], tag)) {
                            x[q] = __uint_as_float((unsigned)w[u][q]);
                            need[u] &= ~(1 << q);
                        }
                }
                more |= need[u] != 0;
            }
            if (more && ok) ok = keep_waiting(it, A.limit, A.abort, A.base, A.status);
        } while (__any_sync(kFull, more) && __all_sync(kFull, ok));
    }
    return ok;
}

// A field warp's whole run.
template <bool MAP, bool TRAJ, bool VEC>
__device__ __forceinline__ unsigned field_loop(const TileArgs &A, const Tile &T, int r0, int r1, const LaneMasks &L,
                                               const WarpSources &src, int *s_ticket, volatile int *s_list, volatile int *s_fail)
{
    const int nrounds = (A.nsteps + A.K - 1) / A.K;
    unsigned live = 0;
    for (int rd = 0, done = 0; rd < nrounds; ++rd) {
        const int kr = min(A.K, A.nsteps - done);
        const int m = s_list[0], n_ovf = s_list[2];
        const bool last = rd + 1 == nrounds;
        unsigned long long *pk = A.packets + (size_t)(rd & 1) * A.cells;
        const unsigned tag = A.base + (unsigned)rd;
        if (m + n_ovf > kTlOwn) {                       // a crowded tile: this warp helps with the cones
            int *ovf = inbox_of(A, rd & 1, T.t) + s_list[1];
            // (its cones from global memory are written in every step)
            const bool may = TRAJ || rd > 0 || wait_neighbours(A, T.tx, T.ty, A.base);
            if (!may) *s_fail = 1;
            for (int s = done; s < done + kr; ++s) {
                field_step_any<MAP, TRAJ, VEC>(A, T, r0, r1, s, L.own, src);
                if (may) live += crowd_cones<TRAJ>(A, T, T.S + (s & 1 ? T.R * kTlW : 0), s, rd & 1, m, n_ovf, ovf, s_ticket + (s & 1));
                if (s + 1 < done + kr || !last) block_sync();   // (before the last barrier the cone warps place the crowd)
            }
        } else {
            switch (r1 - r0) {
#define CUE_TL_CASE(N) \
    case N: field_steps<N, MAP, TRAJ, VEC>(A, T, r0, done, kr, L, src); break;
                CUE_TL_CASE(1) CUE_TL_CASE(2) CUE_TL_CASE(3) CUE_TL_CASE(4) CUE_TL_CASE(5) CUE_TL_CASE(6)
                CUE_TL_CASE(7) CUE_TL_CASE(8) CUE_TL_CASE(9) CUE_TL_CASE(10) CUE_TL_CASE(11) CUE_TL_CASE(12)
                CUE_TL_CASE(13) CUE_TL_CASE(14) CUE_TL_CASE(15)
#undef CUE_TL_CASE
            default:
                for (int j = 0; j + 1 < kr; ++j) block_sync();  // no rows
            }
        }
        done += kr;
        if (!last) send_border<VEC>(A, T, r0, r1, done & 1, L, pk, tag);
        block_sync();
        if (last) break;
        if (!receive_halo<VEC>(A, T, r0, r1, done & 1, L, pk, tag)) *s_fail = 1;
        block_sync();
        if (*s_fail) break;
    }
    return live;
}

// A cone warp's whole run: its 32 cones of each round's list in registers, the next step's noise drawn
// after the step; between rounds the lists are made anew and the cones that left are posted.
template <bool TRAJ>
__device__ __forceinline__ unsigned cone_loop(const TileArgs &A, const Tile &T, int *s_ticket, volatile int *s_list, volatile int *s_fail,
                                              int *s_push, int *s_out, float *s_xi)
{
    const FieldDesc &f = A.f;
    const int lane = threadIdx.x & 31, cw = (threadIdx.x >> 5) - kTlFieldWarps;
    const int n = A.n, cap = A.cap, R = T.R;
    const int nrounds = (A.nsteps + A.K - 1) / A.K;
    unsigned live = 0, bits = 0;
    int lb = 0;
    float crowd = 0.0f;
    for (int rd = 0, done = 0; rd < nrounds; ++rd) {
        const int kr = min(A.K, A.nsteps - done), par = rd & 1;
        const int m = s_list[0], ovf0 = s_list[1], n_ovf = s_list[2];
        int *ovf = inbox_of(A, par, T.t) + ovf0;
        const int slot = cw * 32 + lane;
        // few cones: the second half of the warps draws the first half's noise a step ahead
        if (m + n_ovf > kTlOwn) crowd += (float)kr * crowd_ns(m + n_ovf);
        const bool helped = m + n_ovf <= kTlHelped;
        const int h_slot = slot - kTlHelped, h_id = helped && h_slot >= 0 && h_slot < m ? T.l_id[lb * cap + h_slot] : -1;
        int a = -1;
        float p[2] = {0.f, 0.f}, d[2] = {0.f, 0.f}, xi[2];
        if (slot < m) {
            a = T.l_id[lb * cap + slot];
            p[0] = T.st(cap, lb, 0, slot);
            p[1] = T.st(cap, lb, 1, slot);
            d[0] = T.st(cap, lb, 2, slot);
            d[1] = T.st(cap, lb, 3, slot);
            cone_noise<2>(A.c.key0, A.c.key1, (uint32_t)a, A.step0 + (uint32_t)done, xi);
        }
        auto own_step = [&](int j) {
            const int s = done + j;
            const float *in = T.S + (s & 1 ? R * kTlW : 0);
            if (a >= 0) {
                live++;
                if (helped && j > 0) {
                    xi[0] = s_xi[(s & 1) * 2 * kTlHelped + slot];
                    xi[1] = s_xi[(s & 1) * 2 * kTlHelped + kTlHelped + slot];
                }
                const bool alive = tile_cone_step(A, T, in, xi, p, d, bits);
                if (TRAJ) put_cone<TRAJ>(A, s + 1, a, p, d);
                if (!alive) {
                    if (TRAJ || rd > 0 || neighbours_loaded(A, T.tx, T.ty, s_fail)) {
                        if (!TRAJ) put_cone<false>(A, 0, a, p, d);
                        A.active[a] = 0;
                    }
                    a = -1;
                } else if (!helped && j + 1 < kr) {
                    cone_noise<2>(A.c.key0, A.c.key1, (uint32_t)a, A.step0 + (uint32_t)(s + 1), xi);
                }
            }
            if (h_id >= 0 && j + 1 < kr) {
                float hx[2];
                cone_noise<2>(A.c.key0, A.c.key1, (uint32_t)h_id, A.step0 + (uint32_t)(s + 1), hx);
                s_xi[((s + 1) & 1) * 2 * kTlHelped + h_slot] = hx[0];
                s_xi[((s + 1) & 1) * 2 * kTlHelped + kTlHelped + h_slot] = hx[1];
            }
        };
        if (m + n_ovf > kTlOwn) {                       // a crowded tile
            const bool may = TRAJ || rd > 0 || wait_neighbours(A, T.tx, T.ty, A.base);
            if (!may) *s_fail = 1;
            for (int j = 0; j < kr; ++j) {
                const int s = done + j;
                own_step(j);
                if (may) live += crowd_cones<TRAJ>(A, T, T.S + (s & 1 ? R * kTlW : 0), s, lb, m, n_ovf, ovf, s_ticket + (s & 1));
                if (cw == 0 && lane == 0) s_ticket[(s & 1) ^ 1] = 0;
                if (j + 1 < kr) block_sync();
            }
        } else {
            for (int j = 0; j < kr; ++j) {
                own_step(j);
                if (j + 1 < kr) block_sync();
            }
        }
        done += kr;
        const bool final = rd + 1 == nrounds;
        if (final) {
            if (!TRAJ) {
                const bool may = rd > 0 || n == 0 || wait_neighbours(A, T.tx, T.ty, A.base);
                if (!may) *s_fail = 1;
                if (may && a >= 0) put_cone<false>(A, 0, a, p, d);
                block_sync();                           // the other warps are done with the list
                for (int i = kTlOwn + slot; may && i < m; i += kTlOwn) {
                    const int c = T.l_id[lb * cap + i];
                    const float cp[2] = {T.st(cap, lb, 0, i), T.st(cap, lb, 1, i)}, cd[2] = {T.st(cap, lb, 2, i), T.st(cap, lb, 3, i)};
                    if (c >= 0) put_cone<false>(A, 0, c, cp, cd);
                }
            } else {
                block_sync();
            }
            break;
        }
        // ---- the next round's list, and the cones that left the interior: the cones in registers before
        // the round's last barrier, a crowded tile's others after it
        const unsigned tag = A.base + (unsigned)rd;
        const int np = par ^ 1, nl = lb ^ 1;
        bool extra = false;                             // a cone went through an inbox
        float *gp = cone_pos<TRAJ>(A, done), *gd = cone_dir<TRAJ>(A, done);
        auto place = [&](int c, const float *cp, const float *cd, bool in_arrays) {       // every lane of the warp
            const int ix = clampi((int)floorf(cp[0] * f.inv_h), 0, f.nx - 1), iy = clampi((int)floorf(cp[1] * f.inv_h), 0, f.ny - 1);
            const int dx = ix < T.sx ? -1 : ix >= T.ex ? 1 : 0, dy = iy < T.sy ? -1 : iy >= T.ey ? 1 : 0;
            const unsigned stay = __ballot_sync(kFull, c >= 0 && dx == 0 && dy == 0);
            int base = 0;
            if (lane == 0 && stay) base = atomicAdd(s_push, __popc(stay));
            base = __shfl_sync(kFull, base, 0);
            if (c < 0) return;
            if (stay >> lane & 1) {
                const int at = base + __popc(stay & ((1u << lane) - 1u));
                if (at < cap) {
                    T.l_id[nl * cap + at] = c;
                    T.st(cap, nl, 0, at) = cp[0];
                    T.st(cap, nl, 1, at) = cp[1];
                    T.st(cap, nl, 2, at) = cd[0];
                    T.st(cap, nl, 3, at) = cd[1];
                    return;
                }
            } else {
                const int dir = 4 + 3 * dy + dx, at = atomicAdd(s_out + dir, 1);
                if (at < kTlPost) {
                    ulonglong2 *e = post_box(A, par, T.t + dy * A.gx + dx, 8 - dir) + 3 * at;
                    st_packets(e, packet((unsigned)c, tag), packet(__float_as_uint(cp[0]), tag));
                    st_packets(e + 1, packet(__float_as_uint(cp[1]), tag), packet(__float_as_uint(cd[0]), tag));
                    st_packets(e + 2, packet(__float_as_uint(cd[1]), tag), packet(0u, tag));
                    return;
                }
            }
            extra = true;
            if (!TRAJ && !in_arrays && (rd > 0 || neighbours_loaded(A, T.tx, T.ty, s_fail))) put_cone<false>(A, 0, c, cp, cd);
            const int to = T.t + dy * A.gx + dx;
            inbox_of(A, np, to)[atomicAdd(A.cnt_cur + np * kTilesMax + to, 1)] = c;
        };
        if (n > 0) place(a, p, d, false);
        const bool crowded = m + n_ovf > kTlOwn;
        if (crowded) {
            block_sync();                               // their last step is done: theirs is an extra barrier
            for (int i0 = kTlOwn + cw * 32; i0 < m + n_ovf; i0 += kTlOwn) {
                const int i = i0 + lane;
                int c = -1;
                float cp[2] = {0.f, 0.f}, cd[2] = {0.f, 0.f};
                if (i < m) {
                    c = T.l_id[lb * cap + i];
                    cp[0] = T.st(cap, lb, 0, i);
                    cp[1] = T.st(cap, lb, 1, i);
                    cd[0] = T.st(cap, lb, 2, i);
                    cd[1] = T.st(cap, lb, 3, i);
                } else if (i < m + n_ovf) {
                    c = __ldcg(ovf + i - m);
                    if (c >= 0) {
                        cp[0] = __ldcg(gp + c);
                        cp[1] = __ldcg(gp + n + c);
                        cd[0] = __ldcg(gd + c);
                        cd[1] = __ldcg(gd + n + c);
                    }
                }
                place(c, cp, cd, i >= m);
            }
        }
        const int nx = T.tx + lane % 3 - 1, ny = T.ty + lane / 3 - 1;
        const bool nb = lane < 9 && lane != 4 && nx >= 0 && nx < A.gx && ny >= 0 && ny < A.gy;
        if (n > 0) {
            if (extra) __threadfence();                 // before the number that tells of it goes out
            asm volatile("bar.sync 1, %0;" ::"r"(kTlOwn) : "memory");      // the cone warps have placed theirs
            if (cw == 0 && lane < 9) {
                const int c = s_out[lane];
                const bool used = ovf0 + n_ovf > 0;     // this round's list came from the inbox, in part
                if (c > kTlPost || used) __threadfence();
                if (nb) st_packet(post_box(A, par, ny * A.gx + nx, 8 - lane) + 3 * kTlPost, packet((unsigned)c | (used ? kTlInboxUsed : 0u), tag));
                s_out[lane] = 0;
            }
        }
        block_sync();                                   // the round's last barrier
        if (cw == kTlConeWarps - 1) {
            // ---- arrivals: the number from each neighbour, then its cones, spread over the lanes
            // (in the first round, also: the neighbours have loaded, so this block may write from here on)
            bool ok = TRAJ || rd > 0 || wait_neighbours(A, T.tx, T.ty, A.base);
            if (n > 0) {
                long long it = 0;
                int c = 0;
                if (nb) {
                    const void *q = post_box(A, par, T.t, lane) + 3 * kTlPost;
                    unsigned long long w = ld_packet(q);
                    while (!tagged(w, tag) && ok) {
                        ok = keep_waiting(it, A.limit, A.abort, A.base, A.status);
                        w = ld_packet(q);
                    }
                    c = ok ? (int)((unsigned)w & ~kTlInboxUsed) : 0;
                    if ((unsigned)w & kTlInboxUsed) __threadfence();
                }
                // cones in the inbox: from a neighbour that had more than it can post, or this tile's own
                const int stayed = *s_push;
                __syncwarp();
                if (lane == 0) *s_push = 0;             // for the next round
                int in_box = 0;
                if (__any_sync(kFull, c > kTlPost) || stayed > cap) {
                    __threadfence();
                    if (lane == 0) in_box = min(atomicExch(A.cnt_cur + np * kTilesMax + T.t, 0), n);
                    in_box = __shfl_sync(kFull, in_box, 0);
                }
                c = min(c, kTlPost);
                int upto = c;                           // posted cones from neighbours up to this lane's
#pragma unroll
                for (int o = 1; o < 16; o <<= 1) {
                    const int u = __shfl_up_sync(kFull, upto, o);
                    if (lane >= o) upto += u;
                }
                const int posted = __shfl_sync(kFull, upto, 8);
                const int m0 = min(stayed, cap), room = cap - m0;
                int *box = inbox_of(A, np, T.t);
                for (int i0 = 0; i0 < posted; i0 += 32) {
                    const int i = i0 + lane;
                    int dir = 0, before = 0;
#pragma unroll
                    for (int q = 0; q < 9; ++q) {
                        const int u = __shfl_sync(kFull, upto, q);
                        if (i >= u) {
                            dir = q + 1;
                            before = u;
                        }
                    }
                    if (i < posted) {
                        const ulonglong2 *e = post_box(A, par, T.t, dir) + 3 * (i - before);
                        unsigned long long w[6];
                        for (;;) {
                            ld_packets(e, w[0], w[1]);
                            ld_packets(e + 1, w[2], w[3]);
                            ld_packets(e + 2, w[4], w[5]);
                            if (tagged(w[0], tag) && tagged(w[1], tag) && tagged(w[2], tag) && tagged(w[3], tag) && tagged(w[4], tag)) break;
                            if (!ok || !(ok = keep_waiting(it, A.limit, A.abort, A.base, A.status))) break;
                        }
                        if (ok) {
                            const int q = (int)(unsigned)w[0];
                            const float cp[2] = {__uint_as_float((unsigned)w[1]), __uint_as_float((unsigned)w[2])};
                            const float cd[2] = {__uint_as_float((unsigned)w[3]), __uint_as_float((unsigned)w[4])};
                            if (i < room) {
                                T.l_id[nl * cap + m0 + i] = q;
                                T.st(cap, nl, 0, m0 + i) = cp[0];
                                T.st(cap, nl, 1, m0 + i) = cp[1];
                                T.st(cap, nl, 2, m0 + i) = cd[0];
                                T.st(cap, nl, 3, m0 + i) = cd[1];
                            } else {                    // no room left: to the inbox list, with its state in the arrays
                                if (!TRAJ) put_cone<false>(A, 0, q, cp, cd);
                                box[in_box + i - room] = q;
                            }
                        }
                    }
                }
                const int took = min(posted, room), take = min(in_box, room - took);
                for (int i = lane; i < take; i += 32) { // the inbox's first ones into what room there is
                    const int q = __ldcg(box + i), at = m0 + took + i;
                    T.l_id[nl * cap + at] = q;
                    T.st(cap, nl, 0, at) = __ldcg(gp + q);
                    T.st(cap, nl, 1, at) = __ldcg(gp + n + q);
                    T.st(cap, nl, 2, at) = __ldcg(gd + q);
                    T.st(cap, nl, 3, at) = __ldcg(gd + n + q);
                }
                if (lane == 0) {
                    s_list[0] = m0 + took + take;
                    s_list[1] = take;
                    s_list[2] = in_box + posted - took - take;
                }
            }
            if (!ok) *s_fail = 1;
            // every round's first step finds its ticket at zero: a crowded step clears the next step's only, so
            // its round leaves its last step's as it was
            if (lane < 2) s_ticket[lane] = 0;
        }
        block_sync();
        if (*s_fail) break;
        lb ^= 1;
    }
    if (bits) flag_status(A.status, bits);
    if (crowd > 0.0f && cw == 0 && lane == 0) atomicMax(A.crowd, (int)(crowd / (float)A.nsteps));
    return live;
}

// VEC: rows are multiples of 4 nodes and 16-byte aligned.
template <bool MAP, bool TRAJ, bool VEC>
__global__ void __launch_bounds__(kTlThreads, 1) tiles_kernel(const __grid_constant__ TileArgs A)
{
    constexpr int W = kTlW, W4 = W / 4;
    const FieldDesc &f = A.f;
    const int R = A.ay.W;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int n = A.n, cap = A.cap;
    constexpr int warps = kTlWarps, threads = kTlThreads;
    const bool field_warp = warp < kTlFieldWarps;
    const int fw = warp;                                // a field warp's number

    // ---- shared memory: two field buffers, the map, the sources, the cone lists
    extern __shared__ float4 tl_smem[];
    float *S = reinterpret_cast<float *>(tl_smem);
    float *M = S + 2 * (size_t)R * W;
    int *s_off = reinterpret_cast<int *>(M + (MAP ? (size_t)R * W : 0));   // node offset in the tile
    float *s_e = reinterpret_cast<float *>(s_off + A.n_src);
    float *s_xy = s_e + A.n_src;                                           // [2][n_src]
    __shared__ int s_scnt[kTlFieldWarps], s_ticket[2], s_push, s_list[3], s_fail, s_out[9];
    __shared__ float s_xi[4 * kTlHelped];              // [step parity][2][kTlHelped]

    Tile T;
    T.t = blockIdx.x;
    T.tx = T.t % A.gx;
    T.ty = T.t / A.gx;
    T.sx = A.ax.start(T.tx);
    T.ex = A.ax.end(T.tx);
    T.sy = A.ay.start(T.ty);
    T.ey = A.ay.end(T.ty);
    T.ox = max(0, min(T.sx - (T.tx > 0 ? A.ax.H : 0), f.nx - W));
    T.oy = max(0, min(T.sy - (T.ty > 0 ? A.ay.H : 0), f.ny - R));
    T.R = R;
    T.cx0 = T.ox > 0 ? T.ox + 1 : 0;
    T.cx1 = T.ox + W < f.nx ? T.ox + W - 3 : f.nx - 2;
    T.cy0 = T.oy > 0 ? T.oy + 1 : 0;
    T.cy1 = T.oy + R < f.ny ? T.oy + R - 3 : f.ny - 2;
    T.S = S;
    T.M = M;
    T.l_id = reinterpret_cast<int *>(s_xy + 2 * A.n_src);
    T.l_st = reinterpret_cast<float *>(T.l_id + 2 * cap);
    const int ox = T.ox, oy = T.oy;
    const float *gin = TRAJ ? A.traj_field : (A.cur0 ? A.field1 : A.field0);

    // ---- the tile (and its map) into shared memory
    for (int r = warp; r < R; r += warps) {
        const size_t g = (size_t)(oy + r) * f.nx + ox;
        if constexpr (VEC) {
            tl_smem[r * W4 + lane] = __ldcg(reinterpret_cast<const float4 *>(gin + g) + lane);
            if (MAP) reinterpret_cast<float4 *>(M)[r * W4 + lane] = __ldg(reinterpret_cast<const float4 *>(A.map + g) + lane);
        } else {
            for (int x = lane; x < W; x += 32) {
                S[r * W + x] = __ldcg(gin + g + x);
                if (MAP) M[r * W + x] = __ldg(A.map + g + x);
            }
        }
    }

    // ---- this warp's part of the sweep: rows [r0, r1)
    const int r0 = field_warp ? fw * R / kTlFieldWarps : 0, r1 = field_warp ? (fw + 1) * R / kTlFieldWarps : 0;

    // ---- the point sources of the loaded region, grouped by the warp that sweeps
    // them, each warp's in index order
    auto each_source = [&](const auto &fn) {          // fn(k, off) for this warp's sources, in order
        for (int b = 0; b < A.n_src; b += 32) {
            const int k = b + lane;
            int off = -1;
            if (k < A.n_src) {
                const int cell = __ldg(A.src_cell + k);
                if (cell >= 0 && (long long)cell < (long long)f.nx * f.ny) {
                    const int lx = cell % f.nx - ox, ly = cell / f.nx - oy;
                    if (lx >= 0 && lx < W && ly >= r0 && ly < r1) off = ly * W + lx;
                } else if (T.t == 0 && warp == 0) {
                    flag_status(A.status, kStatusBounds);
                }
            }
            fn(k, off);
        }
    };
    if (field_warp) {
        int c = 0;
        each_source([&](int, int off) { c += __popc(__ballot_sync(kFull, off >= 0)); });
        if (lane == 0) s_scnt[fw] = c;
    }
    if (tid == 0) {
        s_push = 0;
        s_fail = 0;
        s_ticket[0] = s_ticket[1] = 0;
    }
    if (tid < 9) s_out[tid] = 0;
    __syncthreads();
    int src_b = 0, src_e = 0, n_tile_src = 0;
    for (int w = 0; w < kTlFieldWarps; ++w) {
        if (w < fw) src_b += s_scnt[w];
        n_tile_src += s_scnt[w];
    }
    if (field_warp) {
        src_e = src_b;
        each_source([&](int k, int off) {
            const unsigned m = __ballot_sync(kFull, off >= 0);
            if (off >= 0) {
                const int at = src_e + __popc(m & ((1u << lane) - 1u));
                s_off[at] = off;
                s_e[at] = __ldg(A.src_emit + k);
                s_xy[at] = (float)(off % W + ox) * f.h;
                s_xy[A.n_src + at] = (float)(off / W + oy) * f.h;
            }
            src_e += __popc(m);
        });
    }
    const bool stop_on = A.c.stop_r2 >= 0.0f && A.n_src > 0;
    T.stop_xy = A.local_stop ? s_xy : A.src_xyz;
    T.n_stop = stop_on ? (A.local_stop ? n_tile_src : A.n_src) : 0;

    // ---- this tile's cones
    {
        const float *gp = cone_pos<TRAJ>(A, 0), *gd = cone_dir<TRAJ>(A, 0);
        for (int a = tid; a < n; a += threads) {
            const float px = __ldcg(gp + a), py = __ldcg(gp + n + a);
            const int ix = clampi((int)floorf(px * f.inv_h), 0, f.nx - 1), iy = clampi((int)floorf(py * f.inv_h), 0, f.ny - 1);
            if (ix < T.sx || ix >= T.ex || iy < T.sy || iy >= T.ey || !__ldcg(A.active + a)) continue;
            const int at = atomicAdd(&s_push, 1);
            if (at < cap) {
                T.l_id[at] = a;
                T.st(cap, 0, 0, at) = px;
                T.st(cap, 0, 1, at) = py;
                T.st(cap, 0, 2, at) = __ldcg(gd + a);
                T.st(cap, 0, 3, at) = __ldcg(gd + n + a);
            } else {
                inbox_of(A, 0, T.t)[at - cap] = a;
            }
        }
    }
    __syncthreads();
    const int nrounds = (A.nsteps + A.K - 1) / A.K;
    if (tid == 0) {
        if (!TRAJ) st_release_u32(A.flags + kTlFlagWords * T.t, A.base);   // the tile is loaded, its cones are found
        s_list[0] = min(s_push, cap);
        s_list[1] = 0;
        s_list[2] = s_push - min(s_push, cap);
        s_push = 0;
    }
    __syncthreads();

    unsigned live = 0;
    if (field_warp) {
        LaneMasks L{0, 0, 0, 0};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int x = ox + 4 * lane + q;
            const bool own = x >= T.sx && x < T.ex;
            const bool halo = x >= T.sx - A.ax.H && x < T.ex + A.ax.H;
            L.own |= own << q;
            L.edge |= (own && ((T.tx > 0 && x < T.sx + A.ax.H) || (T.tx + 1 < A.gx && x >= T.ex - A.ax.H))) << q;
            L.halo |= halo << q;
            L.halo_side |= (halo && !own) << q;
        }
        const WarpSources src{s_off, s_e, src_b, src_e};
        live = field_loop<MAP, TRAJ, VEC>(A, T, r0, r1, L, src, s_ticket, s_list, &s_fail);
    } else {
        live = cone_loop<TRAJ>(A, T, s_ticket, s_list, &s_fail, &s_push, s_out, s_xi);
    }

    const bool ran = !s_fail;                           // (written before the barrier that ended the loops)
    const int b = A.nsteps & 1;
    const float big = 3.402823466e38f;
    const float *c1 = S + (size_t)b * R * W, *c0 = S + (size_t)(b ^ 1) * R * W;
    bool bad = false;
    if constexpr (!TRAJ) {
        // ---- the end: C^{n+k} and C^{n+k-1} go out.  One of them overwrites the input: every
        // neighbour's flag says that it has loaded its tile (looked at in the first exchange, or here)
        if (nrounds == 1 && warp == 0) {
            const bool ok = wait_neighbours(A, T.tx, T.ty, A.base);
            if (lane == 0) s_push = ok ? 0 : -1;
        }
        __syncthreads();
        if (ran && !(nrounds == 1 && s_push < 0)) {
            const bool flip = (A.cur0 + A.nsteps) & 1;
            float *g1 = flip ? A.field1 : A.field0, *g0 = flip ? A.field0 : A.field1;
            for (int y = T.sy + warp; y < T.ey; y += warps) {
                const size_t g = (size_t)y * f.nx + ox;
                const int l = (y - oy) * W;
                if constexpr (VEC) {
                    const int x = ox + 4 * lane;
                    if (x >= T.sx && x < T.ex) {
                        const float4 v = reinterpret_cast<const float4 *>(c1 + l)[lane];
                        bad |= !(fabsf(v.x) <= big && fabsf(v.y) <= big && fabsf(v.z) <= big && fabsf(v.w) <= big);
                        reinterpret_cast<float4 *>(g1 + g)[lane] = v;
                        reinterpret_cast<float4 *>(g0 + g)[lane] = reinterpret_cast<const float4 *>(c0 + l)[lane];
                    }
                } else {
                    for (int x = T.sx - ox + lane; x < T.ex - ox; x += 32) {
                        bad |= !(fabsf(c1[l + x]) <= big);
                        g1[g + x] = c1[l + x];
                        g0[g + x] = c0[l + x];
                    }
                }
            }
        }
    } else if (ran) {
        for (int y = T.sy + warp; y < T.ey; y += warps)
            for (int x = T.sx - ox + lane; x < T.ex - ox; x += 32) bad |= !(fabsf(c1[(y - oy) * W + x]) <= big);
    }
    if (bad) flag_status(A.status, kStatusNonFinite);
    // the next launch's inbox counts start at zero whatever became of this one
    for (int i = blockIdx.x + (int)gridDim.x * tid; i < 2 * kTilesMax; i += (int)gridDim.x * threads) A.cnt_next[i] = 0;
    const unsigned tot = __reduce_add_sync(kFull, live);
    if (tot && lane == 0) atomicAdd(A.counter, (unsigned long long)tot);
}

int sm_count_t()
{
    static PerDevice count;
    return count.on_current([] {
        int dev = 0, n = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
        return n > 0 ? n : 152;
    });
}

constexpr size_t kTlSmemMax = 227u * 1024u - 3072u;     // a block's limit, less the kernel's static shared memory

size_t tiles_smem(const TilesGeom &g, bool map, int n_src)
{
    return sizeof(float) * (size_t)g.W * g.R * (map ? 3 : 2) + 16 * (size_t)n_src + 40 * (size_t)g.cap;
}

// Tile shape for K steps a round: the fewest rows of 128 columns that cover the grid with a tile per SM.
bool tiles_shape(int nx, int ny, bool cones, float step_len, float h, int K, int sms, TilesGeom &g)
{
    const double drift = cones ? std::ceil((K - 1) * (double)step_len / (double)h * (1.0 + 1e-5)) : 0.0;
    if (drift > 1024.0) return false;
    const int H = cones ? (int)(K + 1 + drift) : K;
    const int W = kTlW, HX = (H + 3) & ~3, most = std::min(sms, kTilesMax);
    if (nx < W || W < 3 * HX) return false;
    const AxisTiles ax{nx, W, HX, 0};
    const int gx = ax.count();
    if (gx > most) return false;
    const int rows = most / gx;
    int R = ny;
    if (rows >= 2) R = std::max((int)(((long long)ny + 2LL * H * (rows - 1) + rows - 1) / rows), 3 * H);
    if (R >= ny) R = ny;                                 // one tile row
    if (R > kTlFieldWarps * kTlMaxRows) return false;
    const AxisTiles ay{ny, R, H, 0};
    if ((long long)gx * ay.count() > most) return false;
    // a cone crosses at most into the next tile in a round
    const double reach = cones ? K * (double)step_len / (double)h * (1.0 + 1e-5) + 1.0 : 0.0;
    if ((gx > 1 && reach > ax.inner()) || (ay.count() > 1 && reach > ay.inner())) return false;
    g.W = W;
    g.R = R;
    g.HX = HX;
    g.HY = H;
    g.gx = gx;
    g.gy = ay.count();
    g.K = K;
    return true;
}

}  // namespace

bool tiles_possible(int nx, int ny, bool cones)
{
    TilesGeom g;
    for (int K = 1; K <= 16; ++K)                        // (a longer step's halo is the wider: it fits no grid that none of these do)
        if (tiles_shape(nx, ny, cones, 0.0f, 1.0f, K, kTilesMax, g)) return true;
    return false;
}

// The steps a round K: microseconds a step by what was measured on GB300 -- a field warp's rows
// (0.1 each; at least 0.75 with cones, their dependent chain), and an exchange shared by the K steps of a round
// (1.9, and 0.045 a node of halo width; 1.6 times that where rows are not whole float4 groups).
// 1024^2 with 4,096 spread cones: K = 3 to 12 took 1.73, 1.48, 1.43, 1.32, 1.35, 1.50, 1.50, 1.43, 1.32, 1.35 us a step,
// the rule picks 7; 1025 x 769: 2.20, 1.87, 1.71, 1.56, 1.51, 1.60, 1.55, 1.51, 1.63, 1.60, it picks 10; 512 x 384 with 2,000:
// 1.45, 1.24, 1.13, 1.04, 0.99, 0.96, 0.97, 0.93, 0.97, 0.98, it picks 12.
bool tiles_geometry(const FieldDesc &f, float step_len, bool map, bool vec, int n_src, int n_axons, int depth, int sms,
                    TilesGeom &best)
{
    if (f.dim != 2 || n_src > kTlMaxSrc) return false;
    const bool cones = n_axons > 0;
    double best_t = 0.0;
    bool found = false;
    for (int K = depth > 0 ? depth : 2; K <= (depth > 0 ? depth : 12); ++K) {
        TilesGeom g;
        if (!tiles_shape(f.nx, f.ny, cones, step_len, f.h, K, sms, g)) continue;
        // on average no more cones than half of what the cone warps hold (a quarter with a map, where the
        // work-list kernel shares any crowd out evenly and is the only other path)
        if (n_axons > (map ? kTlHelped / 2 : kTlHelped) * g.gx * g.gy) continue;
        g.cap = std::min((n_axons + 31) & ~31, 1024);
        if (tiles_smem(g, map, n_src) > kTlSmemMax) continue;
        const int rows = (g.R + kTlFieldWarps - 1) / kTlFieldWarps;
        const double edge = vec ? 1.0 : 1.6, sweep = std::max(0.11 + 0.1 * rows, cones ? 0.75 : 0.0);
        const double t = sweep + edge * (1.9 + 0.045 * (g.HX + g.HY)) / K;
        // (for AUTO's choice: tall tiles' exchanges take longer than that, 7.2 us at 168 rows, 12 where rows are not
        // whole float4 groups; and a launch, which loads the grid, finds the cones and writes two grids, 9 to 20 us, up to 33)
        const double nodes = (double)f.nx * f.ny;
        g.step_us = sweep;
        g.exchange_us = edge * (1.9 + 0.045 * (g.HX + g.HY) + 0.1 * std::max(0, g.R - 130)) + (map ? 1.0 : 0.0);
        g.start_us = vec ? (cones ? 9.5 + 3.4e-6 * nodes : 7.5 + 1.7e-6 * nodes) : cones ? 11.0 + 7.6e-6 * nodes : 10.0 + 5e-6 * nodes;
        if (!found || t < best_t) {
            best = g;
            best_t = t;
            found = true;
        }
    }
    return found;
}

// Flags, inbox counts (2 launches x 2 parities), the abort word; then the post boxes.
static size_t tiles_flags_bytes() { return (sizeof(unsigned) * ((kTlFlagWords + 4) * kTilesMax + 64) + 255) & ~(size_t)255; }
size_t tiles_ctl_bytes() { return tiles_flags_bytes() + sizeof(ulonglong2) * 2 * kTilesMax * 9 * (3 * kTlPost + 1); }

// The kernel's shared-memory allowance on the current device; false where it is refused (the grid then takes the
// path that the engine would have displaced).
template <bool MAP, bool TRAJ, bool VEC>
static bool tiles_allowed_t()
{
    static PerDevice allowed;
    return allowed.on_current([] {
        if (cudaFuncSetAttribute(tiles_kernel<MAP, TRAJ, VEC>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTlSmemMax) == cudaSuccess)
            return 1;
        cudaGetLastError();
        return 0;
    }) == 1;
}

template <bool TRAJ>
static bool tiles_allowed(const Sim &s)
{
    if (s.vec4) return s.src_map ? tiles_allowed_t<true, TRAJ, true>() : tiles_allowed_t<false, TRAJ, true>();
    return s.src_map ? tiles_allowed_t<true, TRAJ, false>() : tiles_allowed_t<false, TRAJ, false>();
}

template <bool MAP, bool TRAJ, bool VEC>
static cudaError_t tiles_launch_t(const TileArgs &A, int grid, size_t smem, cudaStream_t stream)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(kTlThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;         // all blocks co-resident: no wait can starve
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, tiles_kernel<MAP, TRAJ, VEC>, A);
}

template <bool TRAJ = false>
static bool tiles_ready(Sim &s, TilesGeom &g)
{
    // the work-list kernel's own options, its phantom arrivals and stream captures stay with it
    if (s.fd.dim != 2 || !s.wl.tiles_off || s.persist_rows || s.persist_bpsm || s.persist_phantom) return false;
    if (!s.tiles_geom_ready || s.tiles_geom_depth != s.temporal_depth) {
        s.tiles_geom_ok = tiles_geometry(s.fd, s.cd.step_len, s.src_map != nullptr, s.vec4, s.n_src, s.n_axons,
                                         s.temporal_depth, sm_count_t(), s.tiles_geom);
        s.tiles_geom_ready = true;
        s.tiles_geom_depth = s.temporal_depth;
    }
    if (!s.tiles_geom_ok || !tiles_allowed<TRAJ>(s)) return false;
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(s.stream, &cap) != cudaSuccess || cap != cudaStreamCaptureStatusNone) return false;
    g = s.tiles_geom;
    return true;
}

static int tiles_launch(Sim &s, const TilesGeom &g, int nsteps, uint32_t step0, float *traj_field, float *traj_cone)
{
    TileArgs A;
    A.f = s.fd;
    A.c = s.cd;
    A.ax = AxisTiles{s.fd.nx, g.W, g.HX, 0};
    A.ay = AxisTiles{s.fd.ny, g.R, g.HY, 0};
    A.gx = g.gx;
    A.gy = g.gy;
    A.K = g.K;
    A.nsteps = nsteps;
    A.cur0 = s.cur;
    A.step0 = step0;
    A.field0 = s.field[0];
    A.field1 = s.field[1];
    A.map = s.src_map;
    A.src_cell = s.src_cell;
    A.src_emit = s.src_emit;
    A.src_xyz = s.src_xyz();
    A.n_src = s.n_src;
    A.local_stop = 1;
    if (s.cd.stop_r2 >= 0.0f) {
        const double r = std::sqrt((double)s.cd.stop_r2);
        A.local_stop = std::ceil((g.K * (double)s.cd.step_len + r) / (double)s.fd.h * (1.0 + 1e-5)) + 1 <= g.HY;
    }
    A.pos = s.pos;
    A.dir = s.dir;
    A.active = s.active;
    A.n = s.n_axons;
    A.cap = g.cap;

    A.traj_field = traj_field;
    A.traj_cone = traj_cone;
    A.cells = (size_t)s.fd.nx * s.fd.ny;
    unsigned *ctl = reinterpret_cast<unsigned *>(s.ws + s.wl.tiles_off);
    A.flags = ctl;
    int *cnt = reinterpret_cast<int *>(ctl + kTlFlagWords * kTilesMax);
    A.cnt_cur = cnt + (s.tiles_launches & 1) * 2 * kTilesMax;
    A.cnt_next = cnt + ((s.tiles_launches + 1) & 1) * 2 * kTilesMax;
    A.abort = ctl + (kTlFlagWords + 4) * kTilesMax;
    A.crowd = reinterpret_cast<int *>(A.abort + 1);
    A.inbox = reinterpret_cast<int *>(s.ws + s.wl.tiles_inbox_off);
    A.post = reinterpret_cast<ulonglong2 *>(s.ws + s.wl.tiles_off + tiles_flags_bytes());
    A.packets = reinterpret_cast<unsigned long long *>(s.ws + s.wl.tiles_packets_off);
    A.base = s.tiles_base;
    A.limit = s.persist_limit > 0 ? s.persist_limit : kPersistSpinLimit;
    A.status = s.status();
    A.counter = s.cone_counter();
    const int grid = g.gx * g.gy;
    const size_t smem = tiles_smem(g, s.src_map != nullptr, s.n_src);
    cudaError_t e;
    if (traj_field)
        e = s.vec4 ? (A.map ? tiles_launch_t<true, true, true>(A, grid, smem, s.stream)
                            : tiles_launch_t<false, true, true>(A, grid, smem, s.stream))
                   : (A.map ? tiles_launch_t<true, true, false>(A, grid, smem, s.stream)
                            : tiles_launch_t<false, true, false>(A, grid, smem, s.stream));
    else
        e = s.vec4 ? (A.map ? tiles_launch_t<true, false, true>(A, grid, smem, s.stream)
                            : tiles_launch_t<false, false, true>(A, grid, smem, s.stream))
                   : (A.map ? tiles_launch_t<true, false, false>(A, grid, smem, s.stream)
                            : tiles_launch_t<false, false, false>(A, grid, smem, s.stream));
    if (e != cudaSuccess) return CUE_ERR_CUDA;
    s.tiles_base += (unsigned)((nsteps + g.K - 1) / g.K) + 1u;
    s.tiles_launches++;
    s.launches++;
    s.persist_grid = grid;
    return CUE_OK;
}

bool tiles_supported(Sim &s)
{
    TilesGeom g;
    return tiles_ready(s, g);
}

// The modelled time of a run against the other path's: short calls pay for the load of the grid and both buffers' way
// out, large grids for tall tiles and many exchanges, crowds for a tile whose cones its block steps alone (crowd_ns), where
// other paths share them out.  Of 420 measured runs (35 shapes from 129^2 to 1701^2, with and without cones and map, 1 to 256
// steps), the choice is the faster path or within 5% of it in 410, and 20% off at worst (129^2, 6 steps: 16 us, 14 as
// launches).  The crowd's part is read back from the last watched run without waiting, as the fused path's helpers are sized.
bool tiles_faster(Sim &s, int nsteps, double other_us)
{
    TilesGeom g;
    if (!tiles_ready(s, g)) return false;
    if (s.crowd_pending && cudaEventQuery(s.crowd_ev) == cudaSuccess) {
        s.crowd_pending = false;
        s.crowd_us = 1e-3 * *s.crowd_host;
    }
    const int rounds = (nsteps + g.K - 1) / g.K;
    // a depth that was asked for is a wish for the engine: only a crowd speaks against it
    const double plain = s.temporal_depth > 0 ? 0.0 : g.start_us + (s.crowd_us > 0.0 ? 2.5 : 0.0) + nsteps * g.step_us + (rounds - 1) * g.exchange_us;
    return plain + nsteps * s.crowd_us <= other_us;
}

// A crowd that makes the engine the slower one leaves the next 15 runs to the other path; then one run looks
// again, and while the crowd is still there the number left doubles (up to 960).  (One run: many may be queued before its
// readback comes.)
bool tiles_preferred(Sim &s, int nsteps, double other_us)
{
    if (tiles_faster(s, nsteps, other_us)) {
        if (!s.crowd_pending) {
            s.crowd_leave = kTilesCrowdLeave;
            s.crowd_left = -1;
        }
        return true;
    }
    if (s.crowd_us == 0.0) return false;
    if (s.crowd_left < 0) {
        s.crowd_left = s.crowd_leave;
        s.crowd_leave = std::min(2 * s.crowd_leave, 64 * kTilesCrowdLeave);
    }
    if (s.crowd_left-- > 0) return false;
    const double was = s.crowd_us;
    s.crowd_us = 0.0;
    const bool look = !s.crowd_pending && tiles_faster(s, nsteps, other_us);
    s.crowd_us = was;
    if (!look) s.crowd_left = 0;                         // not a run to look with: the next one does
    return look;
}

int run_tiles_if_supported(Sim &s, int nsteps)
{
    TilesGeom g;
    if (!tiles_ready(s, g)) return 1;
    if (nsteps <= 0) return CUE_OK;
    if (s.cd.stop_r2 >= 0.0f && s.n_src > 0 && !s.src_xyz_ready) {
        if (launch_src_xyz(s) != cudaSuccess) return CUE_ERR_CUDA;
        s.src_xyz_ready = true;
    }
    int *crowd = reinterpret_cast<int *>(s.ws + s.wl.tiles_off) + (kTlFlagWords + 4) * kTilesMax + 1;
    const bool watch = s.adapt_helpers && s.path == CUE_PATH_AUTO && s.n_axons > kTlOwn && !s.crowd_pending;
    if (watch && cudaMemsetAsync(crowd, 0, sizeof(int), s.stream) != cudaSuccess) return CUE_ERR_CUDA;
    for (int done = 0; done < nsteps;) {
        const int k = std::min(nsteps - done, kPersistMaxSteps);
        timing_begin(s);
        const int rc = tiles_launch(s, g, k, (uint32_t)s.cone_step, nullptr, nullptr);
        timing_end(s);
        if (rc != CUE_OK) return rc;
        s.cur ^= (k & 1);
        s.field_step += k;
        s.cone_step += k;
        done += k;
    }
    s.persist_used = true;
    if (watch) {
        if (!s.crowd_host && cudaHostAlloc(reinterpret_cast<void **>(&s.crowd_host), sizeof(int), cudaHostAllocDefault) != cudaSuccess)
            s.crowd_host = nullptr;
        if (s.crowd_host && !s.crowd_ev && cudaEventCreateWithFlags(&s.crowd_ev, cudaEventDisableTiming) != cudaSuccess)
            s.crowd_ev = nullptr;
        if (s.crowd_host && s.crowd_ev &&
            cudaMemcpyAsync(s.crowd_host, crowd, sizeof(int), cudaMemcpyDeviceToHost, s.stream) == cudaSuccess &&
            cudaEventRecord(s.crowd_ev, s.stream) == cudaSuccess)
            s.crowd_pending = true;
    }
    return CUE_OK;
}

int run_tiles_trajectory(Sim &s, float *traj_field, float *traj_cone, uint32_t step0, int nsteps)
{
    TilesGeom g;
    if (!tiles_ready<true>(s, g) || nsteps > kPersistMaxSteps) return 1;
    return tiles_launch(s, g, nsteps, step0, traj_field, traj_cone);
}

}  // namespace cue
