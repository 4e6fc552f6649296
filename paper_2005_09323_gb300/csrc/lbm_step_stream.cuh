// Two fused steps per pass over memory, for large ensembles (App. A streaming and
// collision, twice): a block walks down the rows of a channel, computes step t + 1
// of row y + 1 and, from it and the two rows before, step t + 2 of row y, so that
// a population value is read from HBM once and written once for two steps.  A
// single step moves 72 bytes per site (FP32) and
// is bound by HBM; here a site and step move 36 bytes.
//
// Thread = 4 consecutive sites, warp = 128 columns, block = a whole row, so the
// periodic seam needs no halo.  Each warp copies the nine source rows of its
// columns into its own shared memory two rows ahead (cp.async, 16 bytes a lane).
// Of the intermediate step a row's later rows need the populations that move up
// (2, 5, 6) for two rows, kept in the warp's shared memory, the level ones (0, 1,
// 3) for one row, kept in registers, and those that move down (4, 7, 8) at once;
// all in the storage format.  The one-site shift in x is a warp shuffle.  The
// values at the edges of a warp's columns go to its two neighbours through a
// ring of four rows in shared memory, with an mbarrier per warp and row: warps
// wait for their neighbours only, and no block barrier is in the row loop (with
// one, and the rows staged for the block, the warps stood at the barrier for a
// quarter of their time).  Every wait is bounded; on timeout a warp records the
// error and returns.
//
// A launch cuts the rows of all listed clones into one contiguous span per
// block; a span recomputes the intermediate step of one row beyond either end.
// Per site and step the arithmetic, the order of every sum and the storage
// rounding are the register-staged kernel's, so populations and drag partials
// are the same bits.
//
// 16 warps of 128 registers an SM: about 120 instructions per site and step, of
// which the packed BGK collision (lbm_pair.cuh) is 45; FP32 BGK then runs at 0.86
// of the measured copy bandwidth, the other formats are bound by issue slots and
// latency.  Fewer registers and more warps spill and lose (FP16: 178 GLUPS at 128
// registers, 171 at 102, 156 at 85).  Measured, single steps / streamed, GLUPS:
// FP32 BGK 64 x 1024 x 256 94.6 / 158, 256 x 512 x 128 94.4 / 147, 16 x 2048 x 512
// 93.3 / 160; FP32 central moments 93.6 / 123; FP16 BGK 163 / 184 (64 x 1024 x
// 256), 164 / 201 (16 x 2048 x 512); FP16 central moments 142 / 149.  Open channels
// of 513 x 129, 128 of them: FP32 central moments 70.6 / 83.9, FP32 BGK 75.6 / 79.9;
// FP16 central moments 58.0 / 83.9; the work on their columns is a quarter to a
// third of the streamed time.
#pragma once
#include "async_copy.cuh"
#include "lbm_step.cuh"

namespace lbm {

constexpr int kStreamV = 4;             // sites per thread
constexpr int kStreamMaxThreads = 512;  // rows of up to 2048 sites
constexpr int kStreamStages = 2;        // source rows in flight

// the rows a span [s, s1) of the linear row index (listed clone, y) loads: per
// clone the rows [ya, yb) it completes and one row beyond either end
struct StreamWalk {
    int s, s1, ny;
    int li, ya, yb;  // the current piece
    int y, ye;       // the row to load next, the piece's last
    __device__ bool piece()
    {
        if (s >= s1) return false;
        li = s / ny;
        ya = s - li * ny;
        yb = min(ny, ya + (s1 - s));
        y = max(ya - 1, 0);
        ye = min(yb, ny - 1);
        s += yb - ya;
        return true;
    }
    __device__ bool next() { return y++ < ye ? true : piece(); }
};

// the pulled values of direction Q at a thread's sites from the row's stored
// values v at the same sites and the value e beyond the warp's columns
template <int S, bool SCALED, int Q>
__device__ __forceinline__ void stream_pull(float2 (&g)[9][kStreamV / 2], const Vec<typename Codec<S>::T, kStreamV>& v,
                                            typename Codec<S>::T e, bool at_edge, float inv_scale)
{
    using K = Carry<S, SCALED>;
    constexpr int V = kStreamV;
    float d[V];
#pragma unroll
    for (int j = 0; j < V; j += 2) {
        const float2 f = K::in2(&v.e[j], wf(Q), inv_scale);
        d[j] = f.x;
        d[j + 1] = f.y;
    }
    if constexpr (cx(Q) == 1) {
        const float n = __shfl_up_sync(0xffffffffu, d[V - 1], 1);
#pragma unroll
        for (int j = V - 1; j > 0; --j) d[j] = d[j - 1];
        d[0] = at_edge ? K::in(e, wf(Q), inv_scale) : n;
    } else if constexpr (cx(Q) == -1) {
        const float n = __shfl_down_sync(0xffffffffu, d[0], 1);
#pragma unroll
        for (int j = 0; j < V - 1; ++j) d[j] = d[j + 1];
        d[V - 1] = at_edge ? K::in(e, wf(Q), inv_scale) : n;
    }
#pragma unroll
    for (int i = 0; i < V / 2; ++i) g[Q][i] = make_float2(d[2 * i], d[2 * i + 1]);
}

// the same without the shift (a wall returns the node's own population)
template <int S, bool SCALED, int Q>
__device__ __forceinline__ void stream_own(float2 (&g)[9][kStreamV / 2], const Vec<typename Codec<S>::T, kStreamV>& v,
                                           float inv_scale)
{
#pragma unroll
    for (int i = 0; i < kStreamV / 2; ++i) g[Q][i] = Carry<S, SCALED>::in2(&v.e[2 * i], wf(Q), inv_scale);
}

template <int S, bool SCALED>
__device__ __forceinline__ void stream_store(Vec<typename Codec<S>::T, kStreamV>& o, const float2 (&g)[kStreamV / 2],
                                             float w, float scale)
{
#pragma unroll
    for (int i = 0; i < kStreamV / 2; ++i) {
        if constexpr (S == kFP32) {
            const float2 f = add2(g[i], splat(w));
            o.e[2 * i] = f.x;
            o.e[2 * i + 1] = f.y;
        } else {
            Carry<S, SCALED>::out2(&o.e[2 * i], g[i].x, g[i].y, w, scale);
        }
    }
}

// the collision of a thread's sites, on pairs: BGK 161 against 150 GLUPS one site
// at a time, FP16 central moments 149 against 137 (16 x 2048 x 512).  FP32
// central moments in a periodic channel go one site at a time, since on pairs the
// constants and temporaries take registers the row loop does not have (96 bytes
// of spills, 126 against 127 GLUPS at 64 x 1024 x 256, 123 against 134 at 256 x 512 x
// 128).  An open channel's sites relax at their columns' rates om.
template <int S, int COLL, bool OPEN>
__device__ __forceinline__ void stream_collide(float2 (&g)[9][kStreamV / 2], const StepParams& p,
                                               const float2 (&om)[kStreamV / 2])
{
    if constexpr ((COLL == 0 || S != kFP32) && !OPEN) {
        collide2<COLL, kStreamV / 2>(g, p);
    } else if constexpr (OPEN) {
#pragma unroll
        for (int i = 0; i < kStreamV / 2; ++i) collide_at2<COLL>(g, i, p, om[i]);
    } else {
        float f[9][kStreamV];
#pragma unroll
        for (int q = 0; q < 9; ++q)
#pragma unroll
            for (int i = 0; i < kStreamV / 2; ++i) {
                f[q][2 * i] = g[q][i].x;
                f[q][2 * i + 1] = g[q][i].y;
            }
#pragma unroll
        for (int j = 0; j < kStreamV; ++j) collide<COLL, kStreamV>(f, j, p);
#pragma unroll
        for (int q = 0; q < 9; ++q)
#pragma unroll
            for (int i = 0; i < kStreamV / 2; ++i) g[q][i] = make_float2(f[q][2 * i], f[q][2 * i + 1]);
    }
}

// The sites whose two steps feel the obstacle: whole 4-site groups covering the
// columns, and the rows, within two sites of it.  The row stream computes them
// without the obstacle and does not store them; the blocks compute them apart,
// a chunk of rows at a time, before they stream.  (With the bounce-back inside
// the stream the blocks that met the obstacle's rows took twice as long as the
// others: one launch 593 us with and 223 us without an obstacle, 64 x 1024 x 256.)
//
// A group is the sites of one thread of the register-staged kernel whose drag
// partials these are: 4 for FP32, 8 for 16-bit storage.
template <int S>
constexpr int kStreamGroup = S == kFP32 ? 4 : 8;

// the rates of the columns x .. x + 3 of an open channel
__device__ __forceinline__ void stream_rates(const StepParams& p, int x, float2 (&om)[kStreamV / 2])
{
#pragma unroll
    for (int i = 0; i < kStreamV / 2; ++i)
        om[i] = make_float2(x + 2 * i < p.nx ? __ldg(p.om_col + x + 2 * i) : p.bgk.om,
                            x + 2 * i + 1 < p.nx ? __ldg(p.om_col + x + 2 * i + 1) : p.bgk.om);
}

template <int S>
struct StreamRegion {
    static constexpr int G = kStreamGroup<S>;
    int groups;        // groups of a row
    int g0, ng;        // first group (may be negative: the row is periodic) and their number
    int l0, nl;        // the same with one group more on either side, for the intermediate step
    int r0, r1;        // rows
    __host__ __device__ explicit StreamRegion(const StepParams& p)
    {
        groups = p.nx / G;
        g0 = (p.ox0 - 2 + G) / G - 1;  // ox0 >= 1: rounded down
        ng = (p.ox1 + 1) / G - g0 + 1;
        if (ng > groups) {
            g0 = 0;
            ng = groups;
        }
        l0 = g0 - 1;
        nl = ng + 2;
        if (nl > groups) {
            l0 = 0;
            nl = groups;
        }
        r0 = p.oy0 - 2 > 0 ? p.oy0 - 2 : 0;
        r1 = p.oy1 + 2 < p.ny ? p.oy1 + 2 : p.ny;
        if (p.ox1 <= p.ox0) ng = nl = r0 = r1 = 0;
    }
    __host__ __device__ int wrap(int g) const { return g < 0 ? g + groups : (g >= groups ? g - groups : g); }
    __host__ __device__ bool has(int g) const { return wrap(g - g0) < ng; }
    // shared memory for a chunk of rows: the intermediate step with one row more
    // on either side, and both steps' drag terms of each group
    __host__ __device__ size_t bytes(int rows) const
    {
        return (9 * (rows + 2) * G * sizeof(typename Codec<S>::T) + 2 * rows * sizeof(float)) * (size_t)nl;
    }
    // rows of a chunk: at most about one chunk per SM over all clones (the chunks
    // go to the first blocks, which are on different SMs; more chunks recompute
    // more rows: 110 against 105 us per step, 64 x 1024 x 256), at most one group
    // of the intermediate step per thread, at least 2 rows
    __host__ __device__ int chunk(int threads, size_t smem, int sms, int clones) const
    {
        const int per_clone = sms > clones ? sms / clones : 1;
        int r = threads / (nl > 0 ? nl * (G / kStreamV) : 1) - 2, even = (r1 - r0 + per_clone - 1) / per_clone;
        r = r > even ? even : r;
        r = r < 2 ? 2 : r;
        r = r > r1 - r0 ? r1 - r0 : r;
        while (r > 2 && bytes(r) > smem) --r;
        return r;
    }
};

// four sites x .. x + 3 of row y, from stored values at base[q qs + row rs
// + column]: row y is row yc there, site x column xc, the sites beyond them
// columns xl and xr.  Streaming with bounce-back, collision, rest state of solid
// sites; returns the group's momentum exchange with the obstacle so far: where
// two threads share a group, the odd lane continues the sum of the lane before.
// OPEN: also the bars of an open channel's grid and its inlet column (sites past
// the last column are left at rest; the outlet column is the caller's).
template <int S, bool SCALED, int COLL, bool OPEN, bool DRAG = true>
__device__ __forceinline__ float stream_site_group(const StepParams& p, float2 (&g)[9][kStreamV / 2], int x, int y,
                                                   const typename Codec<S>::T* base, int qs, int rs, int yc, int xc,
                                                   int xl, int xr)
{
    using T = typename Codec<S>::T;
    using K = Carry<S, SCALED>;
    constexpr int V = kStreamV;
    uint32_t cols = 0, bars = 0;  // bit i: site x - 1 + i is in the obstacle's, the grid's columns
#pragma unroll
    for (int i = 0; i < V + 2; ++i) {
        cols |= (x - 1 + i >= p.ox0 && x - 1 + i < p.ox1 ? 1u : 0u) << i;
        if (OPEN) bars |= (x - 1 + i >= p.gx0 && x - 1 + i < p.gx1 ? 1u : 0u) << i;
    }
    // (the sites beyond a periodic seam: columns 0 and nx - 1 are never solid)
    auto square_row = [&](int r) { return r >= p.oy0 && r < p.oy1 ? cols : 0u; };
    uint32_t solid[3];  // solid sites among x - 1 .. x + 4 of rows y - 1, y, y + 1
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const int r = y - 1 + d;
        solid[d] = square_row(r);
        if (OPEN && bars != 0u && r >= 0 && r < p.ny && r % p.gperiod >= p.ggap) solid[d] |= bars;
    }
    Vec<T, V> v[9];
    T e[9];
#pragma unroll
    for (int q = 0; q < 9; ++q) {
        const int ys = y - cy(q);
        const bool wall = ys < 0 || ys >= p.ny;  // the wall returns the node's own population
        const T* r = base + (wall ? opp(q) * qs + yc * rs : q * qs + (yc - cy(q)) * rs);
        v[q] = *reinterpret_cast<const Vec<T, V>*>(r + xc);
        if (cx(q) != 0) e[q] = r[wall ? (cx(q) == 1 ? xc : xc + V - 1) : (cx(q) == 1 ? xl : xr)];
    }
    float f[9][V];
#pragma unroll
    for (int q = 0; q < 9; ++q) {
        const bool wall = y - cy(q) < 0 || y - cy(q) >= p.ny;
        float d[V], n = 0.f;
#pragma unroll
        for (int j = 0; j < V; ++j) d[j] = K::in(v[q].e[j], wf(q), p.inv_scale);
        if (cx(q) != 0) n = K::in(e[q], wf(q), p.inv_scale);
#pragma unroll
        for (int j = 0; j < V; ++j) {
            if (cx(q) == 1)
                f[q][j] = wall ? d[j] : (j > 0 ? d[j > 0 ? j - 1 : 0] : n);
            else if (cx(q) == -1)
                f[q][j] = wall ? d[j] : (j + 1 < V ? d[j + 1 < V ? j + 1 : 0] : n);
            else
                f[q][j] = d[j];
        }
        const uint32_t back = q > 0 ? solid[1 - cy(q)] >> (1 - cx(q)) & ((1u << V) - 1u) : 0u;
        if (back != 0u) {
            const Vec<T, V> o = *reinterpret_cast<const Vec<T, V>*>(base + opp(q) * qs + yc * rs + xc);
#pragma unroll
            for (int j = 0; j < V; ++j)
                if (back >> j & 1u) f[q][j] = K::in(o.e[j], wf(q), p.inv_scale);
        }
#pragma unroll
        for (int i = 0; i < V / 2; ++i) g[q][i] = make_float2(f[q][2 * i], f[q][2 * i + 1]);
    }
    if constexpr (OPEN) {
        float2 om[V / 2];
        stream_rates(p, x, om);
        stream_collide<S, COLL, true>(g, p, om);
    } else {
        collide2<COLL, V / 2>(g, p);
    }
    auto sum = [&](float acc) {
#pragma unroll
        for (int j = 0; j < V; ++j) {
            const bool inside = square_row(y) >> (j + 1) & 1u;
#pragma unroll
            for (int q = 1; q < 9; ++q) {
                if (cx(q) == 0) continue;
                const float gq = j & 1 ? g[q][j / 2].y : g[q][j / 2].x;
                if (!inside && (square_row(y + cy(q)) >> (j + 1 + cx(q)) & 1u))
                    acc += 2.0f * (float)cx(q) * (wf(q) + gq);
            }
        }
        return acc;
    };
    float acc = DRAG ? sum(0.f) : 0.f;
    if constexpr (DRAG && kStreamGroup<S> > V) {
        const float before = __shfl_up_sync(0xffffffffu, acc, 1);
        if (threadIdx.x & 1) acc = sum(before);
    }
#pragma unroll
    for (int q = 0; q < 9; ++q)
#pragma unroll
        for (int j = 0; j < V; ++j)
            if (solid[1] >> (j + 1) & 1u || (OPEN && x + j >= p.nx))
                (j & 1 ? g[q][j / 2].y : g[q][j / 2].x) = 0.f;  // rest: f = w
    if (OPEN && x == 0)
#pragma unroll
        for (int q = 0; q < 9; ++q) g[q][0].x = __ldg(p.inlet_g + q * p.ny + y);
    return acc;
}

// the groups of rows [lo, hi) that are not wholly solid, numbered row by row:
// n groups a row, of which [sa, sa + sn) are solid in the obstacle's rows
struct StreamGroups {
    int lo, n, sa, sn, below, inside, total;
    __device__ StreamGroups(const StepParams& p, int lo_, int hi, int n_, int sa_, int sn_)
        : lo(lo_), n(n_), sa(sa_), sn(sn_)
    {
        const int b = min(max(p.oy0 - lo, 0), hi - lo), e = min(max(p.oy1 - lo, 0), hi - lo);
        below = b * n;
        inside = (e - b) * (n - sn);
        total = below + inside + (hi - lo - e) * n;
        rows_b = b;
        rows_e = e;
    }
    int rows_b, rows_e;
    __device__ void at(int i, int& y, int& g) const
    {
        if (i < below) {
            y = lo + i / n;
            g = i % n;
        } else if (i < below + inside) {
            i -= below;
            y = lo + rows_b + i / (n - sn);
            g = i % (n - sn);
            if (g >= sa) g += sn;
        } else {
            i -= below + inside;
            y = lo + rows_e + i / n;
            g = i % n;
        }
    }
};

// both steps of the obstacle's region for every listed clone, in chunks of R
// rows over the blocks, and the drag partials of its rows
template <int S, bool SCALED, int COLL, bool OPEN>
__device__ __noinline__ void stream_obstacle(const StepParams& p, unsigned char* smem, int R)
{
    using T = typename Codec<S>::T;
    constexpr int V = kStreamV, G = kStreamGroup<S>, H = G / V;  // H threads per group
    const StreamRegion<S> rg(p);
    const int nx = p.nx, ny = p.ny, plane = (int)p.plane, tid = threadIdx.x;
    const int chunks = (rg.r1 - rg.r0 + R - 1) / R, tw = rg.nl * G;
    T* const tile = reinterpret_cast<T*>(smem);  // [q][row][tw]
    const int tq = (R + 2) * tw;
    float* const terms = reinterpret_cast<float*>(smem + (size_t)9 * tq * sizeof(T));  // [step][row][nl]
    // whole groups of solid sites: at rest, never read
    const int sg = (p.ox0 + G - 1) / G, sn = max(p.ox1 / G - sg, 0);
    for (int item = blockIdx.x; item < p.n_list * chunks; item += gridDim.x) {
        const int c = p.clone_list[item / chunks];
        const int cur = p.parity[c] ^ p.flip;
        const T* src = static_cast<const T*>(cur ? p.buf1 : p.buf0) + (int64_t)c * p.clone_stride;
        T* dst = static_cast<T*>(cur ? p.buf0 : p.buf1) + (int64_t)c * p.clone_stride;
        const int ra = rg.r0 + item % chunks * R, rb = min(ra + R, rg.r1);
        const int la = max(ra - 1, 0), lb = min(rb + 1, ny);
        const StreamGroups first(p, la, lb, rg.nl, sg - rg.l0, sn), second(p, ra, rb, rg.ng, sg - rg.g0, sn);
        // (whole warps stay in the loops: the drag sums use shuffles)
        for (int i = tid; (i & ~31) < first.total * H; i += blockDim.x) {
            int y, gi;
            first.at(min(i / H, first.total - 1), y, gi);
            const bool in = i < first.total * H;
            const int h = i % H * V, x = rg.wrap(rg.l0 + gi) * G + h;
            float2 g[9][V / 2];
            const float acc = stream_site_group<S, SCALED, COLL, OPEN>(
                p, g, x, y, src, plane, p.pitch, y, x, x == 0 ? nx - 1 : x - 1,
                OPEN ? min(x + V, nx - 1) : (x + V == nx ? 0 : x + V));
            if (in) {
#pragma unroll
                for (int q = 0; q < 9; ++q) {
                    Vec<T, V> o;
                    stream_store<S, SCALED>(o, g[q], wf(q), p.scale);
                    *reinterpret_cast<Vec<T, V>*>(tile + q * tq + (y - la) * tw + gi * G + h) = o;
                }
                if (h + V == G && y >= ra && y < rb) terms[(y - ra) * rg.nl + gi] = acc;
            }
        }
        __syncthreads();
        for (int i = tid; (i & ~31) < second.total * H; i += blockDim.x) {
            int y, gg;
            second.at(min(i / H, second.total - 1), y, gg);
            gg += rg.g0;
            const bool in = i < second.total * H;
            const int gi = rg.wrap(gg - rg.l0), h = i % H * V, x = rg.wrap(gg) * G + h, lx = gi * G + h;
            float2 g[9][V / 2];
            // (beyond the tile's columns only where it is the whole row)
            const float acc = stream_site_group<S, SCALED, COLL, OPEN>(
                p, g, x, y, tile, tq, tw, y - la, lx, lx == 0 ? tw - 1 : lx - 1, lx + V == tw ? 0 : lx + V);
            if (in) {
#pragma unroll
                for (int q = 0; q < 9; ++q) {
                    Vec<T, V> o;
                    stream_store<S, SCALED>(o, g[q], wf(q), p.scale);
                    st_stream<T, V>(dst + q * plane + y * p.pitch + x, o);
                }
                if (h + V == G) terms[(R + y - ra) * rg.nl + gi] = acc;
            }
        }
        const int sa = max(ra, p.oy0), sb = min(rb, p.oy1);
        const int sv = sn * (G / V);
        for (int i = tid; i < max(sb - sa, 0) * sv; i += blockDim.x)
#pragma unroll
            for (int q = 0; q < 9; ++q) {
                Vec<T, V> o;
                const float2 rest[V / 2] = {};
                stream_store<S, SCALED>(o, rest, wf(q), p.scale);
                st_stream<T, V>(dst + q * plane + (sa + i / sv) * p.pitch + sg * G + i % sv * V, o);
            }
        __syncthreads();
        // the partial of a ring row and segment of 32 groups: the register-staged
        // kernel's warp sum
        const int ya = max(ra, p.ry0), yb = min(rb, p.ry1 + 1), nseg = p.rs1 - p.rs0 + 1;
        for (int i = tid >> 5; i < 2 * max(yb - ya, 0) * nseg; i += blockDim.x >> 5) {
            const int step = i & 1, y = ya + (i >> 1) / nseg, seg = p.rs0 + (i >> 1) % nseg;
            const int g = seg * 32 + (tid & 31), gi = rg.wrap(g - rg.l0);
            const bool solid = y >= p.oy0 && y < p.oy1 && g >= sg && g < sg + sn;
            float acc = g < rg.groups && rg.has(g) && !solid ? terms[(step * R + y - ra) * rg.nl + gi] : 0.f;
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
            if ((tid & 31) == 0)
                p.partials[((int64_t)c * p.batch_cap + p.step_in_batch + step) * p.n_slots + (y - p.ry0) * nseg + seg -
                           p.rs0] = acc;
        }
        __syncthreads();
    }
}

// Open channels (Sec. 2).  The stream itself takes 40 us per step and 64 x 513 x
// 129 nodes in FP32 (31 in FP16), the columns below, 8 % of the sites, another 17
// (21): about 1700 instructions for four sites and a step with all their cases.
// Bars and inlet inside the stream instead, in the warp that holds them, made
// every row wait for that warp (67 and 54 us in all, against 58 and 52).
//
// Columns of an open channel whose two steps the row stream does not know, in
// groups as above, over all rows: around the inlet column (range 0), the grid of
// bars (1), and columns nx - 3 .. nx - 1 before and at the outlet (2; it pulls
// from an outlet column that the velocities of three rows give).
template <int S>
struct StreamColumns {
    static constexpr int G = kStreamGroup<S>;
    int g0[3], g1[3], total;  // [g0, g1); groups of a row
    __host__ __device__ explicit StreamColumns(const StepParams& p)
    {
        total = (p.nx - 1) / G + 1;
        g0[0] = 0;
        g1[0] = 1;
        g0[1] = g1[1] = 0;
        if (p.gx1 > p.gx0) {
            g0[1] = p.gx0 >= 2 ? (p.gx0 - 2) / G : 0;
            g1[1] = (p.gx1 + 1) / G + 1;
            if (g0[1] == 0) g1[0] = 0;  // the grid's range holds the inlet's
        }
        g0[2] = (p.nx - 3) / G;
        g1[2] = total;
    }
    __host__ __device__ bool has(int g) const
    {
        return (g >= g0[0] && g < g1[0]) || (g >= g0[1] && g < g1[1]) || g >= g0[2];
    }
    __host__ __device__ static int halo(int r) { return r == 2 ? 3 : 1; }
    // groups of the intermediate step: one more on either side
    __host__ __device__ int l0(int r) const { return g0[r] > 0 ? g0[r] - 1 : 0; }
    __host__ __device__ int l1(int r) const { return g1[r] < total ? g1[r] + 1 : total; }
    __host__ __device__ size_t bytes(int r, int rows) const
    {
        return (size_t)9 * (rows + 2 * halo(r)) * (l1(r) - l0(r)) * G * sizeof(typename Codec<S>::T) +
               (r == 2 ? 4 * sizeof(float) * (rows + 2) : 0);
    }
    // rows of a chunk: two passes of the block over the intermediate step's
    // groups, or what the shared memory holds; 0: not even one row
    __host__ __device__ int chunk(int r, int threads, size_t smem, int ny) const
    {
        int n = 2 * threads / ((l1(r) - l0(r)) * (G / kStreamV)) - 2 * halo(r);
        n = n < 1 ? 1 : (n > ny ? ny : n);
        while (n > 0 && bytes(r, n) > smem) --n;
        return n;
    }
    // the obstacle's region must keep to its own groups, and the ranges be apart
    __host__ __device__ bool apart(const StreamRegion<S>& rg) const
    {
        if (g1[1] > g0[2] || g1[0] > g0[2]) return false;
        if (rg.ng == 0) return true;
        const int a = rg.g0, b = rg.g0 + rg.ng;
        return a >= 1 && a >= g1[0] && b <= g0[2] && (g1[1] == g0[1] || b <= g0[1] || a >= g1[1]) &&
               rg.nl < rg.groups;
    }
};

// both steps of rows [ra, rb) of column range r for listed clone li
template <int S, bool SCALED, int COLL>
__device__ __noinline__ void stream_columns(const StepParams& p, unsigned char* smem, int li, int r, int ra, int rb)
{
    using T = typename Codec<S>::T;
    using K = Carry<S, SCALED>;
    constexpr int V = kStreamV, G = kStreamGroup<S>, H = G / V;
    const StreamColumns<S> cols(p);
    const int nx = p.nx, ny = p.ny, plane = (int)p.plane, tid = threadIdx.x;
    const bool outlet = r == 2;
    const int c = p.clone_list[li], cur = p.parity[c] ^ p.flip;
    const T* src = static_cast<const T*>(cur ? p.buf1 : p.buf0) + (int64_t)c * p.clone_stride;
    T* dst = static_cast<T*>(cur ? p.buf0 : p.buf1) + (int64_t)c * p.clone_stride;
    const int hh = cols.halo(r), la = max(ra - hh, 0), lb = min(rb + hh, ny);
    const int xa = cols.l0(r) * G, tw = (cols.l1(r) - cols.l0(r)) * G, tq = (lb - la) * tw;
    T* const tile = reinterpret_cast<T*>(smem);                                   // [q][row][tw], column xa first
    float* const uv = reinterpret_cast<float*>(smem + (size_t)9 * tq * sizeof(T));  // [4][rows + 2]: as p.open_u
    const int n1 = (lb - la) * (tw / V);
    for (int i = tid; (i & ~31) < n1; i += blockDim.x) {
        const int k = min(i, n1 - 1), y = la + k / (tw / V), x = xa + k % (tw / V) * V;
        float2 g[9][V / 2];
        stream_site_group<S, SCALED, COLL, true, false>(p, g, x, y, src, plane, p.pitch, y, x, max(x - 1, 0),
                                                 min(x + V, nx - 1));
        if (i < n1)
#pragma unroll
            for (int q = 0; q < 9; ++q) {
                Vec<T, V> o;
                stream_store<S, SCALED>(o, g[q], wf(q), p.scale);
                *reinterpret_cast<Vec<T, V>*>(tile + q * tq + (y - la) * tw + x - xa) = o;
            }
    }
    __syncthreads();
    // velocity of a stored node of the tile, as the step kernel leaves it in p.open_u
    auto velocity = [&](int x, int y, float& u, float& v) {
        float h[9];
#pragma unroll
        for (int q = 0; q < 9; ++q) h[q] = K::in(tile[q * tq + (y - la) * tw + x - xa], wf(q), p.inv_scale);
        open_velocity9(h, u, v);
    };
    if (outlet) {  // the outlet column of the intermediate step
        const int oa = max(ra - 2, 0), ob = min(rb + 2, ny);
        for (int y = oa + tid; y < ob; y += blockDim.x) {
            const int ym = max(y - 1, 0), yp = min(y + 1, ny - 1);
            OutletU a;
            velocity(nx - 2, y, a.u2, a.v2);
            velocity(nx - 3, y, a.u3, a.v3);
            velocity(nx - 2, ym, a.u2m, a.v2m);
            velocity(nx - 3, ym, a.u3m, a.v3m);
            velocity(nx - 2, yp, a.u2p, a.v2p);
            velocity(nx - 3, yp, a.u3p, a.v3p);
            a.two = yp - ym == 2;
#pragma unroll
            for (int q = 0; q < 9; ++q)
                tile[q * tq + (y - la) * tw + nx - 1 - xa] =
                    K::out(outlet_g(a, (float)cx(q), (float)cy(q), wf(q), p.bc_pre), wf(q), p.scale);
        }
        __syncthreads();
    }
    // ---- second step; for the outlet also of the rows next to the chunk
    const int pa = outlet ? max(ra - 1, 0) : ra, pb = outlet ? min(rb + 1, ny) : rb, un = pb - pa;
    const int gw = (cols.g1[r] - cols.g0[r]) * H, n2 = un * gw;
    // the register-staged kernel's last vector leaves the row's padding at rest
    const bool pads = (nx - 1) % (32 * G) != 0;
    for (int i = tid; (i & ~31) < n2; i += blockDim.x) {
        const int k = min(i, n2 - 1), y = pa + k / gw, x = cols.g0[r] * G + k % gw * V, lx = x - xa;
        float2 g[9][V / 2];
        stream_site_group<S, SCALED, COLL, true, false>(p, g, x, y, tile, tq, tw, y - la, lx, max(lx - 1, 0),
                                                 min(lx + V, tw - 1));
        if (i >= n2) continue;
        if (outlet)
#pragma unroll
            for (int j = 0; j < V; ++j)
                if (x + j == nx - 2 || x + j == nx - 3) {
                    float h[9], u, v;
#pragma unroll
                    for (int q = 0; q < 9; ++q)
                        h[q] = K::in(K::out(j & 1 ? g[q][j / 2].y : g[q][j / 2].x, wf(q), p.scale), wf(q), p.inv_scale);
                    open_velocity9(h, u, v);
                    float* o = uv + (x + j == nx - 2 ? 0 : 2) * un + y - pa;
                    o[0] = u;
                    o[un] = v;
                }
        if (y < ra || y >= rb) continue;
#pragma unroll
        for (int q = 0; q < 9; ++q) {
            Vec<T, V> o;
            stream_store<S, SCALED>(o, g[q], wf(q), p.scale);
            T* to = dst + q * plane + y * p.pitch + x;
            if (x + V < nx) {
                st_stream<T, V>(to, o);
            } else {
#pragma unroll
                for (int j = 0; j < V; ++j)
                    if (x + j < nx - 1 || (x + j >= nx && pads)) to[j] = o.e[j];
            }
        }
    }
    __syncthreads();
    if (outlet)
        for (int y = ra + tid; y < rb; y += blockDim.x) {
            const int k = y - pa, km = max(y - 1, 0) - pa, kp = min(y + 1, ny - 1) - pa;
            OutletU a;
            a.u2 = uv[k];
            a.v2 = uv[un + k];
            a.u3 = uv[2 * un + k];
            a.v3 = uv[3 * un + k];
            a.u2m = uv[km];
            a.v2m = uv[un + km];
            a.u3m = uv[2 * un + km];
            a.v3m = uv[3 * un + km];
            a.u2p = uv[kp];
            a.v2p = uv[un + kp];
            a.u3p = uv[2 * un + kp];
            a.v3p = uv[3 * un + kp];
            a.two = kp - km == 2;
#pragma unroll
            for (int q = 0; q < 9; ++q)
                dst[q * plane + y * p.pitch + nx - 1] =
                    K::out(outlet_g(a, (float)cx(q), (float)cy(q), wf(q), p.bc_pre), wf(q), p.scale);
        }
    __syncthreads();
}

// keeps the compiler from holding the nine plane offsets of the loads and of
// the stores in registers across the row loop (they cost one instruction each)
__device__ __forceinline__ int stream_opaque(int v)
{
    asm volatile("" : "+r"(v));
    return v;
}

// 16 or 4 bytes global -> shared, asynchronously (cp.async)
__device__ __forceinline__ void stream_copy16(void* to, const void* from)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(smem_addr(to)), "l"(from) : "memory");
}
__device__ __forceinline__ void stream_copy8(void* to, const void* from)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(smem_addr(to)), "l"(from) : "memory");
}
__device__ __forceinline__ void stream_copy4(void* to, const void* from)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(smem_addr(to)), "l"(from) : "memory");
}

// shared memory of one warp: the staged source rows of its columns, the values
// beyond its columns, and the populations that move up, for two rows
template <int S>
struct StreamWarpSmem {
    using VT = Vec<typename Codec<S>::T, kStreamV>;
    VT row[kStreamStages][9][32];
    uint32_t beyond[kStreamStages][8];  // 4 bytes that hold the value left (1, 5, 8) or right (3, 6, 7) of the columns
    VT up[2][3][32];  // directions 2, 5, 6 of the intermediate step, by row mod 2
};

template <int S, bool SCALED, int COLL, bool OPEN>
__global__ void __launch_bounds__(kStreamMaxThreads, 1) step_stream_kernel(const __grid_constant__ StepParams p)
{
    using T = typename Codec<S>::T;
    constexpr int V = kStreamV;
    using VT = Vec<T, V>;
    extern __shared__ __align__(128) unsigned char smem[];
    // edge values of the last rows' intermediate step: per row (mod 4) and warp,
    // directions 3, 6, 7 at the warp's first site and 1, 5, 8 at its last; a
    // warp arrives on edge_ready when a row's values are in place
    __shared__ T edge[4][6][kStreamMaxThreads / 32];
    __shared__ __align__(8) uint64_t edge_ready[4][kStreamMaxThreads / 32];

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarp = blockDim.x >> 5;
    StreamWarpSmem<S>& ws = reinterpret_cast<StreamWarpSmem<S>*>(smem)[warp];
    const int nx = p.nx, ny = p.ny;
    const StreamRegion<S> rg(p);
    // an even share of the rows; a chunk of the obstacle's region takes a block
    // about as long as two of its rows
    const int rows = p.n_list * ny, grid = gridDim.x, bytes = nwarp * (int)sizeof(StreamWarpSmem<S>);
    const int chunk = rg.ng > 0 ? rg.chunk(blockDim.x, bytes, grid / (kStreamMaxThreads / blockDim.x), p.n_list) : 1;
    const int squares = p.n_list * ((rg.r1 - rg.r0 + chunk - 1) / chunk);
    int items = squares, range_rows[3] = {1, 1, 1}, range_chunks[3] = {0, 0, 0};
    if constexpr (OPEN) {
        const StreamColumns<S> cols(p);
        for (int r = 0; r < 3; ++r)
            if (cols.g1[r] > cols.g0[r]) {
                range_rows[r] = cols.chunk(r, blockDim.x, bytes, ny);
                range_chunks[r] = (ny + range_rows[r] - 1) / range_rows[r];
                items += p.n_list * range_chunks[r];
            }
    }
    const int cost = rows >= 8 * grid ? 2 : 0;
    auto span = [&](int b) {
        return (int)((rows + (int64_t)cost * items) * b / grid) - cost * (items / grid * b + min(b, items % grid));
    };
    const int s0 = span(blockIdx.x), s1 = span(blockIdx.x + 1);
    const int x0 = tid * V;
    // an open channel's columns from nx - 1 on are not streamed (its rows' padding
    // is read and feeds only sites computed apart)
    const bool active = OPEN ? x0 < nx - 1 : x0 < nx;
    const int xr = OPEN || active ? x0 : nx - V;
    const bool first = lane == 0, last = lane == 31 || (!OPEN && x0 + V >= nx);  // at the edges of the warp's columns
    const int wl = warp == 0 ? nwarp - 1 : warp - 1, wr = warp + 1 == nwarp ? 0 : warp + 1;
    const bool apart = rg.ng > 0 && rg.has(x0 / kStreamGroup<S>);  // in the obstacle's columns: computed by stream_obstacle
    const bool streamed = active && !(OPEN && StreamColumns<S>(p).has(x0 / kStreamGroup<S>));
    auto collide_row = [&](float2 (&g)[9][V / 2]) {
        float2 om[V / 2] = {};
        if constexpr (OPEN) {
            const float4 o = __ldg(reinterpret_cast<const float4*>(p.om_col + x0));  // padded to the row pitch
            om[0] = make_float2(o.x, o.y);
            om[1] = make_float2(o.z, o.w);
        }
        stream_collide<S, COLL, OPEN>(g, p, om);
    };

    if (tid < 4 * nwarp) mbar_init(smem_addr(&edge_ready[tid & 3][tid >> 2]), 1);
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    __syncthreads();
    if (rg.ng > 0) stream_obstacle<S, SCALED, COLL, OPEN>(p, smem, chunk);
    if constexpr (OPEN) {
        for (int i = blockIdx.x; i < items; i += grid) {  // after the obstacle's chunks, the column ranges'
            int k = i - squares, r = 0;
            if (k < 0) continue;
            while (k >= p.n_list * range_chunks[r]) k -= p.n_list * range_chunks[r++];
            const int ra = k % range_chunks[r] * range_rows[r];
            stream_columns<S, SCALED, COLL>(p, smem, k / range_chunks[r], r, ra, min(ra + range_rows[r], ny));
        }
    }

    StreamWalk w{s0, s1, ny};
    if (!w.piece()) return;
    StreamWalk pw = w;  // position of the next row to load
    bool more = true;
    auto source = [&](int li) {  // the state the launch reads, of the listed clone li
        const int c = p.clone_list[li];
        return static_cast<const T*>((p.parity[c] ^ p.flip) ? p.buf1 : p.buf0) + (int64_t)c * p.clone_stride;
    };
    const T* from_clone = source(w.li);
    // lanes 0..5: the direction whose value beyond the warp's columns the lane
    // fetches, and that value's column (16-bit: the 4 bytes that hold it)
    const int eq = lane == 0 ? 1 : lane == 1 ? 5 : lane == 2 ? 8 : lane == 3 ? 3 : lane == 4 ? 6 : 7;
    const int xw = warp * 32 * V;
    auto edge_col = [&](bool left) {
        if (OPEN) return left ? max(xw - 1, 0) : min(xw + 32 * V, nx - 1);
        return left ? (xw == 0 ? nx - 1 : xw - 1) : (xw + 32 * V >= nx ? 0 : xw + 32 * V);
    };
    const int xe = edge_col(lane < 3);
    auto load_row = [&](int stage) {
        if (more) {
            const T* src = from_clone;
            const int plane = stream_opaque((int)p.plane);
#pragma unroll
            for (int q = 0; q < 9; ++q) {
                // the wall returns the population that left this node
                const bool wall = cy(q) != 0 && (cy(q) == 1 ? pw.y == 0 : pw.y == ny - 1);
                const T* from = src + (wall ? opp(q) * plane + pw.y * p.pitch : q * plane + (pw.y - cy(q)) * p.pitch) + xr;
                if constexpr (sizeof(VT) == 16)
                    stream_copy16(&ws.row[stage][q][lane], from);
                else
                    stream_copy8(&ws.row[stage][q][lane], from);
            }
            if (lane < 6) {  // at a wall the pull has no shift and the value is not used
                const int ey = eq == 5 || eq == 6 ? 1 : (eq == 7 || eq == 8 ? -1 : 0);
                const int sy = min(max(pw.y - ey, 0), ny - 1);
                const T* from = src + eq * plane + sy * p.pitch + xe;
                stream_copy4(&ws.beyond[stage][lane], reinterpret_cast<const void*>(reinterpret_cast<uintptr_t>(from) & ~uintptr_t(3)));
            }
            const int li = pw.li;
            more = pw.next();
            if (more && pw.li != li) from_clone = source(pw.li);
        }
        asm volatile("cp.async.commit_group;\n" ::: "memory");
    };
    for (int i = 0; i < kStreamStages; ++i) load_row(i);
    auto beyond = [&](int stage, int i) {
        const int off = sizeof(T) == 2 ? edge_col(i < 3) & 1 : 0;
        return reinterpret_cast<const T*>(&ws.beyond[stage][i])[off];
    };

    int stage = 0;
    uint32_t k = 0;  // rows so far: ring position k mod 4, pass k / 4
    VT B0{}, B1{}, B3{};
    do {
        const int c = p.clone_list[w.li];
        const int cur = p.parity[c] ^ p.flip;
        T* dst = static_cast<T*>(cur ? p.buf0 : p.buf1) + (int64_t)c * p.clone_stride;
        for (int y1 = w.y; y1 <= w.yb; ++y1, ++k) {
            VT C0, C1, C2, C3, C4, C5, C6, C7, C8;
            const int slot = k & 3;
            const bool real = y1 < ny;  // beyond the last row only its second step remains
            if (real) {
                // ---- first step of row y1
                asm volatile("cp.async.wait_group %0;\n" ::"n"(kStreamStages - 1) : "memory");
                __syncwarp();
                float2 g[9][V / 2];
                const auto& r = ws.row[stage];
                T e1{}, e5{}, e8{}, e3{}, e6{}, e7{};
                if (first) {
                    e1 = beyond(stage, 0);
                    e5 = beyond(stage, 1);
                    e8 = beyond(stage, 2);
                }
                if (last) {
                    e3 = beyond(stage, 3);
                    e6 = beyond(stage, 4);
                    e7 = beyond(stage, 5);
                }
                stream_pull<S, SCALED, 0>(g, r[0][lane], T(), false, p.inv_scale);
                stream_pull<S, SCALED, 2>(g, r[2][lane], T(), false, p.inv_scale);
                stream_pull<S, SCALED, 4>(g, r[4][lane], T(), false, p.inv_scale);
                stream_pull<S, SCALED, 1>(g, r[1][lane], e1, first, p.inv_scale);
                stream_pull<S, SCALED, 5>(g, r[5][lane], e5, first, p.inv_scale);
                stream_pull<S, SCALED, 8>(g, r[8][lane], e8, first, p.inv_scale);
                stream_pull<S, SCALED, 3>(g, r[3][lane], e3, last, p.inv_scale);
                stream_pull<S, SCALED, 6>(g, r[6][lane], e6, last, p.inv_scale);
                stream_pull<S, SCALED, 7>(g, r[7][lane], e7, last, p.inv_scale);
                if (y1 == 0) {  // walls: the node's own populations come back, unshifted
                    stream_own<S, SCALED, 5>(g, r[5][lane], p.inv_scale);
                    stream_own<S, SCALED, 6>(g, r[6][lane], p.inv_scale);
                }
                if (y1 == ny - 1) {
                    stream_own<S, SCALED, 7>(g, r[7][lane], p.inv_scale);
                    stream_own<S, SCALED, 8>(g, r[8][lane], p.inv_scale);
                }
                __syncwarp();
                load_row(stage);  // every lane has read the stage
                stage = stage + 1 == kStreamStages ? 0 : stage + 1;
                collide_row(g);
                auto store = [&](VT& o, int q) { stream_store<S, SCALED>(o, g[q], wf(q), p.scale); };
                store(C0, 0);
                store(C1, 1);
                store(C2, 2);
                store(C3, 3);
                store(C4, 4);
                store(C5, 5);
                store(C6, 6);
                store(C7, 7);
                store(C8, 8);
                if (first) {
                    edge[slot][0][warp] = C3.e[0];
                    edge[slot][1][warp] = C6.e[0];
                    edge[slot][2][warp] = C7.e[0];
                }
                if (last && (OPEN || active)) {
                    edge[slot][3][warp] = C1.e[V - 1];
                    edge[slot][4][warp] = C5.e[V - 1];
                    edge[slot][5][warp] = C8.e[V - 1];
                }
                __syncwarp();
            } else {  // the top wall returns the last row's own 2, 5, 6 in directions 4, 7, 8
                C4 = ws.up[(k + 1) & 1][0][lane];
                C7 = ws.up[(k + 1) & 1][1][lane];
                C8 = ws.up[(k + 1) & 1][2][lane];
                __syncwarp();  // every lane has read the edge values of the rows before
            }
            const VT A2 = ws.up[k & 1][0][lane], A5 = ws.up[k & 1][1][lane], A6 = ws.up[k & 1][2][lane];
            if (real) {
                ws.up[k & 1][0][lane] = C2;
                ws.up[k & 1][1][lane] = C5;
                ws.up[k & 1][2][lane] = C6;
            }
            // the neighbours' edge values of this row.  A warp that waits here
            // has seen its neighbours finish the row before last, so the ring of
            // four rows is never overwritten early.
            if (lane == 0) mbar_arrive(smem_addr(&edge_ready[slot][warp]));
            const bool ok = mbar_wait_cycles(smem_addr(&edge_ready[slot][wl]), (k >> 2) & 1u, kWaitCycles) &&
                            mbar_wait_cycles(smem_addr(&edge_ready[slot][wr]), (k >> 2) & 1u, kWaitCycles);
            if (!__all_sync(0xffffffffu, ok)) {  // a wait ran out: report it and leave, after the copies in flight
                if (lane == 0 && p.err_flag) atomicExch(p.err_flag, 1);
                asm volatile("cp.async.wait_all;\n" ::: "memory");
                return;
            }
            const int yo = y1 - 1;
            if (yo >= w.ya) {
                // ---- second step of row yo
                const int sm1 = (slot + 3) & 3, sm2 = (slot + 2) & 3;
                float2 g[9][V / 2];
                T e1{}, e5{}, e8{}, e3{}, e6{}, e7{};
                if (first) {
                    e1 = edge[sm1][3][wl];
                    e5 = edge[sm2][4][wl];
                    e8 = edge[slot][5][wl];
                }
                if (last) {
                    e3 = edge[sm1][0][wr];
                    e6 = edge[sm2][1][wr];
                    e7 = edge[slot][2][wr];
                }
                stream_pull<S, SCALED, 0>(g, B0, T(), false, p.inv_scale);
                stream_pull<S, SCALED, 2>(g, A2, T(), false, p.inv_scale);
                stream_pull<S, SCALED, 4>(g, C4, T(), false, p.inv_scale);
                stream_pull<S, SCALED, 1>(g, B1, e1, first, p.inv_scale);
                stream_pull<S, SCALED, 5>(g, A5, e5, first, p.inv_scale);
                stream_pull<S, SCALED, 8>(g, C8, e8, first, p.inv_scale);
                stream_pull<S, SCALED, 3>(g, B3, e3, last, p.inv_scale);
                stream_pull<S, SCALED, 6>(g, A6, e6, last, p.inv_scale);
                stream_pull<S, SCALED, 7>(g, C7, e7, last, p.inv_scale);
                if (yo == 0) {  // A holds the row's own 4, 7, 8
                    stream_own<S, SCALED, 5>(g, A5, p.inv_scale);
                    stream_own<S, SCALED, 6>(g, A6, p.inv_scale);
                }
                if (yo == ny - 1) {  // C holds the row's own 2, 5, 6
                    stream_own<S, SCALED, 7>(g, C7, p.inv_scale);
                    stream_own<S, SCALED, 8>(g, C8, p.inv_scale);
                }
                collide_row(g);
                if (streamed && !(apart && yo >= rg.r0 && yo < rg.r1)) {
                    const int plane = stream_opaque((int)p.plane);
                    T* out = dst + yo * p.pitch + x0;
#pragma unroll
                    for (int q = 0; q < 9; ++q) {
                        VT o;
                        stream_store<S, SCALED>(o, g[q], wf(q), p.scale);
                        st_stream<T, V>(out + q * plane, o);
                    }
                }
            }
            if (real) {
                if (y1 == 0) {  // the bottom wall returns row 0's own 4, 7, 8 in directions 2, 5, 6
                    ws.up[(k + 1) & 1][0][lane] = C4;
                    ws.up[(k + 1) & 1][1][lane] = C7;
                    ws.up[(k + 1) & 1][2][lane] = C8;
                }
                B0 = C0;
                B1 = C1;
                B3 = C3;
            }
        }
    } while (w.piece());
}

// threads of a block: a row's columns, in warps (an open channel's without its outlet column)
inline int stream_threads(const StepParams& p)
{
    return ((p.open ? p.nx - 1 : p.nx) + 32 * kStreamV - 1) / (32 * kStreamV) * 32;
}

// blocks an SM holds: of the 512 threads that 128 registers leave room for, those
// that fit its shared memory.  FP32 rows of at most 128 sites: 15 blocks of a warp, not
// 16; a grid of 16 an SM left 152 blocks to a second wave (128 x 64, 494 clones,
// us a step with 16 / 15: BGK 36.4 / 32.4, central moments 50.3 / 42.1)
template <int S>
int stream_blocks_per_sm(int threads)
{
    constexpr int kStatic = 4 * 6 * (kStreamMaxThreads / 32) * (int)sizeof(typename Codec<S>::T) +
                            4 * (kStreamMaxThreads / 32) * (int)sizeof(uint64_t);
    int dev = 0, smem = 228 * 1024, reserved = 1024;
    if (cudaGetDevice(&dev) == cudaSuccess) {
        cudaDeviceGetAttribute(&smem, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
        cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, dev);
    }
    const int bytes = threads / 32 * (int)sizeof(StreamWarpSmem<S>) + kStatic + reserved;
    const int fit = smem / ((bytes + 127) / 128 * 128), most = kStreamMaxThreads / threads;
    return fit < 1 ? 1 : (fit < most ? fit : most);
}

inline int stream_sms()
{
    int sms = 152, dev = 0;
    if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return sms;
}

// whole rows of at most 2048 sites in a block, the work apart in its shared
// memory; in an open channel the column ranges and the obstacle's region apart
template <int S>
bool stream_supported(const StepParams& p)
{
    const int threads = stream_threads(p);
    const size_t smem = threads / 32 * sizeof(StreamWarpSmem<S>);
    const StreamRegion<S> rg(p);
    if (threads > kStreamMaxThreads || rg.bytes(2) > smem || (int64_t)p.n_list * p.ny >= ((int64_t)1 << 31)) return false;
    if (!p.open) return p.nx % kStreamGroup<S> == 0;
    const StreamColumns<S> cols(p);
    if (p.nx < 32 || !cols.apart(rg)) return false;
    for (int r = 0; r < 3; ++r)
        if (cols.g1[r] > cols.g0[r] && cols.chunk(r, threads, smem, p.ny) < 1) return false;
    return true;
}

// whether calls of four steps and more take less time streamed than in single steps
// of the default variant.  In units of a streamed row's time, with R rows a block, a
// block takes R + 2 of them (it recomputes two), c for every row's worth of sites
// computed apart, and d shared by the SM's blocks, whose apart work and first rows
// overlap with the others' rows; single steps take `gain` rows for each row.  16-bit
// steps are bound by instructions: there the lanes that the single step's 256-column
// segments leave idle count, and the warps that the SM lacks where rows of 5, 6 or 7
// warps leave some out.  The figures are fitted to 952 measurements, single and
// streamed, channels of 64 to 2049 columns, 4 to 48 rows a block, obstacles up to 3/4
// and grids up to 64 columns wide; the choice costs 0.4 % on average, at most 10 %
// (16-bit rows of 640 and 2049 columns), 17 % where it stays with single steps.
// Some (us a step, single / streamed):
//   FP32 BGK      1024 x 256, 32 x 32 square, 15 clones 45.8 / 29.9; with 200 x 200 48.3 / 49.5
//   FP32 CM       1024 x 256, 15 clones 45.4 / 38.9; 200 x 200, 48 clones 151 / 176
//   FP16 BGK      2048 x 512, 12 clones 78.7 / 66.1; 256 x 64, 32 x 32, 247 clones 36.2 / 45.8
//   FP16 CM       2048 x 512, 12 clones 90.1 / 88.5; 512 x 128, 64 x 64, 190 clones 107 / 129
//   open FP32 CM  513 x 129, 61 clones 58.9 / 56.4; 2049 x 513, 4 clones 52.9 / 61.4
//   open FP32 BGK 513 x 129, 118 clones 104 / 98.9; bars of 64 columns, 127 clones 114 / 124
//   open FP16 CM  513 x 129, 66 clones 76.5 / 54.7; 769 x 193, 22 clones 40.8 / 48.2
template <int S>
bool stream_pays(const StepParams& p)
{
    constexpr int G = kStreamGroup<S>;
    const int threads = stream_threads(p), ctas = stream_blocks_per_sm<S>(threads);
    const double rows = (double)p.n_list * p.ny / ((double)ctas * stream_sms());
    const StreamRegion<S> rg(p);
    double apart = (double)rg.ng * G * (rg.r1 - rg.r0) / ((double)p.nx * p.ny);
    if (p.open) {
        const StreamColumns<S> cols(p);
        for (int r = 0; r < 3; ++r)
            if (cols.g1[r] > cols.g0[r]) apart += (double)(cols.g1[r] - cols.g0[r]) * G / p.nx;
    }
    struct Cost {
        double gain, c, d;
    };
    const bool bgk = p.coll == 0;
    const Cost k = S == kFP32 ? (p.open ? (bgk ? Cost{1.6, 3.0, 20.0} : Cost{1.8, 1.0, 20.0})
                                        : (bgk ? Cost{1.5, 3.0, 1.0} : Cost{1.35, 3.0, 1.0}))
                              : (p.open ? Cost{2.2, 0.0, 20.0} : (bgk ? Cost{1.6, 8.0, 9.0} : Cost{1.1, 2.0, 1.0}));
    double gain = k.gain;
    if (S != kFP32) {
        const int segments = ((p.open ? p.nx - 1 : p.nx) + 32 * G - 1) / (32 * G);
        gain *= (double)segments * 32 * G / (threads * kStreamV) * (ctas * threads) / kStreamMaxThreads;
    }
    return rows * (gain - 1.0 - k.c * apart) >= 2.0 + k.d / ctas;
}

template <int S, bool SCALED, int COLL, bool OPEN>
cudaError_t launch_stream_kernel(const StepParams& p, cudaStream_t s)
{
    const int threads = stream_threads(p);
    const int ctas = stream_blocks_per_sm<S>(threads), sms = stream_sms();
    const size_t smem = threads / 32 * sizeof(StreamWarpSmem<S>);
    const int64_t rows = (int64_t)p.n_list * p.ny;
    const int grid = (int)(rows < (int64_t)ctas * sms ? rows : (int64_t)ctas * sms);
    const cudaError_t e = cudaFuncSetAttribute(step_stream_kernel<S, SCALED, COLL, OPEN>,
                                               cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               (int)(kStreamMaxThreads / 32 * sizeof(StreamWarpSmem<S>)));
    if (e != cudaSuccess) return e;
    step_stream_kernel<S, SCALED, COLL, OPEN><<<grid, threads, smem, s>>>(p);
    return cudaGetLastError();
}

// one launch of two steps, or of a single one by the register-staged kernel
// with the same drag segments
template <int S, bool OPEN>
cudaError_t launch_stream_of(const StepParams& p, cudaStream_t s)
{
    if (p.tb_steps == 1) {
        if constexpr (OPEN)
            return launch_step_open<S, kStreamGroup<S>, 4>(p, s);
        else
            return launch_step<S, kStreamGroup<S>, 4>(p, s);
    }
    if (!stream_supported<S>(p) || p.tb_steps != 2) return cudaErrorInvalidValue;
    const bool scaled = S != kFP32 && p.scale != 1.0f;
    if (p.coll == 1)
        return scaled ? launch_stream_kernel<S, S != kFP32, 1, OPEN>(p, s) : launch_stream_kernel<S, false, 1, OPEN>(p, s);
    return scaled ? launch_stream_kernel<S, S != kFP32, 0, OPEN>(p, s) : launch_stream_kernel<S, false, 0, OPEN>(p, s);
}

template <int S>
cudaError_t launch_stream(const StepParams& p, cudaStream_t s)
{
    return launch_stream_of<S, false>(p, s);
}

template <int S>
cudaError_t launch_stream_open(const StepParams& p, cudaStream_t s)
{
    return launch_stream_of<S, true>(p, s);
}

}  // namespace lbm
