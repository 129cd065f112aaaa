// Axis permutation of a row-major tensor (the "T" of TTGT, Section 5.1): out axis t = in axis
// perm[t].  Moves bytes only, so it is exact for any payload.  Axes that stay adjacent and in
// order are fused first, and a surviving innermost axis widens the element (up to 16 bytes) where
// the buffers are aligned for it.  One kernel then moves tiles (see TilePerm), one copies long surviving runs
// that fill no tile (k_perm_runs), one transposes two long axes of ragged tensors (k_perm_plane).
#include <algorithm>
#include <cstdint>

#include "kernels.cuh"

namespace tn {

namespace {

constexpr int kMaxRank = 32;

struct PermPlan {
    int32_t rank;                 // fused output rank, without the surviving innermost axis
    int64_t odim[kMaxRank];       // output dims, axis 0 slowest
    int64_t istride[kMaxRank];    // input stride of each output axis
    int64_t ostride[kMaxRank];    // output stride of each output axis
    int64_t inner;                // extent of the innermost axis where it survives (stride 1 on both sides), else 1
    int64_t total;
};

// One tile: `inner` (or a chunk of it) x group A x group B x group C.  A is a run of the output's
// innermost axes, B a run of the input's innermost axes, each without the axes that the other one has
// taken (these are whole inside the tile, so the run goes on past them), C further axes of the output
// that fill the tile where A and B cannot (they are not needed when the surviving inner run is
// long).  The last axis of each group may be cut into chunks; the chunk numbers and all other axes
// form the tile index.  A block reads a tile with consecutive threads along (inner, B) -- the input's
// order -- and writes it along (inner, A) -- the output's order -- through shared memory, or straight
// from registers when the two orders agree (no A or no B).
// Bound by HBM.  Everything that depends on the position inside the tile (two offsets and a
// shared-memory index per element) is computed once per block, which then moves up to kTileRun
// tiles: only a base changes from tile to tile, the next tile's loads are in flight while the
// current one is written, and tiles of 8 to 16 KB leave room for several blocks per SM.  Measured on
// 2^26 complex64: all axes reversed 169 us, 6.4 TB/s (297 us with 64 x 64 tiles, one per block, whose
// indices were divided out per element); reversed but for rows of 16 to 512 bytes 164-176 us (470-860
// us when each row was copied by a group of lanes); (37, 5, 129, 3, 61) complex128 shuffled 29 us
// (70 us with 32 x 32 tiles of one axis pair, mostly empty).  Shuffles that put one of the input's
// last axes first in the output need the runs that go on past the other group's axes: one of 2^26
// complex64 takes 168 us, 249 us with runs that stop there (64 bytes and less).
struct TileAxis {
    int64_t in, out;                            // strides
    uint32_t dim;                               // extent inside the tile, or number of tiles along the axis
    uint32_t below;                             // tile index: product of the dims before
};
// The kernel's parameters.  Every block reads them before its first load, so the axes are packed: with an array of
// 32 axes for each group (2.3 KB) a block of a small or ragged tensor spent longer on its parameters and tables than
// on its data ((83910, 88) complex64 transposed 39 us, 34 us packed).
struct TilePerm {
    int32_t ti, ta, tb, tc;                     // tile edges
    int32_t pitch;                              // shared-memory row of tb * ti elements, odd
    int32_t direct;                             // read and write order agree: no shared memory
    uint32_t mi, ma, mb;                        // ceil(2^32 / edge), 0 for an edge of 1
    int32_t na, nb, nc, nr;                     // axes of each group, innermost first, and of the tile index
    uint32_t n_tiles;
    int32_t run;                                // tiles per block
    int32_t lanes;                              // lanes that add up a tile's base: nr up to a power of two, at most 32
    struct Cut {
        int64_t dim;                            // the cut axis' extent
        int32_t axis;                           // tile-index axis that numbers the chunks (-1: whole)
        int32_t len;                            // chunk length
        int32_t before;                         // product of the group's tile extents before the cut axis
    } cut[4];                                   // of inner, A, B, C
    TileAxis ax[kMaxRank + 4];                  // of A, B, C and the tile index, one after the other
};
constexpr int kTileRun = 8;    // most tiles per block
constexpr int kTileEdge = 32;  // elements of the runs on both sides

// Quotient of e < 2^16 by an edge d <= 2^12 from m = ceil(2^32 / d): exact, as e d < 2^32.
__device__ __forceinline__ uint32_t quot(uint32_t e, uint32_t m) { return m ? __umulhi(e, m) : e; }

// Offsets in the input and in the output of a multi-index below the product of n axes' extents.
__device__ __forceinline__ void digits_off(uint32_t idx, int32_t n, const TileAxis *ax, int64_t &in, int64_t &out) {
    in = out = 0;
#pragma unroll 1
    for (int32_t t = 0; t < n; ++t) {
        uint32_t q = 0;
        if (t + 1 < n) q = idx / ax[t].dim;
        in += (int64_t)(idx - q * ax[t].dim) * ax[t].in;
        out += (int64_t)(idx - q * ax[t].dim) * ax[t].out;
        idx = q;
    }
}

// RAGGED: some cut axis has a short last chunk.  O: type of the offsets inside a tile.
template <typename E, int PER, bool RAGGED, typename O>
__global__ void __launch_bounds__(256, !RAGGED && sizeof(E) == 16 ? 5 : 0) k_perm_tile(const E *__restrict__ in, E *__restrict__ out,
                                                   const __grid_constant__ TilePerm g) {
    extern __shared__ __align__(16) char dyn[];
    __shared__ int64_t s_base[kTileRun][2];
    __shared__ ushort4 s_lim[kTileRun];   // extents of each tile in inner, A, B, C where short of the edges
    __shared__ int32_t s_edge[kTileRun];  // some extent is short
    O *in_a = reinterpret_cast<O *>(dyn), *in_b = in_a + g.ta, *in_c = in_b + g.tb;   // input offsets of the indices
    O *out_a = in_c + g.tc, *out_b = out_a + g.ta, *out_c = out_b + g.tb;             // output offsets
    const TileAxis *A = g.ax, *B = A + g.na, *C = B + g.nb, *R = C + g.nc;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t t0 = blockIdx.x * (uint32_t)g.run, nt = min((uint32_t)g.run, g.n_tiles - t0);
    // tile bases: a warp per tile, the last warp first (the first ones compute the tables below), a lane per axis of
    // the tile index (at most 36: two rounds)
    for (uint32_t t = 7 - warp; t < nt; t += 8) {
        int64_t si = 0, so = 0;
        uint32_t short_axes = 0;
        uint16_t lim[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) lim[q] = 0xffff;
        for (int x = lane; x < g.nr; x += 32) {
            const uint32_t d = ((t0 + t) / R[x].below) % R[x].dim;
            si += (int64_t)d * R[x].in;
            so += (int64_t)d * R[x].out;
            if (RAGGED) {
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    if (g.cut[q].axis == x) {
                        const int64_t left = g.cut[q].dim - (int64_t)d * g.cut[q].len;
                        if (left < g.cut[q].len) {
                            lim[q] = (uint16_t)(left * g.cut[q].before);
                            short_axes = 1;
                        }
                    }
            }
        }
#pragma unroll 1
        for (int o = g.lanes >> 1; o > 0; o >>= 1) {
            si += __shfl_xor_sync(0xffffffffu, si, o);
            so += __shfl_xor_sync(0xffffffffu, so, o);
        }
        if (lane == 0) {
            s_base[t][0] = si;
            s_base[t][1] = so;
        }
        if (RAGGED) {
            const int edge = __any_sync(0xffffffffu, short_axes != 0);
#pragma unroll
            for (int q = 0; q < 4; ++q) lim[q] = (uint16_t)__reduce_min_sync(0xffffffffu, (unsigned)lim[q]);
            if (lane == 0) {
                s_lim[t] = make_ushort4(lim[0], lim[1], lim[2], lim[3]);
                s_edge[t] = edge;
            }
        }
    }
    // the input and output offsets of each A, B and C index
    for (int i = tid; i < g.ta + g.tb + g.tc; i += 256) {
        const bool b = i >= g.ta, c = i >= g.ta + g.tb;
        int64_t oi, oo;
        digits_off(c ? i - g.ta - g.tb : b ? i - g.ta : i, c ? g.nc : b ? g.nb : g.na, c ? C : b ? B : A, oi, oo);
        in_a[i] = (O)oi;
        out_a[i] = (O)oo;
    }
    __syncthreads();
    // per element of this thread: where it is read (order c, a, b, i) and written (order c, b, a, i)
    const uint32_t ti = g.ti, ta = g.ta, tb = g.tb, n = ti * ta * tb * (uint32_t)g.tc;
    O rd[PER], wr[PER];
    uint32_t sr[PER];        // shared-memory indices: store at the low half, load from the high half
    uint2 dr[PER], dw[PER];  // indices in inner, A, B, C, against s_lim
#pragma unroll
    for (int u = 0; u < PER; ++u) {
        const uint32_t e = tid + u * 256;
        rd[u] = wr[u] = -1;
        sr[u] = 0;
        if (RAGGED) dr[u] = dw[u] = make_uint2(0, 0);
        if (e < n) {
            uint32_t q = quot(e, g.mi), i = e - q * ti, q2 = quot(q, g.mb), b = q - q2 * tb, c = quot(q2, g.ma),
                     a = q2 - c * ta;
            rd[u] = in_a[a] + in_b[b] + in_c[c] + (O)i;
            sr[u] = (c * ta + a) * (uint32_t)g.pitch + b * ti + i;
            if (RAGGED) dr[u] = make_uint2(i | a << 16, b | c << 16);
            q2 = quot(q, g.ma), a = q - q2 * ta, c = quot(q2, g.mb), b = q2 - c * tb;
            wr[u] = out_a[a] + out_b[b] + out_c[c] + (O)i;
            sr[u] |= ((c * ta + a) * (uint32_t)g.pitch + b * ti + i) << 16;
            if (RAGGED) dw[u] = make_uint2(i | a << 16, b | c << 16);
        }
    }
    E *tile = reinterpret_cast<E *>(dyn);
    // inside the extents of tile t (all of it unless the tile is at an edge)
    auto inside = [&](uint32_t t, const uint2 &d) {
        if (!RAGGED || !s_edge[t]) return true;
        const ushort4 l = s_lim[t];
        return (d.x & 0xffffu) < l.x && (d.x >> 16) < l.y && (d.y & 0xffffu) < l.z && (d.y >> 16) < l.w;
    };
    E v[PER];
    auto load = [&](uint32_t t) {
        const E *src = in + s_base[t][0];
#pragma unroll
        for (int u = 0; u < PER; ++u)
            if (rd[u] >= 0 && inside(t, dr[u])) v[u] = __ldg(src + rd[u]);
    };
    load(0);
    __syncthreads();   // the offset tables give way to the tile
    for (uint32_t t = 0; t < nt; ++t) {
        E *dst = out + s_base[t][1];
        if (g.direct) {
#pragma unroll
            for (int u = 0; u < PER; ++u)
                if (wr[u] >= 0 && inside(t, dw[u])) dst[wr[u]] = v[u];
            if (t + 1 < nt) load(t + 1);
            continue;
        }
#pragma unroll
        for (int u = 0; u < PER; ++u)
            if (rd[u] >= 0) tile[sr[u] & 0xffffu] = v[u];
        __syncthreads();
        if (t + 1 < nt) load(t + 1);
#pragma unroll
        for (int u = 0; u < PER; ++u)
            if (wr[u] >= 0 && inside(t, dw[u])) dst[wr[u]] = tile[sr[u] >> 16];
        if (t + 1 < nt) __syncthreads();
    }
}

// Long surviving runs of which no whole number fills a tile: G lanes copy one run (or a chunk of it), kRunLoads loads
// in flight each, sharing the division of its number into axes; with fewer lanes for short runs a warp has
// several runs in flight.  Bound by HBM from 4 bytes an element, by the loads issued below that.  Ragged tiles of
// 1024 elements (or tiles half empty) kept too few bytes in flight: (1291, 1301, 1307) with its outer axes exchanged
// 5.4 ms in complex64 (6.5 TB/s) and 1.3 ms in bytes, 14.1 and 7.4 ms in tiles, 5.5 and 2.1 ms with a warp
// per run and four loads; (1436, 1437, 65) complex64 358 us, 771 and 810 us.
constexpr int kRunChunk = 2048, kRunLoads = 6;
template <typename E, int G>
__global__ void __launch_bounds__(256) k_perm_runs(const E *__restrict__ in, E *__restrict__ out,
                                                   const __grid_constant__ TilePerm g) {
    constexpr uint32_t per = 32 / G;
    constexpr int U = kRunLoads;
    const uint32_t lane = threadIdx.x & 31, sub = lane & (G - 1), grp = lane / G;
    const uint32_t warps = gridDim.x * 8;
    for (uint32_t t0 = (blockIdx.x * 8 + (threadIdx.x >> 5)) * per; t0 < g.n_tiles; t0 += warps * per) {
        const uint32_t t = t0 + grp;
        int64_t si = 0, so = 0;
        for (int x = sub; x < g.nr; x += G) {
            const uint32_t d = (t / g.ax[x].below) % g.ax[x].dim;
            si += (int64_t)d * g.ax[x].in;
            so += (int64_t)d * g.ax[x].out;
        }
#pragma unroll 1
        for (int o = g.lanes >> 1; o > 0; o >>= 1) {
            si += __shfl_xor_sync(0xffffffffu, si, o);
            so += __shfl_xor_sync(0xffffffffu, so, o);
        }
        const E *src = in + __shfl_sync(0xffffffffu, si, lane - sub);
        E *dst = out + __shfl_sync(0xffffffffu, so, lane - sub);
        int32_t n = t < g.n_tiles ? g.ti : 0;
        if (g.cut[0].axis >= 0)   // the chunk number is the first axis
            n = (int32_t)min((int64_t)n, g.cut[0].dim - (int64_t)(t % g.ax[0].dim) * n);
        for (int32_t i0 = sub; i0 < n; i0 += G * U) {
            E v[U];
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (i0 + G * u < n) v[u] = __ldg(src + i0 + G * u);
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (i0 + G * u < n) dst[i0 + G * u] = v[u];
        }
    }
}

// The tile index of plan p's runs; false where they are too few to fill the GPU (2048 are six warps an SM in each
// pass; 812 runs of 20011 complex64 numbers took the same time either way).
bool run_perm(const PermPlan &p, TilePerm &g) {
    const int64_t chunks = (p.inner + kRunChunk - 1) / kRunChunk;
    g.ti = (int32_t)((p.inner + chunks - 1) / chunks);
    g.cut[0] = {p.inner, chunks > 1 ? 0 : -1, g.ti, 1};
    int64_t tiles = 1;
    g.nr = 0;
    auto axis = [&](int64_t dim, int64_t in, int64_t out) {
        if (dim > 0x7fffffffLL || tiles > 0x7fffffffLL / dim) return false;
        g.ax[g.nr++] = {in, out, (uint32_t)dim, (uint32_t)tiles};
        tiles *= dim;
        return true;
    };
    if (chunks > 1 && !axis(chunks, g.ti, g.ti)) return false;
    for (int32_t t = p.rank - 1; t >= 0; --t)
        if (!axis(p.odim[t], p.istride[t], p.ostride[t])) return false;
    for (g.ta = 8; g.ta < 32 && g.ta * kRunLoads < g.ti;) g.ta *= 2;
    for (g.lanes = 1; g.lanes < std::min(g.nr, g.ta);) g.lanes *= 2;
    g.n_tiles = (uint32_t)tiles;
    return tiles >= 2048;
}

// The transposition of two long axes (the output's innermost and the input's innermost), one 32 x 32 tile of
// them a block: no tables, next to no set-up, eight blocks an SM.  Taken where the general kernel's tiles would be ragged
// and the 32 x 32 ones are at least half full.  Against the ragged tiles it takes 0.5 to 0.9 of the time over 300 shapes
// of 2^18 to 2^27 elements (at a fill of 0.52 to 0.56 as much or less): (1354, 625) complex64 hot in L2 4.2 us, 10.3 us;
// (745, 12738) float32 18.5 us, 28 us; (6466, 2337) complex64 39 us, 56 us; (1158, 1430) complex128 12.4 us, 16.4 us.
template <typename E>
__global__ void __launch_bounds__(256) k_perm_plane(const E *__restrict__ in, E *__restrict__ out,
                                                    const __grid_constant__ TilePerm g) {
    __shared__ E tile[32][33];
    const TileAxis *ax = g.ax;   // tiles of the two axes, then the others
    uint32_t blk = blockIdx.x, q = blk / (uint32_t)g.ta;
    const uint32_t a0 = (blk - q * g.ta) * 32;
    blk = q;
    q = blk / (uint32_t)g.tb;
    const uint32_t b0 = (blk - q * g.tb) * 32;
    for (int32_t x = 2; x < g.nr; ++x) {
        blk = q;
        q = x + 1 < g.nr ? blk / ax[x].dim : 0;
        in += (int64_t)(blk - q * ax[x].dim) * ax[x].in;
        out += (int64_t)(blk - q * ax[x].dim) * ax[x].out;
    }
    const uint32_t tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    E v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const uint32_t a = a0 + ty + 8 * u, b = b0 + tx;
        if (a < ax[0].dim && b < ax[1].dim) v[u] = __ldg(in + (int64_t)a * ax[0].in + b);
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) tile[ty + 8 * u][tx] = v[u];
    __syncthreads();
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const uint32_t b = b0 + ty + 8 * u, a = a0 + tx;
        if (a < ax[0].dim && b < ax[1].dim) out[(int64_t)b * ax[1].out + a] = tile[tx][ty + 8 * u];
    }
}

// The two axes of plan p and its other ones, where k_perm_plane takes them (see there).
bool plane_perm(const PermPlan &p, TilePerm &g) {
    if (p.inner != 1 || p.rank < 2) return false;
    const int32_t a = p.rank - 1;
    int32_t b = 0;
    while (p.istride[b] != 1) ++b;
    const int64_t da = p.odim[a], db = p.odim[b], ta = (da + 31) / 32, tb = (db + 31) / 32;
    int64_t tiles = p.total / (da * db);
    if (da > 0x7fffffffLL || db > 0x7fffffffLL || 2 * da * db < (ta * 32) * (tb * 32)) return false;
    if (ta > 0x7fffffffLL / tb || tiles > 0x7fffffffLL / (ta * tb)) return false;
    tiles *= ta * tb;
    g.ta = (int32_t)ta;
    g.tb = (int32_t)tb;
    g.n_tiles = (uint32_t)tiles;
    g.nr = 0;
    auto axis = [&](int32_t t) { g.ax[g.nr++] = {p.istride[t], p.ostride[t], (uint32_t)p.odim[t], 0}; };
    axis(a);
    axis(b);
    for (int32_t t = a - 1; t >= 0; --t)
        if (t != b) axis(t);
    return true;
}

// Builds the tiles of plan p: runs of about `edge` elements on both sides, at most `area` elements.
// false if the tensor has too many of them.
bool tile_perm(const PermPlan &p, int32_t edge, int32_t area, TilePerm &g) {
    // fixed arrays: a small permutation costs little more than its launch
    char used[kMaxRank] = {};
    int32_t by_in[kMaxRank];  // axes by increasing input stride
    for (int32_t t = 0; t < p.rank; ++t) by_in[t] = t;
    std::sort(by_in, by_in + p.rank, [&](int32_t x, int32_t y) { return p.istride[x] < p.istride[y]; });
    struct Axis { int64_t dim, in, out; };
    struct Axes {
        Axis a[kMaxRank + 4];
        int32_t n = 0;
        void push_back(const Axis &x) { a[n++] = x; }
        Axis &back() { return a[n - 1]; }
    } A, B, C, R;
    // an edge of at most t splits n indices into chunks of equal length
    auto chunk = [](int64_t n, int64_t t) {
        const int64_t c = (n + t - 1) / t;
        return (n + c - 1) / c;
    };
    auto prod = [](const Axes &v) {
        int64_t x = 1;
        for (int32_t i = 0; i < v.n; ++i) x *= v.a[i].dim;
        return x;
    };
    int32_t ia = p.rank - 1, ib = 0;
    auto take = [&](Axes &v, int32_t t) {
        v.push_back({p.odim[t], p.istride[t], p.ostride[t]});
        used[t] = 1;
    };
    // a run goes on past the axes of the other group unless that one's last axis is about to be cut (past a cut
    // axis nothing is contiguous)
    auto grow_a = [&](int64_t lim, int64_t lim_b) {
        while (ia >= 0 && used[ia] && prod(B) <= lim_b) --ia;
        if (ia < 0 || used[ia] || prod(A) >= lim) return false;
        take(A, ia--);
        return true;
    };
    auto grow_b = [&](int64_t lim, int64_t lim_a) {
        while (ib < p.rank && used[by_in[ib]] && prod(A) <= lim_a) ++ib;
        if (ib >= p.rank || used[by_in[ib]] || prod(B) >= lim) return false;
        take(B, by_in[ib++]);
        return true;
    };
    for (TilePerm::Cut &c : g.cut) c = {0, -1, 1, 1};
    // cuts the last axis of a group so that its extent is at most lim
    auto cut = [&](Axes &v, int64_t lim, int q) {
        if (v.n == 0) return;
        Axis &last = v.back();
        const int64_t before = prod(v) / last.dim, len = chunk(last.dim, std::max<int64_t>(1, lim / before));
        if (len < last.dim) {
            R.push_back({(last.dim + len - 1) / len, last.in * len, last.out * len});
            g.cut[q] = {last.dim, R.n - 1, (int32_t)len, (int32_t)before};   // index into R, renumbered below
            last.dim = len;
        }
    };
    int64_t ti = p.inner;
    if (ti > area) {
        ti = chunk(p.inner, area);
        R.push_back({(p.inner + ti - 1) / ti, ti, ti});
        g.cut[0] = {p.inner, 0, (int32_t)ti, 1};
    }
    int64_t lim_a = std::max<int64_t>(1, edge / ti), lim_b = std::max<int64_t>(1, area / (ti * lim_a));
    if (ti >= edge) lim_b = 1;   // long surviving runs: whole rows, in the order of the output (C)
    for (bool more = true; more;) {   // in turn, so that neither takes all the short axes
        const bool ga = grow_a(lim_a, lim_b), gb = grow_b(lim_b, lim_a);
        more = ga || gb;
    }
    // a group that is blocked short of its edge leaves more of the tile to the other
    if (ti < edge && prod(A) < lim_a) {
        lim_b = std::max(lim_b, area / (ti * prod(A)));
        while (grow_b(lim_b, lim_a)) {}
    }
    if (ti < edge && prod(B) < lim_b) {
        lim_a = std::max(lim_a, area / (ti * prod(B)));
        while (grow_a(lim_a, lim_b)) {}
    }
    cut(A, lim_a, 1);
    cut(B, lim_b, 2);
    const int64_t ta = prod(A), tb = prod(B), room = std::max<int64_t>(1, area / (ti * ta * tb));
    for (int32_t t = p.rank - 1; t >= 0 && prod(C) < room; --t)
        if (!used[t]) take(C, t);
    cut(C, room, 3);
    const int64_t tc = prod(C);
    if (ti * ta * tb * tc > area) return false;
    g.ti = (int32_t)ti;
    g.ta = (int32_t)ta;
    g.tb = (int32_t)tb;
    g.tc = (int32_t)tc;
    g.pitch = (int32_t)((tb * ti) | 1);
    g.direct = ta == 1 || tb == 1;
    auto magic = [](int64_t d) { return d == 1 ? 0u : (uint32_t)(((uint64_t(1) << 32) + d - 1) / d); };
    g.mi = magic(ti);
    g.ma = magic(ta);
    g.mb = magic(tb);
    g.na = A.n;
    g.nb = B.n;
    g.nc = C.n;
    TileAxis *ax = g.ax;
    for (const Axes *v : {&A, &B, &C})
        for (int32_t i = 0; i < v->n; ++i) *ax++ = {v->a[i].in, v->a[i].out, (uint32_t)v->a[i].dim, 0};
    // the tile index: chunk numbers and the other axes, innermost in the output first, so that
    // consecutive tiles write neighbouring runs
    for (int32_t t = 0; t < p.rank; ++t)
        if (!used[t]) R.push_back({p.odim[t], p.istride[t], p.ostride[t]});
    int32_t ord[kMaxRank + 4];
    for (int32_t i = 0; i < R.n; ++i) ord[i] = i;
    std::sort(ord, ord + R.n, [&](int32_t x, int32_t y) { return R.a[x].out < R.a[y].out; });
    g.nr = R.n;
    for (g.lanes = 1; g.lanes < std::min(g.nr, 32);) g.lanes *= 2;
    int64_t tiles = 1;
    int32_t cuts[4] = {-1, -1, -1, -1};
    for (int32_t i = 0; i < g.nr; ++i) {
        const Axis &x = R.a[ord[i]];
        if (x.dim > 0x7fffffffLL || tiles > 0x7fffffffLL / x.dim) return false;
        *ax++ = {x.in, x.out, (uint32_t)x.dim, (uint32_t)tiles};
        tiles *= x.dim;
        for (int q = 0; q < 4; ++q)
            if (g.cut[q].axis == ord[i]) cuts[q] = i;
    }
    for (int q = 0; q < 4; ++q) g.cut[q].axis = cuts[q];
    g.n_tiles = (uint32_t)tiles;
    return true;
}

// per_sm: several tiles per block once every SM has that many blocks.
template <typename E, int PER, bool RAGGED, typename O>
cudaError_t launch_tiles(const E *in, E *out, TilePerm &g, int32_t per_sm, cudaStream_t st) {
    g.run = (int32_t)std::min<int64_t>(kTileRun, ((int64_t)g.n_tiles + 152 * per_sm - 1) / (152 * per_sm));
    const size_t tables = (size_t)(g.ta + g.tb + g.tc) * 2 * sizeof(O);
    const size_t smem = std::max(tables, g.direct ? 0 : (size_t)g.tc * g.ta * g.pitch * sizeof(E));
    const unsigned blocks = (g.n_tiles + g.run - 1) / g.run;
    k_perm_tile<E, PER, RAGGED, O><<<blocks, 256, smem, st>>>(in, out, g);
    return cudaGetLastError();
}

template <typename E, int G>
cudaError_t launch_runs(const E *in, E *out, const TilePerm &g, cudaStream_t st) {
    constexpr unsigned per = 8 * (32 / G);
    const unsigned nb = std::min<unsigned>((g.n_tiles + per - 1) / per, 152 * 8);
    k_perm_runs<E, G><<<nb, 256, 0, st>>>(in, out, g);
    return cudaGetLastError();
}

// Tiles of 2048 elements of up to 8 bytes where no chunk is short, of 1024 otherwise: a 16-byte element
// fills 16 KB with 1024, and the bookkeeping of ragged tiles costs registers per element (four of their blocks of
// up to 8 bytes an element fit an SM: a target of six left a second wave half empty).
template <typename E>
cudaError_t perm_launch(const void *src, void *dst, const PermPlan &p, cudaStream_t st) {
    if (p.total == 0) return cudaSuccess;
    const E *in = static_cast<const E *>(src);
    E *out = static_cast<E *>(dst);
    constexpr int AREA = sizeof(E) <= 8 ? 2048 : 1024;
    const bool wide = p.total > 0x7fffffffLL, runs = p.inner >= kTileEdge;
    TilePerm g;
    // no chunk is short, and of long surviving runs of up to 8 bytes an element enough fit in to fill the tile
    auto whole = [runs](const TilePerm &t, int32_t area) {
        bool r = !runs || sizeof(E) == 16 || 4 * t.ti * t.tc >= 3 * area;
        for (const TilePerm::Cut &c : t.cut) r = r && (c.axis < 0 || c.dim % c.len == 0);
        return r;
    };
    if (!wide && p.total > 152 * 6 * 1024) {   // enough tiles to choose their size
        if (!tile_perm(p, kTileEdge, AREA, g)) return cudaErrorInvalidValue;
        if (whole(g, AREA)) return launch_tiles<E, AREA / 256, false, int32_t>(in, out, g, 6, st);
    }
    if (!tile_perm(p, kTileEdge, 1024, g)) return cudaErrorInvalidValue;
    if (!wide && whole(g, 1024)) return launch_tiles<E, 4, false, int32_t>(in, out, g, 6, st);
    if (TilePerm r; runs && run_perm(p, r)) {
        switch (r.ta) {
            case 8: return launch_runs<E, 8>(in, out, r, st);
            case 16: return launch_runs<E, 16>(in, out, r, st);
            default: return launch_runs<E, 32>(in, out, r, st);
        }
    }
    if (TilePerm r; plane_perm(p, r)) {
        k_perm_plane<E><<<r.n_tiles, 256, 0, st>>>(in, out, r);
        return cudaGetLastError();
    }
    constexpr int32_t per_sm = sizeof(E) == 16 ? 6 : 4;
    return wide ? launch_tiles<E, 4, true, int64_t>(in, out, g, per_sm, st)
                : launch_tiles<E, 4, true, int32_t>(in, out, g, per_sm, st);
}

// The fused plan of a permutation; false if it has too many axes.
bool perm_plan(int32_t rank, const int64_t *dims, const int32_t *perm, PermPlan &p) {
    // input strides (rank <= kMaxRank)
    if (rank > kMaxRank) return false;
    int64_t istr[kMaxRank];
    int64_t acc = 1;
    for (int32_t t = rank - 1; t >= 0; --t) { istr[t] = acc; acc *= dims[t]; }
    p = PermPlan{};
    p.total = acc;
    p.inner = 1;
    // output axes (dims of 1 dropped), fused when adjacent in the input in the same order
    int64_t od[kMaxRank], is[kMaxRank];
    int32_t n = 0;
    for (int32_t t = 0; t < rank; ++t) {
        const int64_t d = dims[perm[t]], s = istr[perm[t]];
        if (d == 1) continue;
        if (n && is[n - 1] == d * s) {
            od[n - 1] *= d;
            is[n - 1] = s;
        } else {
            od[n] = d;
            is[n++] = s;
        }
    }
    if (n && is[n - 1] == 1) p.inner = od[--n];
    p.rank = n;
    acc = p.inner;
    for (int32_t t = p.rank - 1; t >= 0; --t) {
        p.odim[t] = od[t];
        p.istride[t] = is[t];
        p.ostride[t] = acc;
        acc *= od[t];
    }
    return true;
}

// Moves elements of `by` times the size where the surviving run is a multiple of it.
void widen(PermPlan &p, int64_t by) {
    p.inner /= by;
    p.total /= by;
    for (int32_t t = 0; t < p.rank; ++t) {
        p.istride[t] /= by;   // multiples of the whole surviving run
        p.ostride[t] /= by;
    }
}

}  // namespace

cudaError_t launch_permute(const void *src, void *dst, int32_t elem_bytes, int32_t rank,
                           const int64_t *dims, const int32_t *perm, cudaStream_t stream) {
    PermPlan p;
    if (!perm_plan(rank, dims, perm, p)) return cudaErrorInvalidValue;
    const uintptr_t at = reinterpret_cast<uintptr_t>(src) | reinterpret_cast<uintptr_t>(dst);
    while (elem_bytes < 16 && p.inner % 2 == 0 && at % (2 * (uintptr_t)elem_bytes) == 0 && p.total > 0) {
        widen(p, 2);
        elem_bytes *= 2;
    }
    switch (elem_bytes) {
        case 1: return perm_launch<uint8_t>(src, dst, p, stream);
        case 2: return perm_launch<uint16_t>(src, dst, p, stream);
        case 4: return perm_launch<uint32_t>(src, dst, p, stream);
        case 8: return perm_launch<uint64_t>(src, dst, p, stream);
        case 16: return perm_launch<uint4>(src, dst, p, stream);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace tn
