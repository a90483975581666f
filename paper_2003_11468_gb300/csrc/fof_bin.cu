// Binning: a two-level counting sort of the particles into cells of side
// >= l_x (the paper matches tree-node size to the linking length for the
// neighbour search, Sec. 3.1; here the tree is a uniform periodic grid).
//
//   bin_count    validate every coordinate, histogram of bricks, and each
//                particle's rank in its brick (what the count's atomic returns)
//   scan         exclusive prefix sum of the brick counts
//   bin_scatter  each particle to its brick's start + rank (float4: x, y, z,
//                local index)
//   brick_sort   one CTA per brick (a cluster of eight for the few bricks
//                that hold many particles): cell histogram and scan in shared
//                memory, scatter into cell order, cell_start of the brick,
//                and the forest initialisation parent[s] = s (Sec. 3.1)
//
// Bricks exist so that both the counters' atomics and the scattered writes
// stay in L2: the brick count is small enough that every brick's write head
// is L2-resident, which turns the random-order scatter into full-sector DRAM
// writes.
#include <cooperative_groups.h>

#include "fof_internal.cuh"

namespace fofgpu {

namespace {

__device__ __forceinline__ unsigned lanemask_lt()
{
    unsigned m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

__device__ __forceinline__ bool coord_ok(float x, float xmax)
{
    return x >= 0.0f && x <= xmax;     // false for NaN
}

// brick of particle i (concatenated brick index) and its float4 record
__device__ __forceinline__ int64_t brick_of(const float* __restrict__ pos, int64_t i,
                                            const BoxDev& b, float4& rec, bool& ok)
{
    float x = __ldg(pos + 3 * i);
    float y = __ldg(pos + 3 * i + 1);
    float z = __ldg(pos + 3 * i + 2);
    ok = coord_ok(x, b.xmax) && coord_ok(y, b.xmax) && coord_ok(z, b.xmax);
    rec = make_float4(x, y, z, __int_as_float((int)(i - b.p0)));
    return b.brick0 + brick_local(b, cell_coord(x, b), cell_coord(y, b), cell_coord(z, b));
}

// One tile of particles per CTA in both kernels, not a stride over the input.
// CTAs start in order, so particles of neighbouring rank are stored at about
// the same time and a brick's sectors fill up while they are in L2; CTAs that
// stride over the input drift apart, and half-filled sectors leave L2 (768^3
// box, scatter by the count's ranks: 11.8 ms striding, 6.5 ms by tiles; 7.9 ms
// with a cursor atomic per particle instead).  The tiles of kBinStreams evenly
// spaced places of the input take turns: inputs list a blob's particles one
// after the other, and tiles of one place alone would all count into that
// blob's few bricks (a batch of 512 boxes: count 8.1 ms in input order, 2.5 ms
// with 64 places).
//
// The particle's rank in its brick (what the count's atomic returns) goes to
// rank[i], so that the scatter needs no atomic.  The counters lie `pad` words
// apart (brick_pad).
constexpr int kBinThreads = 256;
constexpr int kBinItems = 4;
constexpr int kBinTile = kBinThreads * kBinItems;
constexpr int kBinStreams = 64;

__host__ __device__ __forceinline__ int64_t bin_tiles_per_stream(int64_t n, int streams)
{
    return ((n + kBinTile - 1) / kBinTile + streams - 1) / streams;
}

// First particle of this CTA's tile (may lie past the end).
__device__ __forceinline__ int64_t bin_tile_base(int64_t n, int streams)
{
    return ((int64_t)(blockIdx.x % streams) * bin_tiles_per_stream(n, streams) + blockIdx.x / streams) * kBinTile;
}

__global__ void __launch_bounds__(kBinThreads) k_bin_count(const float* __restrict__ pos, Geometry g,
                                                           int* __restrict__ bcount, int pad,
                                                           int* __restrict__ rank, int streams,
                                                           int* __restrict__ err)
{
    pdl_trigger();
    const int lane = threadIdx.x & 31;
    const int64_t base = bin_tile_base(g.total_n, streams) + threadIdx.x;
    int bad = 0;
    int brick[kBinItems], off[kBinItems];
    unsigned peers[kBinItems];
    BoxCursor box;
#pragma unroll
    for (int k = 0; k < kBinItems; ++k) {
        const int64_t i = base + k * kBinThreads;
        const BoxDev& b = g.boxes[box.at(g.box_p0, g.nbox, i - lane, i, lane)];
        brick[k] = -1;
        if (i < g.total_n) {
            float4 rec;
            bool ok;
            brick[k] = (int)brick_of(pos, i, b, rec, ok);   // fits in 31 bits (checked when the plan is made)
            bad |= !ok;
        }
    }
#pragma unroll
    for (int k = 0; k < kBinItems; ++k) {
        peers[k] = __match_any_sync(kFull, brick[k]);
        off[k] = 0;
        if (lane == __ffs(peers[k]) - 1 && brick[k] >= 0)
            off[k] = atomicAdd(bcount + (int64_t)brick[k] * pad, __popc(peers[k]));
    }
#pragma unroll
    for (int k = 0; k < kBinItems; ++k) {
        const int first = __shfl_sync(kFull, off[k], __ffs(peers[k]) - 1);
        if (brick[k] >= 0)
            rank[base + k * kBinThreads] = first + __popc(peers[k] & lanemask_lt());
    }
    if (__syncthreads_or(bad) && threadIdx.x == 0)
        atomicOr(err, kErrRange);
}

// The same where all brick counters fit in shared memory: a CTA counts a tile
// of particles there and adds each brick's count to the global counter once.
// Few bricks mean many particles per counter: without the tile, every
// particle of a large blob in random order is an atomic on one address (about
// 1.7 ns each; 2 million particles in random order, one atomic each: 158 us,
// through the tile 30 us).
constexpr int kCountThreads = 1024;

template <int kItems>
__global__ void __launch_bounds__(kCountThreads) k_bin_count_tile(const float* __restrict__ pos, Geometry g,
                                                                  int* __restrict__ bcount, int pad,
                                                                  int* __restrict__ rank, int* __restrict__ err)
{
    extern __shared__ int tile_count[];                  // [total_bricks]: the tile's count, then its first rank
    pdl_trigger();
    const int lane = threadIdx.x & 31;
    const int nb = (int)g.total_bricks;
    const int64_t base = (int64_t)blockIdx.x * (kItems * kCountThreads) + threadIdx.x;
    int brick[kItems], local[kItems];
    int bad = 0;
    BoxCursor box;
#pragma unroll
    for (int k = 0; k < kItems; ++k) {
        const int64_t i = base + k * kCountThreads;
        const BoxDev& b = g.boxes[box.at(g.box_p0, g.nbox, i - lane, i, lane)];
        brick[k] = -1;
        if (i < g.total_n) {
            float4 rec;
            bool ok;
            brick[k] = (int)brick_of(pos, i, b, rec, ok);
            bad |= !ok;
        }
    }
    for (int b = threadIdx.x; b < nb; b += kCountThreads) tile_count[b] = 0;
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kItems; ++k) {
        const unsigned peers = __match_any_sync(kFull, brick[k]);
        const int leader = __ffs(peers) - 1;
        int off = 0;
        if (lane == leader && brick[k] >= 0)
            off = atomicAdd(tile_count + brick[k], __popc(peers));
        local[k] = __shfl_sync(kFull, off, leader) + __popc(peers & lanemask_lt());
    }
    __syncthreads();
    for (int b = threadIdx.x; b < nb; b += kCountThreads) {
        const int c = tile_count[b];
        if (c)
            tile_count[b] = atomicAdd(bcount + (int64_t)b * pad, c);
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kItems; ++k)
        if (brick[k] >= 0)
            rank[base + k * kCountThreads] = tile_count[brick[k]] + local[k];
    if (__syncthreads_or(bad) && threadIdx.x == 0)
        atomicOr(err, kErrRange);
}

__global__ void __launch_bounds__(kBinThreads) k_bin_scatter(const float* __restrict__ pos, Geometry g,
                                                             const int* bstart, const int* rank, int streams,
                                                             float4* __restrict__ tmp, int* __restrict__ err)
{
    pdl_wait();
    pdl_trigger();
    const int64_t base = bin_tile_base(g.total_n, streams) + threadIdx.x;
    float4 rec[kBinItems];
    int64_t brick[kBinItems];
    int r[kBinItems];
    const int lane = threadIdx.x & 31;
    BoxCursor box;
#pragma unroll
    for (int k = 0; k < kBinItems; ++k) {
        const int64_t i = base + k * kBinThreads;
        const BoxDev& b = g.boxes[box.at(g.box_p0, g.nbox, i - lane, i, lane)];
        brick[k] = -1;
        if (i < g.total_n) {
            bool ok;
            r[k] = rank[i];
            brick[k] = brick_of(pos, i, b, rec[k], ok);
        }
    }
#pragma unroll
    for (int k = 0; k < kBinItems; ++k) {
        if (brick[k] < 0)
            continue;
        const int64_t slot = (int64_t)bstart[brick[k]] + r[k];
        if (slot < bstart[brick[k] + 1])
            tmp[slot] = rec[k];
        else
            atomicOr(err, kErrInternal);
    }
}

// ------------------------------------------------------------------------
// device-wide exclusive scan of the brick counts, in one pass over the tiles
// (decoupled look-back)
// ------------------------------------------------------------------------

constexpr int kScanThreads = 256;
constexpr int kScanItems = 8;
constexpr int kScanTile = kScanThreads * kScanItems;   // 2048

__device__ __forceinline__ int block_exclusive_scan(int v, int* smem_warp, int& total)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int x = v;
    for (int o = 1; o < 32; o <<= 1) {
        int y = __shfl_up_sync(kFull, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) smem_warp[wid] = x;
    __syncthreads();
    if (wid == 0) {
        int nw = blockDim.x >> 5;
        int t = lane < nw ? smem_warp[lane] : 0;
        for (int o = 1; o < 32; o <<= 1) {
            int y = __shfl_up_sync(kFull, t, o);
            if (lane >= o) t += y;
        }
        if (lane < nw) smem_warp[lane] = t;   // inclusive warp totals
    }
    __syncthreads();
    int warp_off = wid ? smem_warp[wid - 1] : 0;
    total = smem_warp[(blockDim.x >> 5) - 1];
    __syncthreads();
    return warp_off + x - v;
}

// out[i] for i in [0, len]: out[len] is the grand total (a virtual zero is
// appended to the input, so the scan covers len + 1 entries).  The counts lie
// `pad` words apart.
// `heavy` (or null): entries above heavy_from are listed there.
__global__ void __launch_bounds__(kScanThreads) k_scan(const int* in, int pad, int* __restrict__ out,
                                                       int64_t len, unsigned long long* __restrict__ state,
                                                       int* __restrict__ ticket, int heavy_from,
                                                       int* __restrict__ heavy, int* __restrict__ n_heavy,
                                                       int* __restrict__ err)
{
    __shared__ int sw[32];
    __shared__ int s_tile, s_before;
    pdl_wait();
    pdl_trigger();
    if (threadIdx.x == 0)
        s_tile = atomicAdd(ticket, 1);
    __syncthreads();
    const int tile = s_tile;
    const int64_t base = (int64_t)tile * kScanTile + (int64_t)threadIdx.x * kScanItems;
    int v[kScanItems];
    int s = 0;
#pragma unroll
    for (int k = 0; k < kScanItems; ++k)
        v[k] = base + k < len ? in[(base + k) * pad] : 0;
#pragma unroll
    for (int k = 0; k < kScanItems; ++k) {
        s += v[k];
        if (heavy && v[k] > heavy_from)
            heavy[atomicAdd(n_heavy, 1)] = (int)(base + k);
    }
    int total;
    int ex = block_exclusive_scan(s, sw, total);
    if (threadIdx.x < kWarp) {
        const int before = lookback(state, tile, total, threadIdx.x, err);
        if (threadIdx.x == 0)
            s_before = before;
    }
    __syncthreads();
    ex += s_before;
#pragma unroll
    for (int k = 0; k < kScanItems; ++k) {
        if (base + k <= len) out[base + k] = ex;
        ex += v[k];
    }
}

// ------------------------------------------------------------------------
// per-brick cell sort
// ------------------------------------------------------------------------

constexpr int kMaxR3 = 4096;   // r <= 16

struct CellLists {
    int64_t* list[4];          // dense cells, team cells (small), big cells, team cells (from the back end)
    int* n[4];
    int64_t team_cap;
};

// which list a cell of h particles belongs to: 0 dense, 1 small team, 2 big,
// 3 large team, -1 none
__device__ __forceinline__ int cell_list(int h, const BoxDev& b, int dense_min)
{
    if (is_big(h, b))
        return 2;
    if (is_sub(h, b, dense_min))
        return 0;
    if (h < b.team_min || h > kTeamSelfMax)
        return -1;
    return h <= kTeamSplit ? 1 : 3;
}

__device__ __forceinline__ int* list_counter(const CellLists& L, int l)
{
    return l == 0 ? L.n[0] : (l == 1 ? L.n[1] : (l == 2 ? L.n[2] : L.n[3]));
}

// A brick's listed cells are counted as four 16-bit fields of one word (at most
// kMaxR3 cells per brick).
__device__ __forceinline__ unsigned long long list_one(int l)
{
    return l < 0 ? 0ull : 1ull << (16 * l);
}

// The cell `key` of h particles from slot `start` on, as entry `at` (past the
// brick's base) of its list.
__device__ __forceinline__ void list_cell(const CellLists& L, const int* list_base, int l, int at, int h, int64_t key,
                                          int start)
{
    const int64_t pos = list_base[l] + at;
    if (l == 0)
        L.list[0][pos] = key;
    else if (l == 2)
        L.list[2][pos] = key;
    else
        L.list[1][l == 1 ? pos : L.team_cap - 1 - pos] = ((int64_t)h << 32) | (uint32_t)start;
}

// What the cell code of a particle inside its brick needs of its box (in
// registers: the box table would be read again after every store).
struct CodeGeo {
    float inv_hf;
    int nf, q, rmask;
    uint32_t magic_q;
};

__device__ __forceinline__ CodeGeo code_geo(const BoxDev& b)
{
    return CodeGeo{b.inv_hf, b.nf, b.q, b.r - 1, b.magic_q};
}

__device__ __forceinline__ int code_axis(float x, const CodeGeo& c)
{
    int g = (int)__fmul_rn(x, c.inv_hf);       // cell_coord
    g = min(max(g, 0), c.nf - 1);
    return (c.q == 1 ? g : (int)__umulhi((unsigned)g, c.magic_q)) & c.rmask;
}

__device__ __forceinline__ int code_of(const float4& p, const CodeGeo& c)
{
    return (int)local_code(code_axis(p.x, c), code_axis(p.y, c), code_axis(p.z, c));
}

// One CTA per brick of up to heavy_from particles.  A mean brick has 1,200
// particles in 4,096 cells, most of them empty, and what bounds it is the
// chain: load, histogram, scan, cursors, scatter.  So
//   * the next brick's records are copied ahead into shared memory (cp.async)
//     while this one is sorted;
//   * the sort goes through the list of each slot's source, so that the four
//     words of a slot are stored in slot order, as whole lines: stored from the
//     particles' side they were 2.7 sectors a particle, which an SM writes at
//     about two cycles each, two thirds of the kernel's time;
//   * counts and cursors are 16-bit halves of shared-memory words, eight cells
//     to a load, so two histograms fit and take turns (the one not in use is
//     cleared meanwhile) and a brick takes three barriers;
//   * the lists are looked at only in bricks that hold a cell for one, and
//     their reservations return while the scatter runs.
// Warp w owns the cells of per_warp consecutive groups of eight, lane by lane,
// so the histogram is read and written conflict-free; a lane's groups share one
// warp scan as 16-bit fields.  Registers are what limits the copies and loads
// in flight: this kernel has no spill, and the forms that had took 10 to 50% longer.  Both sort kernels, before (1,024
// threads, 32-bit counts, twelve barriers) and after, us: 4 million particles
// (two steps) 537 and 254, 8 million 360 and 216, 512 boxes of 650,000 12850 and
// 7500, 453 million (768^3) 12200 and 8990.
constexpr int kSortThreads = 256;
constexpr int kSortWarps = kSortThreads / 32;
constexpr int kSortBlocks = 4;
constexpr int kSortKeep = 2;                           // records of a brick copied ahead per thread
constexpr int kFlight = 2;                             // loads in flight per thread beyond them
constexpr int kSortGroups = kMaxR3 / (8 * kSortThreads);   // groups of eight cells per lane
static_assert(kSortGroups <= 4 && kBrickMax < 65536, "16-bit counts, four fields");

struct SortSmem {
    float4 rec[2][kSortKeep * kSortThreads];
    unsigned short source[kHeavyBrick];        // record that goes to each slot of the brick
    unsigned hist[2][kMaxR3 / 2];
    int part[kSortWarps];
    unsigned long long list_pack;
    int list_base[4];
};

// +1 on cell c's 16-bit half; returns its value before
__device__ __forceinline__ int bump(unsigned* hist, int c)
{
    const int sh = (c & 1) * 16;
    return (int)((atomicAdd(hist + (c >> 1), 1u << sh) >> sh) & 0xffffu);
}

__device__ __forceinline__ int half_of(const unsigned* hist, int c)
{
    return (int)((hist[c >> 1] >> ((c & 1) * 16)) & 0xffffu);
}

__global__ void __launch_bounds__(kSortThreads, kSortBlocks)
    k_brick_sort(Geometry g, const float4* tmp, const int* bstart,
                 float4* __restrict__ sorted, int* __restrict__ parent, int* __restrict__ minorig,
                 int* __restrict__ cnt, int* __restrict__ cell_start, int dense_min, CellLists lists,
                 int heavy_from, const unsigned* beside, int* __restrict__ err)
{
    // beside k_brick_sort_heavy where that runs just before (it needs nothing
    // of it), else after the scatter
    if (beside)
        pdl_join(beside);
    else
        pdl_wait();
    pdl_trigger();
    extern __shared__ float4 sort_raw[];
    SortSmem& S = *reinterpret_cast<SortSmem*>(sort_raw);
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    for (int c = tid; c < kMaxR3; c += kSortThreads) S.hist[0][c] = 0u;     // both
    if (tid == 0)
        S.list_pack = 0ull;
    __syncthreads();
    const int64_t nb = g.total_bricks, stride = gridDim.x;
    auto fetch = [&](int s0, int s1, int buf) {                // one commit group
        if (s1 - s0 <= heavy_from) {
#pragma unroll
            for (int i = 0; i < kSortKeep; ++i) {
                const int k = i * kSortThreads + tid;
                if (slot_before(s0, k, s1))
                    cp_async16(&S.rec[buf][k], tmp + s0 + k);
            }
        }
        cp_async_commit();
    };
    int64_t gb = blockIdx.x;
    int s0 = 0, s1 = 0, n0 = 0, n1 = 0;                        // this brick's and the next one's slots
    if (gb < nb) {
        s0 = bstart[gb];
        s1 = bstart[gb + 1];
    }
    if (gb + stride < nb) {
        n0 = bstart[gb + stride];
        n1 = bstart[gb + stride + 1];
    }
    fetch(s0, s1, 0);
    int bi = 0, buf = 0, hb = 0;               // record buffer and histogram of this brick
    for (; gb < nb; gb += stride, buf ^= 1) {
        cp_async_wait_all();
        const int a0 = s0, a1 = s1;
        s0 = n0;
        s1 = n1;
        if (gb + 2 * stride < nb) {
            n0 = bstart[gb + 2 * stride];
            n1 = bstart[gb + 2 * stride + 1];
        } else {
            n0 = n1 = 0;
        }
        const float4* rec = S.rec[buf];
        unsigned* hist = S.hist[hb];
        if (a1 - a0 > heavy_from) {            // k_brick_sort_heavy's (block-uniform)
            __syncthreads();                   // the last brick's records have been read
            fetch(s0, s1, buf ^ 1);
            continue;
        }
        // the next box, one of the 32 from it, or by search (box by box a million
        // boxes of one brick took 89 ms, so 5.9; by search alone 64 boxes of 2 million
        // particles took 3 us longer)
        if (bi + 1 < g.nbox && g.box_brick0[bi + 1] <= gb) {
            const unsigned past = __ballot_sync(kFull, bi + 1 + lane < g.nbox && g.box_brick0[bi + 1 + lane] <= gb);
            bi = past == kFull ? box_of_warp(g.box_brick0, g.nbox, gb, lane) : bi + __popc(past);
        }
        const BoxDev& b = g.boxes[bi];
        const CodeGeo cg = code_geo(b);
        const int n = a1 - a0, r3 = (cg.rmask + 1) * (cg.rmask + 1) * (cg.rmask + 1);
        int code[kSortKeep];
#pragma unroll
        for (int i = 0; i < kSortKeep; ++i) {
            const int k = i * kSortThreads + tid;
            if (k < n) {
                code[i] = code_of(rec[k], cg);
                bump(hist, code[i]);
            }
        }
        for (int kb = kSortKeep * kSortThreads + tid; kb < n; kb += kFlight * kSortThreads) {
            float4 v[kFlight];
#pragma unroll
            for (int i = 0; i < kFlight; ++i)
                if (kb + i * kSortThreads < n)
                    v[i] = tmp[a0 + kb + i * kSortThreads];
#pragma unroll
            for (int i = 0; i < kFlight; ++i)
                if (kb + i * kSortThreads < n)
                    bump(hist, code_of(v[i], cg));
        }
        __syncthreads();
        // every thread has finished the previous brick: its record buffer takes
        // the next one's
        fetch(s0, s1, buf ^ 1);
        // and its histogram is cleared for it
        for (int q = tid; q < kMaxR3 / 8; q += kSortThreads)
            reinterpret_cast<uint4*>(S.hist[hb ^ 1])[q] = make_uint4(0u, 0u, 0u, 0u);
        hb ^= 1;
        const int octs = (r3 + 7) / 8, per_warp = (octs + kSortWarps - 1) / kSortWarps;
        const int q0 = wid * per_warp, q1 = min(q0 + per_warp, octs);
        const int listed_from = min(min(b.team_min, dense_min), kDenseMax + 1);
        unsigned long long sums = 0ull;        // 16-bit field i: particles of this lane's group i
        unsigned most = 0u;                    // largest count, in either half
#pragma unroll
        for (int i = 0; i < kSortGroups; ++i) {
            const int q = q0 + i * 32 + lane;
            const uint4 h = q < q1 ? reinterpret_cast<const uint4*>(hist)[q] : make_uint4(0u, 0u, 0u, 0u);
            const unsigned t = h.x + h.y + h.z + h.w;                  // halves add up without a carry
            sums |= (unsigned long long)((t & 0xffffu) + (t >> 16)) << (16 * i);
            most = __vmaxu2(most, __vmaxu2(__vmaxu2(h.x, h.y), __vmaxu2(h.z, h.w)));
        }
        unsigned long long inc = sums;
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long y = __shfl_up_sync(kFull, inc, o);
            if (lane >= o) inc += y;
        }
        const unsigned long long all = __shfl_sync(kFull, inc, 31);
        if (lane == 0)
            S.part[wid] = (int)((all & 0xffffu) + ((all >> 16) & 0xffffu) + ((all >> 32) & 0xffffu) + (all >> 48));
        const bool listed = __syncthreads_or((int)max(most & 0xffffu, most >> 16) >= listed_from);
        const int64_t cbase = b.cell0 + (gb - b.brick0) * (int64_t)r3;
        unsigned full = 0u;                    // this lane's groups with a listed cell
        unsigned long long list_at = 0ull;     // this thread's entries of each list start there
        {
            // particles in the groups before
            int base = (int)__reduce_add_sync(kFull, lane < wid ? (unsigned)S.part[lane] : 0u);
            unsigned long long mine = 0ull;    // listed cells of this thread
            unsigned long long before = inc - sums;
#pragma unroll 1
            for (int i = 0; i < kSortGroups; ++i) {
                const int q = q0 + i * 32 + lane;
                if (q < q1) {
                    uint4* cells = reinterpret_cast<uint4*>(hist) + q;
                    const uint4 h = *cells;
                    int x = base + (int)(before & 0xffffu);
                    // a half-word pair of counts becomes the pair of its cursors
                    auto cursors = [&](unsigned w) {
                        const int lo = x, hi = x + (int)(w & 0xffffu);
                        x = hi + (int)(w >> 16);
                        return make_int2(lo, hi);
                    };
                    const int2 p0 = cursors(h.x), p1 = cursors(h.y), p2 = cursors(h.z), p3 = cursors(h.w);
                    *cells = make_uint4((unsigned)(p0.x | (p0.y << 16)), (unsigned)(p1.x | (p1.y << 16)),
                                        (unsigned)(p2.x | (p2.y << 16)), (unsigned)(p3.x | (p3.y << 16)));
                    int* out = cell_start + cbase + 8 * q;
                    if (8 * q + 8 <= r3 && (cbase & 3) == 0) {
                        reinterpret_cast<int4*>(out)[0] = make_int4(a0 + p0.x, a0 + p0.y, a0 + p1.x, a0 + p1.y);
                        reinterpret_cast<int4*>(out)[1] = make_int4(a0 + p2.x, a0 + p2.y, a0 + p3.x, a0 + p3.y);
                    } else {                   // bricks of fewer than 8 cells, or after one
                        for (int u = 0; u < 8 && 8 * q + u < r3; ++u) out[u] = a0 + half_of(hist, 8 * q + u);
                    }
                    const unsigned top = __vmaxu2(__vmaxu2(h.x, h.y), __vmaxu2(h.z, h.w));
                    if ((int)max(top & 0xffffu, top >> 16) >= listed_from) {
                        full |= 1u << i;
                        auto listed_pair = [&](unsigned w) {
                            mine += list_one(cell_list((int)(w & 0xffffu), b, dense_min)) +
                                    list_one(cell_list((int)(w >> 16), b, dense_min));
                        };
                        listed_pair(h.x);
                        listed_pair(h.y);
                        listed_pair(h.z);
                        listed_pair(h.w);
                    }
                }
                base += (int)((all >> (16 * i)) & 0xffffu);
                before >>= 16;
            }
            // the end of the last cell (the next brick writes the same value)
            if (tid == 0)
                cell_start[cbase + r3] = a1;
            if (mine)
                list_at = atomicAdd(&S.list_pack, mine);
        }
        __syncthreads();
        // one reservation per list and brick (a shared counter per cell would
        // serialise millions of atomics on one address); it returns meanwhile
        int reserved = 0;
        if (listed && tid < 4) {
            const int cells = (int)((S.list_pack >> (16 * tid)) & 0xffffu);
            if (cells)
                reserved = atomicAdd(list_counter(lists, tid), cells);
        }
        if (n <= kHeavyBrick) {
            // each slot's source, then all of the slot's words in slot order:
            // the stores are whole lines
#pragma unroll
            for (int i = 0; i < kSortKeep; ++i) {
                const int k = i * kSortThreads + tid;
                if (k < n)
                    S.source[bump(hist, code[i])] = (unsigned short)k;
            }
            for (int kb = kSortKeep * kSortThreads + tid; kb < n; kb += kFlight * kSortThreads) {
                float4 v[kFlight];
#pragma unroll
                for (int i = 0; i < kFlight; ++i)
                    if (kb + i * kSortThreads < n)
                        v[i] = tmp[a0 + kb + i * kSortThreads];
#pragma unroll
                for (int i = 0; i < kFlight; ++i)
                    if (kb + i * kSortThreads < n) {
                        const int at = bump(hist, code_of(v[i], cg));
                        if (at < n)
                            S.source[at] = (unsigned short)(kb + i * kSortThreads);
                        else
                            atomicOr(err, kErrInternal);
                    }
            }
            __syncthreads();
            for (int t = tid; t < n; t += kSortThreads) {
                const int k = min((int)S.source[t], n - 1);
                const float4 v = k < kSortKeep * kSortThreads ? rec[k] : tmp[a0 + k];
                sorted[a0 + t] = v;
                minorig[a0 + t] = __float_as_int(v.w);
                parent[a0 + t] = a0 + t;
                cnt[a0 + t] = 1;
            }
        } else {
            for (int k = tid; k < n; k += kSortThreads) {
                const float4 v = k < kSortKeep * kSortThreads ? rec[k] : tmp[a0 + k];
                const int slot = a0 + bump(hist, code_of(v, cg));
                if (slot < a1) {
                    sorted[slot] = v;
                    minorig[slot] = __float_as_int(v.w);
                } else {
                    atomicOr(err, kErrInternal);
                }
                parent[a0 + k] = a0 + k;
                cnt[a0 + k] = 1;
            }
        }
        if (listed) {
            if (tid < 4)
                S.list_base[tid] = reserved;
            __syncthreads();
            if (tid == 0)
                S.list_pack = 0ull;
            // the cursors now hold each cell's end
            for (; full; full &= full - 1u) {
                const int c0 = 8 * (q0 + (__ffs(full) - 1) * 32 + lane);
                int start = c0 ? half_of(hist, c0 - 1) : 0;
                for (int c = c0; c < c0 + 8; ++c) {
                    const int end = half_of(hist, c), size = end - start;
                    const int l = c < r3 ? cell_list(size, b, dense_min) : -1;
                    if (l >= 0) {
                        list_cell(lists, S.list_base, l, (int)((list_at >> (16 * l)) & 0xffffu), size, cbase + c,
                                  a0 + start);
                        list_at += list_one(l);
                    }
                    start = end;
                }
            }
        }
    }
    cp_async_wait_all();
    if (beside)
        pdl_wait();
}

// Bricks above kHeavyBrick particles: a cluster of CTAs per brick, each CTA
// with its share of the particles and its own histogram; CTA r also owns an
// equal share of the cells, whose counts it sums over the cluster through
// distributed shared memory and turns into every CTA's cursors.  One CTA of
// 1,024 threads took 570 us for the fullest brick of the 256^3 box (350,000
// particles); the 150 bricks above kHeavyBrick together take 154 us here (260
// with 1,024 threads per CTA, of which fewer clusters run at a time; 768^3 box,
// fixed shares of the bricks against tickets: 4.48 and 2.88 ms).  At two CTAs of
// 64 registers per SM it spills 32 bytes a thread.
constexpr int kCluster = 8;
constexpr int kHeavyThreads = 512;
constexpr int kHeavyBlocks = 2;
constexpr int kHeavyFlight = 4;                 // loads in flight per thread
static_assert(kMaxR3 / kCluster <= kHeavyThreads, "one cell per thread");

__global__ void __cluster_dims__(kCluster, 1, 1) __launch_bounds__(kHeavyThreads, kHeavyBlocks)
    k_brick_sort_heavy(Geometry g, const float4* __restrict__ tmp, const int* bstart, const int* heavy,
                       const int* n_heavy, int* __restrict__ ticket, float4* __restrict__ sorted,
                       int* __restrict__ parent, int* __restrict__ minorig, int* __restrict__ cnt,
                       int* __restrict__ cell_start, int dense_min, CellLists lists, unsigned* pass_on,
                       int* __restrict__ err)
{
    pdl_wait();
    pdl_pass_on(pass_on);
    namespace cg = cooperative_groups;
    __shared__ int hist[kMaxR3];
    __shared__ int part[kWarp];
    __shared__ unsigned long long list_pack;
    __shared__ int list_base[4];
    __shared__ int cells_total;                    // particles in this CTA's cells
    __shared__ int next_item;                      // rank 0's: the cluster's next brick
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = (int)cluster.block_rank();
    const int n = *n_heavy;
    // a cluster's first brick by its number, the others by ticket: the fullest
    // brick of a box can hold a third of what all of them hold
    int next = 0;
    for (int it = blockIdx.x / kCluster; it < n; it = next) {
        int drawn = 0;
        if (rank == 0 && threadIdx.x == 0)
            drawn = atomicAdd(ticket, 1);
        const int64_t gb = heavy[it];
        const int s0 = bstart[gb], s1 = bstart[gb + 1];
        const BoxDev& b = g.boxes[box_of_warp(g.box_brick0, g.nbox, gb, threadIdx.x & 31)];
        const CodeGeo geo = code_geo(b);
        const int r3 = b.r * b.r * b.r;
        for (int c = threadIdx.x; c < r3; c += kHeavyThreads) hist[c] = 0;
        __syncthreads();
        // this CTA's particles
        const SlotRange own_slots = slot_share(s0, s1 - s0, rank, kCluster);
        const int k0 = own_slots.first, kn = own_slots.count;
        for (int kb = threadIdx.x; kb < kn; kb += kHeavyFlight * kHeavyThreads) {
            float4 v[kHeavyFlight];
#pragma unroll
            for (int i = 0; i < kHeavyFlight; ++i)
                if (kb + i * kHeavyThreads < kn)
                    v[i] = tmp[k0 + kb + i * kHeavyThreads];
#pragma unroll
            for (int i = 0; i < kHeavyFlight; ++i)
                if (kb + i * kHeavyThreads < kn)
                    atomicAdd(hist + code_of(v[i], geo), 1);
        }
        cluster.sync();
        // this CTA's cells, one per thread: the cluster's counts and each
        // CTA's offset in the cell
        const int own = (r3 + kCluster - 1) / kCluster;
        const int c = rank * own + threadIdx.x;
        const bool mine = (int)threadIdx.x < own && c < r3;
        int before[kCluster], h = 0;
#pragma unroll
        for (int q = 0; q < kCluster; ++q) {
            before[q] = h;
            if (mine)
                h += *cluster.map_shared_rank(hist + c, q);
        }
        if (threadIdx.x == 0)
            list_pack = 0ull;
        int total;
        const int ex = block_exclusive_scan(h, part, total);
        const int l = mine ? cell_list(h, b, dense_min) : -1;
        unsigned long long at = 0ull;
        if (l >= 0)
            at = atomicAdd(&list_pack, list_one(l));
        if (threadIdx.x == 0) {
            cells_total = total;
            if (rank == 0)
                next_item = (int)(gridDim.x / kCluster) + drawn;
        }
        cluster.sync();
        next = *cluster.map_shared_rank(&next_item, 0);
        int start = s0 + ex;
        for (int q = 0; q < rank; ++q)
            start += *cluster.map_shared_rank(&cells_total, q);
        const int64_t cbase = b.cell0 + (gb - b.brick0) * (int64_t)r3;
        if (mine) {
#pragma unroll
            for (int q = 0; q < kCluster; ++q)
                *cluster.map_shared_rank(hist + c, q) = start + before[q];
            cell_start[cbase + c + 1] = start + h;
            if (c == 0)
                cell_start[cbase] = s0;
        }
        int reserved = 0;
        if (threadIdx.x < 4) {
            const int cells = (int)((list_pack >> (16 * threadIdx.x)) & 0xffffu);
            if (cells)
                reserved = atomicAdd(list_counter(lists, threadIdx.x), cells);
        }
        cluster.sync();
        for (int kb = threadIdx.x; kb < kn; kb += kHeavyFlight * kHeavyThreads) {
            float4 v[kHeavyFlight];
#pragma unroll
            for (int i = 0; i < kHeavyFlight; ++i)
                if (kb + i * kHeavyThreads < kn)
                    v[i] = tmp[k0 + kb + i * kHeavyThreads];
#pragma unroll
            for (int i = 0; i < kHeavyFlight; ++i) {
                if (kb + i * kHeavyThreads < kn) {
                    const int k = k0 + kb + i * kHeavyThreads;
                    const int slot = atomicAdd(hist + code_of(v[i], geo), 1);
                    if (slot < s1) {
                        sorted[slot] = v[i];
                        minorig[slot] = __float_as_int(v[i].w);
                    } else {
                        atomicOr(err, kErrInternal);
                    }
                    parent[k] = k;
                    cnt[k] = 1;
                }
            }
        }
        // after the last cluster barrier no other CTA touches this one's memory
        if (threadIdx.x < 4)
            list_base[threadIdx.x] = reserved;
        __syncthreads();
        if (l >= 0)
            list_cell(lists, list_base, l, (int)((at >> (16 * l)) & 0xffffu), h, cbase + c, start);
    }
}

// ------------------------------------------------------------------------
// incremental re-binning (the group finder run again on moved particles)
// ------------------------------------------------------------------------

// For every binned slot s of the previous run: the particle's new position
// (pos[p0 + local index]) replaces its old one in sorted[s] and tmp[s], and
// flags record whether it left its cell (bit 0) or its brick (bit 1).  When
// no particle left its brick, the slots are still grouped by brick, so
// tmp[] is a valid brick-order array for k_brick_sort; when no particle left
// its cell, sorted[] and the cell starts and lists are valid as they are.
__global__ void __launch_bounds__(256) k_relink_check(const float* __restrict__ pos, Geometry g,
                                                      float4* __restrict__ sorted, float4* __restrict__ tmp,
                                                      int* __restrict__ flags, int* __restrict__ err)
{
    pdl_trigger();
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    int f = 0, bad = 0;
    for (int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; s < g.total_n; s += stride) {
        const BoxDev& b = g.boxes[box_of(g.box_p0, g.nbox, s)];
        const float4 old = sorted[s];
        const int o = __float_as_int(old.w);
        // a record that binning never wrote names no particle: bin again
        const bool named = (unsigned long long)o < (unsigned long long)b.n;
        const int64_t i = b.p0 + (named ? o : 0);
        float4 rec;
        bool ok;
        const int64_t nb = brick_of(pos, i, b, rec, ok);
        bad |= !ok;
        const int ox = cell_coord(old.x, b), oy = cell_coord(old.y, b), oz = cell_coord(old.z, b);
        const int nx = cell_coord(rec.x, b), ny = cell_coord(rec.y, b), nz = cell_coord(rec.z, b);
        if (nx != ox || ny != oy || nz != oz)
            f |= 1;
        if (!named || nb != b.brick0 + brick_local(b, ox, oy, oz))
            f |= 2;
        sorted[s] = rec;
        tmp[s] = rec;
    }
    f = __reduce_or_sync(kFull, f);
    if ((threadIdx.x & 31) == 0 && f)
        atomicOr(flags, f);
    if (__syncthreads_or(bad) && threadIdx.x == 0)
        atomicOr(err, kErrRange);
}

// Forest and label initialisation of the binned slots (what k_brick_sort
// does while it sorts): parent[s] = s, cnt[s] = 1, minorig[s] = local index.
__global__ void __launch_bounds__(256) k_forest_init(int64_t total, const float4* sorted,
                                                     int* __restrict__ parent, int* __restrict__ minorig,
                                                     int* __restrict__ cnt)
{
    pdl_wait();
    pdl_trigger();
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; s < total; s += stride) {
        parent[s] = (int)s;
        cnt[s] = 1;
        minorig[s] = __float_as_int(sorted[s].w);
    }
}

}  // namespace

// ------------------------------------------------------------------------
// launchers
// ------------------------------------------------------------------------

static int grid_for(int64_t items, int threads, int per_sm)
{
    int64_t want = (items + threads - 1) / threads;
    int64_t cap = (int64_t)sm_count() * per_sm;
    if (want < 1) want = 1;
    return (int)(want < cap ? want : cap);
}

// Words between brick counters: L2 serialises atomics on one 128-byte line
// (about 1.7 ns each), so counters that many particles share get a line or a
// sector of their own while that costs at most 4 MB.
int brick_pad(int64_t bricks)
{
    return bricks <= kTileBricks ? 32 : (bricks <= 131072 ? 8 : 1);
}

// Small problems count in shared-memory tiles: they spend the launch either
// way, and it bounds what a blob in random order costs.  Above, the padded
// counters and the turns of k_bin_count take less, in every order of the input
// (tiles and k_bin_count, us: 2 million in random order 39 and 54; 8 million
// blob by blob 110 and 65, in random order 138 and 132; 16.8 million 221 and 120,
// 292 and 216, in cell order 132 and 73).
static bool count_by_tile(const Geometry& g)
{
    return g.total_bricks <= kTileBricks && g.total_n <= 1 << 22;
}

template <int kItems>
static cudaError_t run_count_tile(const float* pos, const Geometry& g, const Work& w, cudaStream_t s)
{
    const int64_t tile = (int64_t)kItems * kCountThreads;
    k_bin_count_tile<kItems><<<(unsigned)((g.total_n + tile - 1) / tile), kCountThreads,
                               sizeof(int) * (size_t)g.total_bricks, s>>>(
        pos, g, w.bcount, brick_pad(g.total_bricks), w.parent, &w.status->err);
    return cudaGetLastError();
}

cudaError_t launch_bin_count(const float* pos, const Geometry& g, const Work& w, cudaStream_t s)
{
    if (g.total_n == 0)
        return cudaSuccess;
    // the forest is not in use yet: its array holds the ranks
    if (count_by_tile(g)) {
        // few particles per thread while that would leave SMs without a tile
        if (g.total_n <= (int64_t)sm_count() * kCountThreads)
            return run_count_tile<1>(pos, g, w, s);
        if (g.total_n <= (int64_t)sm_count() * kCountThreads * 8)
            return run_count_tile<4>(pos, g, w, s);
        return run_count_tile<8>(pos, g, w, s);
    }
    k_bin_count<<<(unsigned)(bin_tiles_per_stream(g.total_n, kBinStreams) * kBinStreams), kBinThreads, 0, s>>>(
        pos, g, w.bcount, brick_pad(g.total_bricks), w.parent, kBinStreams, &w.status->err);
    return cudaGetLastError();
}

int64_t scan_tiles(int64_t len)
{
    return (len + 1 + kScanTile - 1) / kScanTile;          // len + 1 outputs
}

cudaError_t launch_scan(int64_t n, const int* in, int pad, int* out, int64_t len, unsigned long long* state,
                        int* ticket, int heavy_from, int* heavy, int* n_heavy, int* err, cudaStream_t s)
{
    return launch_next(n, k_scan, scan_tiles(len), kScanThreads, 0, s, in, pad, out, len, state, ticket, heavy_from,
                       heavy, n_heavy, err);
}

cudaError_t launch_bin_scatter(const float* pos, const Geometry& g, const Work& w, cudaStream_t s)
{
    if (g.total_n == 0)
        return cudaSuccess;
    // in the order in which the ranks were given out
    const int streams = count_by_tile(g) ? 1 : kBinStreams;
    return launch_next(g.total_n, k_bin_scatter, bin_tiles_per_stream(g.total_n, streams) * streams, kBinThreads, 0, s,
                       pos, g, w.bstart, w.parent, streams, w.tmp, &w.status->err);
}

cudaError_t launch_brick_sort(const Geometry& g, const Work& w, int dense_min, cudaStream_t s)
{
    if (g.total_bricks == 0)
        return cudaSuccess;
    const CellLists lists = {{w.dense_list, w.team_list, w.big_list, w.team_list},
                             {w.n_dense, w.n_team, w.n_big, w.n_team_hi},
                             w.team_cap};
    if (heavy_bricks(g.total_n)) {
        int64_t clusters = g.total_n / kHeavyBrick;
        // twice the resident clusters: the others take over while the last bricks
        // of the first end, and k_brick_sort has the rest (both kernels, with 1
        // and 2 times, 8 million particles: 219 and 209 us, 16.8 million 421 and
        // 404; with half as many 234 and 474)
        const int64_t most = (int64_t)sm_count() * 2 * kHeavyBlocks / kCluster;
        if (clusters > most) clusters = most;
        cudaError_t e = launch_next(g.total_n, k_brick_sort_heavy, clusters * kCluster, kHeavyThreads, 0, s, g, w.tmp,
                                    w.bstart, w.heavy_list, w.n_heavy, w.heavy_ticket, w.sorted, w.parent, w.minorig,
                                    w.cnt, w.cell_start, dense_min, lists, w.status->passed_on + kPassBrickOrder,
                                    &w.status->err);
        if (e != cudaSuccess) return e;
    }
    // the shared-memory opt-in is per device; setting it again is harmless
    static bool configured[64] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64 || !configured[dev]) {
        e = cudaFuncSetAttribute(k_brick_sort, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(SortSmem));
        if (e != cudaSuccess) return e;
        if (dev >= 0 && dev < 64) configured[dev] = true;
    }
    int64_t blocks = g.total_bricks;
    int64_t cap = (int64_t)sm_count() * kSortBlocks;
    if (blocks > cap) blocks = cap;
    const bool beside = heavy_bricks(g.total_n);
    return launch_kernel(g.total_n <= (beside ? kBesideMax : kDependentMax), k_brick_sort, blocks, kSortThreads,
                         sizeof(SortSmem), s, g, w.tmp, w.bstart, w.sorted, w.parent, w.minorig, w.cnt, w.cell_start,
                         dense_min, lists, heavy_from(g.total_n),
                         beside ? w.status->passed_on + kPassBrickOrder : (unsigned*)nullptr, &w.status->err);
}

// Bricks above this many particles go to k_brick_sort_heavy: the limit of the
// 16-bit counts while a plan's particles all fit them (no brick can be above,
// and the launch is saved), else the size from which one CTA's chain is the
// longer one.
int heavy_from(int64_t total_n)
{
    return total_n <= kBrickMax ? kBrickMax : kHeavyBrick;
}

bool heavy_bricks(int64_t total_n)
{
    return total_n > kBrickMax;
}

cudaError_t launch_relink_check(const float* pos, const Geometry& g, const Work& w, int* flags,
                                cudaStream_t s)
{
    if (g.total_n == 0)
        return cudaSuccess;
    k_relink_check<<<grid_for(g.total_n, 256, 8), 256, 0, s>>>(pos, g, w.sorted, w.tmp, flags,
                                                             &w.status->err);
    return cudaGetLastError();
}

cudaError_t launch_forest_init(const Geometry& g, const Work& w, cudaStream_t s)
{
    if (g.total_n == 0)
        return cudaSuccess;
    return launch_next(g.total_n, k_forest_init, grid_for(g.total_n, 256, 8), 256, 0, s, g.total_n, w.sorted, w.parent,
                       w.minorig, w.cnt);
}

}  // namespace fofgpu
