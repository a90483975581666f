// Binning: a two-level counting sort of the particles into cells of side
// >= l_x (the paper matches tree-node size to the linking length for the
// neighbour search, Sec. 3.1; here the tree is a uniform periodic grid).
//
//   bin_count    validate every coordinate, histogram of bricks, and each
//                particle's rank in its brick (what the count's atomic returns)
//   scan         exclusive prefix sum of the brick counts
//   bin_scatter  each particle to its brick's start + rank (float4: x, y, z,
//                local index)
//   brick_sort   one CTA per brick: cell histogram and scan in shared
//                memory, scatter into cell order, cell_start of the brick,
//                and the forest initialisation parent[s] = s (Sec. 3.1)
//
// Bricks exist so that both atomics (brick cursors) and the scattered
// writes stay in L2: the brick count is small enough that every brick's
// write head is L2-resident, which turns the random-order scatter into
// full-sector DRAM writes.
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
// with a cursor atomic per particle instead).  The tiles of kBinStreams evenly spaced places of the input
// take turns: inputs list a blob's particles one after the other, and tiles of
// one place alone would all count into that blob's few bricks (a batch of 512
// boxes: count 8.1 ms in input order, 2.5 ms with 64 places).
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
    const int lane = threadIdx.x & 31;
    const int64_t base = bin_tile_base(g.total_n, streams) + threadIdx.x;
    int bad = 0;
    int brick[kBinItems], off[kBinItems];
    unsigned peers[kBinItems];
#pragma unroll
    for (int k = 0; k < kBinItems; ++k) {
        const int64_t i = base + k * kBinThreads;
        brick[k] = -1;
        if (i < g.total_n) {
            const BoxDev& b = g.boxes[box_of(g.box_p0, g.nbox, i)];
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
    const int lane = threadIdx.x & 31;
    const int nb = (int)g.total_bricks;
    const int64_t base = (int64_t)blockIdx.x * (kItems * kCountThreads) + threadIdx.x;
    int brick[kItems], local[kItems];
    int bad = 0;
#pragma unroll
    for (int k = 0; k < kItems; ++k) {
        const int64_t i = base + k * kCountThreads;
        brick[k] = -1;
        if (i < g.total_n) {
            const BoxDev& b = g.boxes[box_of(g.box_p0, g.nbox, i)];
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
                                                             const int* __restrict__ bstart,
                                                             const int* __restrict__ rank, int streams,
                                                             float4* __restrict__ tmp, int* __restrict__ err)
{
    const int64_t base = bin_tile_base(g.total_n, streams) + threadIdx.x;
    float4 rec[kBinItems];
    int64_t brick[kBinItems];
    int r[kBinItems];
#pragma unroll
    for (int k = 0; k < kBinItems; ++k) {
        const int64_t i = base + k * kBinThreads;
        brick[k] = -1;
        if (i < g.total_n) {
            const BoxDev& b = g.boxes[box_of(g.box_p0, g.nbox, i)];
            bool ok;
            r[k] = rank[i];
            brick[k] = brick_of(pos, i, b, rec[k], ok);
        }
    }
#pragma unroll
    for (int k = 0; k < kBinItems; ++k) {
        if (brick[k] < 0)
            continue;
        const int64_t slot = (int64_t)__ldg(bstart + brick[k]) + r[k];
        if (slot < __ldg(bstart + brick[k] + 1))
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

// The same for 64-bit words (fields that never carry into each other).
__device__ __forceinline__ unsigned long long block_exclusive_scan64(unsigned long long v,
                                                                     unsigned long long* smem_warp,
                                                                     unsigned long long& total)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    unsigned long long x = v;
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long y = __shfl_up_sync(kFull, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) smem_warp[wid] = x;
    __syncthreads();
    if (wid == 0) {
        const int nw = blockDim.x >> 5;
        unsigned long long t = lane < nw ? smem_warp[lane] : 0ull;
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long y = __shfl_up_sync(kFull, t, o);
            if (lane >= o) t += y;
        }
        if (lane < nw) smem_warp[lane] = t;
    }
    __syncthreads();
    const unsigned long long warp_off = wid ? smem_warp[wid - 1] : 0ull;
    total = smem_warp[(blockDim.x >> 5) - 1];
    __syncthreads();
    return warp_off + x - v;
}

// out[i] for i in [0, len]: out[len] is the grand total (a virtual zero is
// appended to the input, so the scan covers len + 1 entries).  The counts lie
// `pad` words apart.
__global__ void __launch_bounds__(kScanThreads) k_scan(const int* __restrict__ in, int pad, int* __restrict__ out,
                                                       int64_t len, unsigned long long* __restrict__ state,
                                                       int* __restrict__ ticket, int* __restrict__ err)
{
    __shared__ int sw[32];
    __shared__ int s_tile, s_before;
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
    for (int k = 0; k < kScanItems; ++k)
        s += v[k];
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

constexpr int kSortThreads = 1024;
constexpr int kMaxR3 = 4096;   // r <= 16

__global__ void __launch_bounds__(kSortThreads) k_brick_sort(Geometry g, const float4* __restrict__ tmp,
                                                             const int* __restrict__ bstart,
                                                             float4* __restrict__ sorted,
                                                             int* __restrict__ parent,
                                                             int* __restrict__ minorig,
                                                             int* __restrict__ cnt,
                                                             int* __restrict__ cell_start,
                                                             int* __restrict__ err,
                                                             int64_t* __restrict__ dense_list,
                                                             int* __restrict__ n_dense,
                                                             int dense_min,
                                                             int64_t* __restrict__ team_list,
                                                             int* __restrict__ n_team,
                                                             int* __restrict__ n_team_hi,
                                                             int64_t team_cap,
                                                             int64_t* __restrict__ big_list,
                                                             int* __restrict__ n_big)
{
    __shared__ int hist[kMaxR3];
    __shared__ int sw[32];
    __shared__ unsigned long long sw64[32];
    __shared__ int list_base[4];
    for (int64_t gb = blockIdx.x; gb < g.total_bricks; gb += gridDim.x) {
        const int bi = box_of(g.box_brick0, g.nbox, gb);
        const BoxDev& b = g.boxes[bi];
        const int r3 = b.r * b.r * b.r;
        const int m = b.r - 1;
        const int s0 = bstart[gb], s1 = bstart[gb + 1];
        for (int c = threadIdx.x; c < r3; c += blockDim.x) hist[c] = 0;
        __syncthreads();
        for (int k = s0 + threadIdx.x; k < s1; k += blockDim.x) {
            float4 p = tmp[k];
            int lc = local_code(cell_coord(p.x, b) & m, cell_coord(p.y, b) & m, cell_coord(p.z, b) & m);
            atomicAdd(hist + lc, 1);
        }
        __syncthreads();
        // exclusive scan of hist[0..r3): each thread owns a contiguous run
        const int per = (r3 + blockDim.x - 1) / blockDim.x;
        const int c0 = threadIdx.x * per;
        int run = 0;
        for (int c = c0; c < c0 + per && c < r3; ++c) run += hist[c];
        int total;
        int ex = block_exclusive_scan(run, sw, total);
        const int ex0 = ex;
        const int64_t cbase = b.cell0 + (gb - b.brick0) * (int64_t)r3;
        int nd = 0, nt = 0, nth = 0, nbg = 0;   // this thread's dense, team (small, large) and big cells
        for (int c = c0; c < c0 + per && c < r3; ++c) {
            const int h = hist[c];
            ex += h;
            if (is_big(h, b))
                ++nbg;
            else if (is_sub(h, b, dense_min))
                ++nd;
            else if (h >= b.team_min && h <= kTeamSplit)
                ++nt;
            else if (h >= b.team_min && h <= kTeamSelfMax)
                ++nth;
        }
        // list slots: one reservation per brick (a shared counter per cell
        // would serialise millions of atomics on one address).  The four
        // counts (each at most kMaxR3 per brick) share one scan as 16-bit
        // fields of a 64-bit word.
        unsigned long long tot4;
        const unsigned long long o4 = block_exclusive_scan64(
            (unsigned long long)nd | ((unsigned long long)nt << 16) | ((unsigned long long)nth << 32) |
                ((unsigned long long)nbg << 48),
            sw64, tot4);
        const int nd_tot = (int)(tot4 & 0xffffu), nt_tot = (int)((tot4 >> 16) & 0xffffu);
        const int nth_tot = (int)((tot4 >> 32) & 0xffffu), nb_tot = (int)(tot4 >> 48);
        int od = (int)(o4 & 0xffffu), ot = (int)((o4 >> 16) & 0xffffu);
        int oth = (int)((o4 >> 32) & 0xffffu), obg = (int)(o4 >> 48);
        if (threadIdx.x == 0) {
            list_base[0] = nd_tot ? atomicAdd(n_dense, nd_tot) : 0;
            list_base[1] = nt_tot ? atomicAdd(n_team, nt_tot) : 0;
            list_base[2] = nb_tot ? atomicAdd(n_big, nb_tot) : 0;
            list_base[3] = nth_tot ? atomicAdd(n_team_hi, nth_tot) : 0;
        }
        __syncthreads();
        od += list_base[0];
        ot += list_base[1];
        obg += list_base[2];
        oth += list_base[3];
        ex = ex0;
        for (int c = c0; c < c0 + per && c < r3; ++c) {
            const int h = hist[c];
            const int start = s0 + ex;
            hist[c] = ex;                       // becomes the cursor
            ex += h;
            if (is_big(h, b))
                big_list[obg++] = cbase + c;
            else if (is_sub(h, b, dense_min))
                dense_list[od++] = cbase + c;
            else if (h >= b.team_min && h <= kTeamSplit)
                team_list[ot++] = ((int64_t)h << 32) | (uint32_t)start;
            else if (h >= b.team_min && h <= kTeamSelfMax)
                team_list[team_cap - 1 - oth++] = ((int64_t)h << 32) | (uint32_t)start;
        }
        __syncthreads();
        for (int k = s0 + threadIdx.x; k < s1; k += blockDim.x) {
            float4 p = tmp[k];
            int lc = local_code(cell_coord(p.x, b) & m, cell_coord(p.y, b) & m, cell_coord(p.z, b) & m);
            int slot = s0 + atomicAdd(hist + lc, 1);
            if (slot >= s1) {
                atomicOr(err, kErrInternal);
                continue;
            }
            sorted[slot] = p;
            minorig[slot] = __float_as_int(p.w);
        }
        for (int k = s0 + threadIdx.x; k < s1; k += blockDim.x) {
            parent[k] = k;
            cnt[k] = 1;
        }
        // the cursors now hold each cell's end: the cell starts, written
        // coalesced (cell c + 1 starts where c ends; the next brick writes
        // the same value at its first cell)
        __syncthreads();
        for (int c = threadIdx.x; c < r3; c += blockDim.x)
            cell_start[cbase + c + 1] = s0 + hist[c];
        if (threadIdx.x == 0)
            cell_start[cbase] = s0;
        __syncthreads();
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
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    int f = 0, bad = 0;
    for (int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; s < g.total_n; s += stride) {
        const BoxDev& b = g.boxes[box_of(g.box_p0, g.nbox, s)];
        const float4 old = sorted[s];
        const int o = __float_as_int(old.w);
        const int64_t i = b.p0 + o;
        float4 rec;
        bool ok;
        const int64_t nb = brick_of(pos, i, b, rec, ok);
        bad |= !ok;
        const int ox = cell_coord(old.x, b), oy = cell_coord(old.y, b), oz = cell_coord(old.z, b);
        const int nx = cell_coord(rec.x, b), ny = cell_coord(rec.y, b), nz = cell_coord(rec.z, b);
        if (nx != ox || ny != oy || nz != oz)
            f |= 1;
        if (nb != b.brick0 + brick_local(b, ox, oy, oz))
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
__global__ void __launch_bounds__(256) k_forest_init(int64_t total, const float4* __restrict__ sorted,
                                                     int* __restrict__ parent, int* __restrict__ minorig,
                                                     int* __restrict__ cnt)
{
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
    if (g.total_bricks <= kTileBricks) {
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

cudaError_t launch_scan(const int* in, int pad, int* out, int64_t len, unsigned long long* state, int* ticket,
                        int* err, cudaStream_t s)
{
    k_scan<<<(unsigned)scan_tiles(len), kScanThreads, 0, s>>>(in, pad, out, len, state, ticket, err);
    return cudaGetLastError();
}

cudaError_t launch_bin_scatter(const float* pos, const Geometry& g, const Work& w, cudaStream_t s)
{
    if (g.total_n == 0)
        return cudaSuccess;
    // in the order in which the ranks were given out
    const int streams = g.total_bricks <= kTileBricks ? 1 : kBinStreams;
    k_bin_scatter<<<(unsigned)(bin_tiles_per_stream(g.total_n, streams) * streams), kBinThreads, 0, s>>>(
        pos, g, w.bstart, w.parent, streams, w.tmp, &w.status->err);
    return cudaGetLastError();
}

cudaError_t launch_brick_sort(const Geometry& g, const Work& w, int dense_min, cudaStream_t s)
{
    if (g.total_bricks == 0)
        return cudaSuccess;
    int64_t blocks = g.total_bricks;
    int64_t cap = (int64_t)sm_count() * 4 * 16;
    if (blocks > cap) blocks = cap;
    k_brick_sort<<<(unsigned)blocks, kSortThreads, 0, s>>>(g, w.tmp, w.bstart, w.sorted, w.parent,
                                                         w.minorig, w.cnt, w.cell_start,
                                                         &w.status->err, w.dense_list, w.n_dense,
                                                         dense_min, w.team_list, w.n_team, w.n_team_hi,
                                                         w.team_cap, w.big_list, w.n_big);
    return cudaGetLastError();
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
    k_forest_init<<<grid_for(g.total_n, 256, 8), 256, 0, s>>>(g.total_n, w.sorted, w.parent, w.minorig,
                                                             w.cnt);
    return cudaGetLastError();
}

}  // namespace fofgpu
