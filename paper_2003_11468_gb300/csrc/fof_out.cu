// Flattening the forest into outputs.
//
//   finalize   full pointer jumping: parent[s] = root(s) for every slot; each
//              non-root adds itself to its root's size and offers its input
//              index to the root's minimum.  Roots were initialised with
//              size 1 and their own index, so they take part in no atomic:
//              the paper's early elimination of singletons (Sec. 3.4.2),
//              with the atomic additions of its parallel size count
//              (Sec. 3.4.1) aggregated per warp.  Once per run: the sizes
//              are sums, so a second fof_groups finds them final (Status::flat)
//              and only clears the words that the outputs count in.
//   outputs    (label, size) of every slot's group stored at the input index;
//              per-box group and catalogue counts.
//   catalogue  ids[i] = smallest index of i's group; sizes[label] = size, 0
//              elsewhere; (label, size) entries in ascending label order.
#include <algorithm>

#include "fof_internal.cuh"

namespace fofgpu {

namespace {

// Root of slot s by a plain walk, then parent[s] = root.  `ordered`: every
// parent is at most its child (hooks onto the smaller root), checked.
__device__ __forceinline__ int final_root(int* __restrict__ parent, int s, int p, bool ordered, int* err)
{
    if (p == s)
        return s;
    int x = p;
    int q = parent[x];
    for (int step = 0; q != x; ++step) {
        if ((ordered && q > x) || step >= kFindCap) {   // corrupted forest: report
            atomicOr(err, kErrInternal);
            break;
        }
        x = q;
        q = parent[x];
    }
    if (p != x)
        parent[s] = x;
    return x;
}

// The words that fof_groups counts in start at zero, whatever ran before: also
// where a graph replays fof_groups alone, which no state of the host could tell.
__device__ __forceinline__ void clear_group_words(int* words, int64_t n)
{
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        words[i] = 0;
}

// Bound by the latency of the walk to the root, so a slot's own words are read
// one slot ahead (453 million slots: 1.97 and 1.54 ms; with 16 CTAs per SM in
// the grid instead of 8, 1.48).
__global__ void __launch_bounds__(256) k_finalize(int64_t total, int* __restrict__ parent,
                                                  int* __restrict__ minorig, int* __restrict__ cnt,
                                                  int* group_words, int64_t n_group_words, Status* status,
                                                  bool ordered)
{
    pdl_wait();
    pdl_trigger();
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    int p_next = 0, mo_next = 0;
    if (s < total) {
        p_next = parent[s];
        mo_next = minorig[s];
    }
    const bool flat = status->flat != 0;       // used last: its load overlaps the walk
    clear_group_words(group_words, n_group_words);
    for (; s - threadIdx.x < total; s += stride) {
        const bool valid = s < total;
        const int p = p_next, mo = mo_next;
        // the next slot's words: only this thread writes them, unless the slot
        // is a root, whose words are not used
        if (s + stride < total) {
            p_next = parent[s + stride];
            mo_next = minorig[s + stride];
        }
        unsigned active = __ballot_sync(kFull, valid);
        if (!valid)
            continue;
        const int root = final_root(parent, (int)s, p, ordered, &status->err);
        bool nonroot = root != (int)s;
        unsigned nr = __ballot_sync(active, nonroot);
        if (!nonroot)
            continue;
        unsigned peers = __match_any_sync(nr, root);
        int leader = __ffs(peers) - 1;
        unsigned mn = __reduce_min_sync(peers, (unsigned)mo);
        if ((threadIdx.x & 31) == leader && !flat) {
            atomicAdd(cnt + root, __popc(peers));
            atomicMin(minorig + root, (int)mn);
        }
    }
}

// The same finalisation with the paper's hash-table size count (Sec. 3.4.1):
// each block gathers (root, count, smallest index) of the non-roots of
// kHashBatch consecutive slot tiles in an open-addressing table in shared
// memory, then adds each entry to the root with one atomic per entry (roots
// are not entered: their own contribution is the initial size 1, Sec.
// 3.4.2).  A slot whose probe sequence finds no room adds itself directly.
constexpr int kHashSlots = 4096;     // power of two
constexpr int kHashBatch = 8;        // tiles of 256 slots per flush: <= 2048 keys, load <= 1/2
constexpr int kHashProbes = 16;

__global__ void __launch_bounds__(256) k_finalize_hash(int64_t total, int* __restrict__ parent,
                                                       int* __restrict__ minorig, int* __restrict__ cnt,
                                                       int* group_words, int64_t n_group_words, Status* status,
                                                       bool ordered)
{
    pdl_wait();
    pdl_trigger();
    clear_group_words(group_words, n_group_words);
    if (status->flat)
        return;
    __shared__ int hkey[kHashSlots];
    __shared__ int hcnt[kHashSlots];
    __shared__ int hmin[kHashSlots];
    for (int k = threadIdx.x; k < kHashSlots; k += blockDim.x)
        hkey[k] = -1;
    __syncthreads();
    const int64_t span = (int64_t)blockDim.x * kHashBatch;
    for (int64_t b0 = (int64_t)blockIdx.x * span; b0 < total; b0 += (int64_t)gridDim.x * span) {
        for (int t = 0; t < kHashBatch; ++t) {
            const int64_t s = b0 + (int64_t)t * blockDim.x + threadIdx.x;
            if (s >= total)
                break;
            const int root = final_root(parent, (int)s, parent[s], ordered, &status->err);
            if (root == (int)s)
                continue;
            const int mo = minorig[s];
            uint32_t h = uf_priority(root) & (kHashSlots - 1);
            bool placed = false;
            for (int probe = 0; probe < kHashProbes; ++probe, h = (h + 1) & (kHashSlots - 1)) {
                const int k = atomicCAS(&hkey[h], -1, root);
                if (k == -1 || k == root) {
                    if (k == -1) {            // the first insert initialises the entry
                        hcnt[h] = 0;
                        hmin[h] = INT_MAX;
                    }
                    placed = true;
                    break;
                }
            }
            if (!placed) {                    // no room on the probe path: add directly
                atomicAdd(cnt + root, 1);
                atomicMin(minorig + root, mo);
            }
            // entries are counted in the second pass, after every entry of
            // the batch has been initialised
        }
        __syncthreads();
        // second pass over the same slots: the table entries are initialised
        for (int t = 0; t < kHashBatch; ++t) {
            const int64_t s = b0 + (int64_t)t * blockDim.x + threadIdx.x;
            if (s >= total)
                break;
            const int root = parent[s];   // fully compressed by the first pass
            if (root == (int)s)
                continue;
            uint32_t h = uf_priority(root) & (kHashSlots - 1);
            for (int probe = 0; probe < kHashProbes; ++probe, h = (h + 1) & (kHashSlots - 1)) {
                if (hkey[h] == root) {
                    atomicAdd(&hcnt[h], 1);
                    atomicMin(&hmin[h], minorig[s]);
                    break;
                }
            }
        }
        __syncthreads();
        for (int k = threadIdx.x; k < kHashSlots; k += blockDim.x) {
            const int r = hkey[k];
            if (r >= 0) {
                atomicAdd(cnt + r, hcnt[k]);
                atomicMin(minorig + r, hmin[k]);
                hkey[k] = -1;
            }
        }
        __syncthreads();
    }
}

// Outputs go back to input order in two passes:
//   scatter  for every binned slot: the label and size of its group as one
//            8-byte pair (label, size if the input is its group's label, else
//            0).  Up to kDirectMax inputs the pair is stored at the input's
//            index: the pairs then stay in L2, and nothing but the store is
//            needed.  Above, a sector of the pair array would leave L2 between
//            its stores (a read-modify-write of DRAM for each), so the pairs
//            are appended to the bucket of the input's tile instead, whose
//            write heads stay in L2.  A tile holds exactly kOutTile inputs (the
//            last one fewer), so bucket t starts at t * kOutTile.  (Direct and
//            bucketed, this kernel when its CTAs strode over the slots: 2
//            million inputs 25 and 270 us, the buckets' cursors sharing lines;
//            16.7 million 0.27 and 0.38 ms; 453 million 17.2 and 7.4 ms.)
//   write    one CTA per tile: ids and sizes written out coalesced (a bucket's
//            pairs placed in shared memory first), and the tile's catalogue
//            entries (sizes at least thr, ascending label).  Up to kDirectMax
//            inputs the entries are compacted at once, at an offset found by
//            a decoupled look-back over the earlier tiles: no scan launch and
//            no second read of the sizes.  Above, the look-back's chain over
//            the tiles takes longer than the tiles themselves (453 million
//            inputs: 2.6 ms), so the kernel leaves the tile's count, and a
//            scan and k_catalogue follow (1.3 ms in all).
constexpr int kScatterThreads = 256, kScatterWarps = kScatterThreads / 32;
constexpr int kScatterTiles = 4;             // tiles of kScatterThreads slots per CTA
constexpr int kScatterStreams = 64;          // places of the slots that take turns (buckets)

// Bound by the scattered stores and the cursors' atomics.  A slot's words are
// read one slot ahead, and nothing waits for another load but the group's words
// for the root.  A CTA takes kScatterTiles consecutive tiles, and CTAs start in
// order, so that the slots at work lie close together; CTAs that stride over the
// slots drift apart, and a sector of the pairs is written in several pieces.
// Buckets: neighbouring slots also use the same few cursors (a batch's boxes have
// a hundred each), so chunks of kScatterStreams evenly spaced places take turns
// (a batch of 512 boxes: 21.1 ms with 1 place, 4.1 with 16, 3.3 with 64 and 256).
// The box counters get one addition per CTA: one per warp would be more atomics
// on one address than the rest takes.  Striding before and so, us: 2 million slots
// 25 and 20, 16.8 million 261 and 233 (1 tile: 222, but 7.8 instead of 5.6 ms in
// the 768^3 box, and 70 instead of 49 for 4 million), 453 million 7370 and 5620,
// the batch 4430 and 3270.

template <bool kDirect>
__global__ void __launch_bounds__(kScatterThreads) k_outputs_scatter(Geometry g, const float4* sorted,
                                                         const int* parent,
                                                         const int* minorig, const int* cnt, int32_t thr,
                                                         unsigned long long* __restrict__ n_groups,
                                                         unsigned long long* __restrict__ n_cat,
                                                         int2* __restrict__ pairs,
                                                         int* __restrict__ out_cursor, int per, int streams,
                                                         Status* status)
{
    pdl_wait();
    pdl_trigger();
    if (blockIdx.x == 0 && threadIdx.x == 0)
        status->flat = 1;                       // every CTA of the finalisation has read it
    __shared__ int s_box[kScatterWarps];
    __shared__ int2 s_acc[kScatterWarps];
    const int lane = threadIdx.x & 31;
    int acc_box = -1;                           // per-warp box counts not yet added
    int acc_ng = 0, acc_nk = 0;
    // this CTA's slots
    constexpr int stride = kScatterThreads;
    const int64_t chunk = (int64_t)(blockIdx.x % streams) * (gridDim.x / streams) + blockIdx.x / streams;
    int64_t s = chunk * per * stride + threadIdx.x;
    const int64_t end = min(g.total_n, (chunk + 1) * per * stride);
    BoxCursor box;
    int root_next = 0, mo_next = 0, cnt_next = 0;
    if (s < end) {
        root_next = parent[s];
        mo_next = minorig[s];
        cnt_next = cnt[s];
    }
    for (; s - threadIdx.x < end; s += stride) {
        const bool valid = s < end;
        const int root = root_next, own = mo_next, own_cnt = cnt_next;
        if (s + stride < end) {                 // the next slot's words
            root_next = parent[s + stride];
            mo_next = minorig[s + stride];
            cnt_next = cnt[s + stride];
        }
        unsigned active = __ballot_sync(kFull, valid);
        const int bi = box.at(g.box_p0, g.nbox, s - lane, s, lane);
        if (!valid)
            continue;
        const bool is_root = root == (int)s;
        // the input index o of slot s: minorig keeps it for every non-root
        // (the label pass only lowers roots' entries) and for singleton
        // roots; only a root of a larger group reads it from the binned record.
        // The loads do not wait for one another.
        int label = own, size = own_cnt, o = own;
        if (!is_root) {
            label = minorig[root];
            size = cnt[root];
        } else if (own_cnt != 1) {
            o = __float_as_int(sorted[s].w);
        }
        const int64_t p0 = g.boxes[bi].p0;
        // a record that binning never wrote is reported, and stays inside the box
        const bool ok = (unsigned long long)o < (unsigned long long)g.boxes[bi].n;
        const int64_t gidx = p0 + (ok ? o : 0);
        int64_t at = gidx;
        int2 e = make_int2(label, o == label ? size : 0);
        bool room = ok;
        if constexpr (!kDirect) {
            const int tile = (int)(gidx / kOutTile);
            const unsigned peers = __match_any_sync(active, tile);
            const int leader = __ffs(peers) - 1;
            int off = 0;
            if (lane == leader)
                off = atomicAdd(out_cursor + tile, __popc(peers));
            off = __shfl_sync(active, off, leader) + __popc(peers & ((1u << lane) - 1u));
            room = ok && off < kOutTile;
            at = (int64_t)tile * kOutTile + off;
            // a bucket's pair: (place in the tile | is-label << 31, size or label);
            // a label is its own input's box-local index
            e = make_int2((int)(gidx % kOutTile) | (o == label ? (int)0x80000000u : 0), o == label ? size : label);
        }
        if (room)
            pairs[at] = e;
        else
            atomicOr(&status->err, kErrInternal);
        const bool in_cat = is_root && size >= thr;
        // per-box counts: summed in registers while the warp stays inside one
        // box and added once per box (one counter per box would otherwise
        // take an atomic from every warp, all on one address)
        const int bi0 = __shfl_sync(active, bi, 0);
        const unsigned roots = __ballot_sync(active, is_root), cats = __ballot_sync(active, in_cat);
        if (__all_sync(active, bi == bi0)) {
            if (bi0 != acc_box) {
                if (lane == 0 && acc_box >= 0) {
                    if (acc_ng) atomicAdd(n_groups + acc_box, (unsigned long long)acc_ng);
                    if (acc_nk) atomicAdd(n_cat + acc_box, (unsigned long long)acc_nk);
                }
                acc_box = bi0;
                acc_ng = acc_nk = 0;
            }
            acc_ng += __popc(roots);
            acc_nk += __popc(cats);
        } else {
            unsigned bpeers = __match_any_sync(active, bi);
            int bleader = __ffs(bpeers) - 1;
            int ng = __popc(roots & bpeers);
            int nk = __popc(cats & bpeers);
            if (lane == bleader) {
                if (ng) atomicAdd(n_groups + bi, (unsigned long long)ng);
                if (nk) atomicAdd(n_cat + bi, (unsigned long long)nk);
            }
        }
    }
    // lane 0 took part in every iteration (its slot is the warp's smallest)
    if (lane == 0) {
        s_box[threadIdx.x >> 5] = acc_box;
        s_acc[threadIdx.x >> 5] = make_int2(acc_ng, acc_nk);
    }
    __syncthreads();
    // the CTA's warps mostly end in one box: one addition for each run of them
    if (threadIdx.x == 0) {
        int box = -1, ng = 0, nk = 0;
        for (int w = 0; w <= kScatterWarps; ++w) {
            const int wb = w < kScatterWarps ? s_box[w] : -1;
            if (wb != box) {
                if (ng) atomicAdd(n_groups + box, (unsigned long long)ng);
                if (nk) atomicAdd(n_cat + box, (unsigned long long)nk);
                box = wb;
                ng = nk = 0;
            }
            if (w < kScatterWarps) {
                ng += s_acc[w].x;
                nk += s_acc[w].y;
            }
        }
    }
}

constexpr int kOutThreads = 512;
constexpr int kOutItems = kOutTile / kOutThreads;       // 8 rows of 512 inputs
constexpr int kOutWarps = kOutThreads / 32;
static_assert(kOutItems * kOutWarps == 4 * kWarp, "four row counts per lane of warp 0");

// Exclusive prefix of the 128 row counts of a tile, in place, by warp 0;
// returns their sum.
__device__ __forceinline__ int scan_rows(int* s_cnt, int lane)
{
    int c[4], sum = 0;
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        c[r] = sum;
        sum += s_cnt[4 * lane + r];
    }
    int x = sum;
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(kFull, x, o);
        if (lane >= o) x += y;
    }
#pragma unroll
    for (int r = 0; r < 4; ++r)
        s_cnt[4 * lane + r] = x - sum + c[r];
    return __shfl_sync(kFull, x, 31);
}

template <bool kDirect>
__global__ void __launch_bounds__(kOutThreads) k_outputs_write(Geometry g, const int2* pairs,
                                                               int32_t* __restrict__ ids,
                                                               int32_t* __restrict__ sizes, int32_t thr,
                                                               int2* __restrict__ cat, int64_t cap,
                                                               unsigned long long* __restrict__ tile_state,
                                                               int* __restrict__ ticket,
                                                               int* __restrict__ out_cursor, Status* status)
{
    pdl_wait();
    pdl_trigger();
    __shared__ int s_tile, s_off;
    __shared__ int s_cnt[kOutItems * kOutWarps];
    __shared__ int2 placed[kDirect ? 1 : kOutTile];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    // tiles are handed out in order, so every earlier tile is running or done
    int tile = blockIdx.x;
    if constexpr (kDirect) {
        if (threadIdx.x == 0)
            s_tile = atomicAdd(ticket, 1);
        __syncthreads();
        tile = s_tile;
    }
    const int64_t base = (int64_t)tile * kOutTile;
    int2 e[kOutItems];
    unsigned in[kOutItems];
#pragma unroll
    for (int k = 0; k < kOutItems; ++k) {
        const int64_t i = base + k * kOutThreads + threadIdx.x;
        e[k] = i < g.total_n ? pairs[i] : make_int2(0, 0);
    }
    if constexpr (!kDirect) {
        // the box of the tile's first input, and where it ends
        const int bi = box_of_warp(g.box_p0, g.nbox, base, lane);
        const int64_t p0 = g.boxes[bi].p0, p1 = p0 + g.boxes[bi].n;
#pragma unroll
        for (int k = 0; k < kOutItems; ++k) {
            const int64_t i = base + k * kOutThreads + threadIdx.x;
            if (i < g.total_n) {
                const int off = e[k].x & (kOutTile - 1);
                if (e[k].x < 0) {                        // the input is its group's label
                    const int64_t gidx = base + off;
                    e[k].x = (int)(gidx - (gidx < p1 ? p0 : g.boxes[box_of(g.box_p0, g.nbox, gidx)].p0));
                } else {
                    e[k] = make_int2(e[k].y, 0);
                }
                placed[off] = e[k];
            }
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < kOutItems; ++k)
            e[k] = base + k * kOutThreads + threadIdx.x < g.total_n ? placed[k * kOutThreads + threadIdx.x]
                                                                    : make_int2(0, 0);
    }
#pragma unroll
    for (int k = 0; k < kOutItems; ++k) {
        const int64_t i = base + k * kOutThreads + threadIdx.x;
        if (i < g.total_n) {
            ids[i] = e[k].x;
            sizes[i] = e[k].y;
        }
        in[k] = __ballot_sync(kFull, e[k].y >= thr);     // thr >= 1: never past the end
        if (lane == 0)
            s_cnt[k * kOutWarps + wid] = __popc(in[k]);
    }
    __syncthreads();
    if (wid == 0) {
        const int mine = scan_rows(s_cnt, lane);
        if constexpr (!kDirect) {
            if (lane == 0)
                out_cursor[tile] = mine;                 // the bucket has been read
            return;
        }
        const int before = lookback(tile_state, tile, mine, lane, &status->err);
        if (lane == 0) {
            s_off = before;
            if (base + kOutTile >= g.total_n)            // the last tile knows the total
                status->n_cat_total = before + mine;
        }
    }
    if constexpr (!kDirect)
        return;
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kOutItems; ++k) {
        if (e[k].y >= thr) {
            const int64_t off = (int64_t)s_off + s_cnt[k * kOutWarps + wid] + __popc(in[k] & ((1u << lane) - 1u));
            if (off < cap)
                cat[off] = e[k];                         // the input is its label
        }
    }
}

// Catalogue above kDirectMax inputs: one CTA per output tile that holds
// entries writes them in ascending label order from tile_off[tile] on.
__global__ void __launch_bounds__(kOutThreads) k_catalogue(Geometry g, const int32_t* sizes, const int* tile_off,
                                                           int32_t thr, int2* __restrict__ cat, int64_t cap,
                                                           int64_t n_tiles, Status* status)
{
    pdl_wait();
    pdl_trigger();
    __shared__ int s_cnt[kOutItems * kOutWarps];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (blockIdx.x == 0 && threadIdx.x == 0)
        status->n_cat_total = tile_off[n_tiles];
    for (int64_t tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
        const int t0 = tile_off[tile];
        if (tile_off[tile + 1] == t0)
            continue;                                    // block-uniform
        int size[kOutItems];
        unsigned in[kOutItems];
#pragma unroll
        for (int k = 0; k < kOutItems; ++k) {
            const int64_t i = tile * kOutTile + k * kOutThreads + threadIdx.x;
            size[k] = i < g.total_n ? sizes[i] : 0;
        }
#pragma unroll
        for (int k = 0; k < kOutItems; ++k) {
            in[k] = __ballot_sync(kFull, size[k] >= thr);
            if (lane == 0)
                s_cnt[k * kOutWarps + wid] = __popc(in[k]);
        }
        __syncthreads();
        if (wid == 0)
            scan_rows(s_cnt, lane);
        __syncthreads();
#pragma unroll
        for (int k = 0; k < kOutItems; ++k) {
            if (size[k] >= thr) {
                const int64_t off =
                    (int64_t)t0 + s_cnt[k * kOutWarps + wid] + __popc(in[k] & ((1u << lane) - 1u));
                if (off < cap) {
                    const int64_t i = tile * kOutTile + k * kOutThreads + threadIdx.x;
                    cat[off] = make_int2((int)(i - g.boxes[box_of(g.box_p0, g.nbox, i)].p0), size[k]);
                }
            }
        }
        __syncthreads();
    }
}

}  // namespace

static int grid_for(int64_t items, int threads, int per_sm)
{
    int64_t want = (items + threads - 1) / threads;
    int64_t cap = (int64_t)sm_count() * per_sm;
    if (want < 1) want = 1;
    return (int)(want < cap ? want : cap);
}

cudaError_t launch_finalize(const Geometry& g, const Work& w, const UfArgs& uf, int size_count, cudaStream_t s)
{
    if (g.total_n == 0)
        return cudaSuccess;
    const bool ordered = uf.link == 0;
    if (size_count == 1)
        return launch_next(g.total_n, k_finalize_hash, grid_for(g.total_n, 256 * kHashBatch, 4), 256, 0, s, g.total_n,
                           w.parent, w.minorig, w.cnt, w.group_words, w.n_group_words, w.status, ordered);
    return launch_next(g.total_n, k_finalize, grid_for(g.total_n, 256, 16), 256, 0, s, g.total_n, w.parent, w.minorig,
                       w.cnt, w.group_words, w.n_group_words, w.status, ordered);
}

cudaError_t launch_outputs(const Geometry& g, const Work& w, int32_t* ids, int32_t* sizes, int32_t min_size,
                           int2* cat, int64_t cap, cudaStream_t s)
{
    if (g.total_n == 0)
        return cudaSuccess;
    const int32_t thr = min_size < 1 ? 1 : min_size;
    int2* pairs = (int2*)w.tmp;            // the brick-order copy is dead by now
    const int64_t tiles = (g.total_n + kScatterThreads - 1) / kScatterThreads;
    // as many slots per CTA as leave eight CTAs to an SM
    const int per = (int)std::min<int64_t>(kScatterTiles, std::max<int64_t>(1, tiles / ((int64_t)sm_count() * 8)));
    const bool direct = g.total_n <= kDirectMax;
    const int streams = direct ? 1 : kScatterStreams;
    const int64_t chunks = (tiles + per - 1) / per;
    cudaError_t e = launch_next(g.total_n, direct ? k_outputs_scatter<true> : k_outputs_scatter<false>,
                                (chunks + streams - 1) / streams * streams, kScatterThreads, 0, s, g, w.sorted,
                                w.parent, w.minorig, w.cnt, thr, w.n_groups, w.n_cat, pairs, w.out_cursor, per,
                                streams, w.status);
    if (e != cudaSuccess)
        return e;
    return launch_next(g.total_n, direct ? k_outputs_write<true> : k_outputs_write<false>, w.n_tiles, kOutThreads, 0, s,
                       g, (const int2*)pairs, ids, sizes, thr, cat, cap, w.tile_state, w.tile_ticket, w.out_cursor,
                       w.status);
}

int catalogue_launches(const Geometry& g)
{
    return g.total_n <= kDirectMax ? 0 : 2;     // k_outputs_write leaves it behind too
}

cudaError_t launch_catalogue(const Geometry& g, const Work& w, const int32_t* sizes, int32_t min_size, int2* cat,
                             int64_t cap, cudaStream_t s)
{
    if (catalogue_launches(g) == 0)
        return cudaSuccess;
    const int32_t thr = min_size < 1 ? 1 : min_size;
    cudaError_t e = launch_scan(g.total_n, w.out_cursor, 1, w.tile_off, w.n_tiles, w.tile_state, w.tile_ticket, 0,
                                nullptr, nullptr, &w.status->err, s);
    if (e != cudaSuccess)
        return e;
    return launch_next(g.total_n, k_catalogue, grid_for(w.n_tiles * kOutThreads, kOutThreads, 4), kOutThreads, 0, s, g, sizes,
                       w.tile_off, thr, cat, cap, w.n_tiles, w.status);
}

}  // namespace fofgpu
