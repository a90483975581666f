// Dense cells: the paper's self and pair tasks (Sec. 3.1, Fig. 1) for cells
// that hold many particles, done in shared memory.
//
// A cell with T <= m <= kDenseMax particles (T = dense_min) in a box whose
// cells can be split ("subdivided" cells) is cut into q^3 sub-cells of side
// hf with l_x/2 < hf <= l_x / (sqrt(3) (1 + 2^-7)).  Two facts follow from
// the float32 cell-index margin (fof_plan.cu, setup_box):
//   * every two particles of one sub-cell are linked (the sub-cell diameter
//     is below l_x even with the index rounding), so a sub-cell is a clique;
//   * every linked pair lies at most 2 sub-cells apart on each axis.
// Hence the groups inside a dense cell follow from a union-find over its
// sub-cells and one linking pair per pair of sub-cells within +-2.
//
//   dense_self   one CTA per subdivided cell: its slots are sorted by sub-cell
//                (in shared memory and in the binned order), sub-cells that
//                share a face are joined, then every sub-cell that is still
//                outside the group of the fullest one searches its whole +-2
//                window; the cell's forest goes to the global parent array
//                (roots = smallest slot, as union-by-root onto the lower
//                offset gives).  Then every particle of the 26 neighbour cells
//                that are NOT subdivided is linked against the sub-cells
//                within its +-2 window with the global CAS union.
//   dense_pairs  one CTA per subdivided cell A: each forward neighbour B
//                that is subdivided too, B's particles against A's sub-cells.
//                If both cells are one group each and their roots already
//                agree there is nothing to do.
//
// What bounds them is the chain of one cell, not the chip: a box of 60,000
// particles has ten dense cells.  So the searches are spread over a warp
// (32 candidates at a time: the particles of a row of sub-cells are
// contiguous), and a particle outside is tested against the group of the
// fullest sub-cell only while its own root differs from that group's, with
// one union per 32 particles and root.  An earlier version searched with one
// thread per particle or sub-cell and united it with each sub-cell of the
// window whose recorded root looked different, which is every one of them
// once the group's root has moved.  dense_self + dense_pairs before and after,
// us: 60,000 particles 359 and 66, 2 million 422 and 95, 16.8 million (256^3)
// 1107 and 370, 453 million (768^3) 8328 and 3940.
#include "fof_internal.cuh"

namespace fofgpu {

namespace {

struct DenseSmem {
    float4* P;           // [kM] positions of the cell in sub-cell order (slot order)
    int* sstart;         // [kMaxQ3 + 1] sub-cell starts in P
    int* lpar;           // [kMaxQ3] forest over the sub-cells, then the global node of each one's group
    unsigned short* skey;  // [kM] sub-cell of each particle
    unsigned short* ng;  // [kMaxQ3] sub-cells outside the fullest one's group
    unsigned* rowng;     // [kMaxQ * kMaxQ] per (z, y) row: bit x = such a sub-cell
    int* misc;           // scalars
    int* nbj0;           // [26] first slot of each neighbour cell
    int* nbpref;         // [27] prefix of the neighbour particle counts to visit
};

// Two size classes of dense cells, each its own instantiation: cells up to
// kDenseSmall particles need a fifth of the shared memory, so six CTAs (of
// 256 threads, 40 registers, 90 to 100 bytes spilled) share an SM and barrier
// stalls of one cell overlap the work of five others; larger cells take two CTAs of 512 threads per SM.
constexpr int kDenseSmall = 768;

template <int kM>
__host__ __device__ constexpr size_t dense_smem_bytes()
{
    return (size_t)kM * (16 + 2) + (size_t)(kMaxQ3 + 1) * 4 + (size_t)kMaxQ3 * (4 + 2) +
           (size_t)kMaxQ * kMaxQ * 4 + 256;
}

template <int kM>
__device__ __forceinline__ DenseSmem carve(unsigned char* base)
{
    DenseSmem s;
    size_t off = 0;
    s.P = (float4*)(base + off);            off += (size_t)kM * 16;
    s.misc = (int*)(base + off);
    s.nbj0 = s.misc + 8;
    s.nbpref = s.misc + 36;
    off += 256;
    s.sstart = (int*)(base + off);          off += (size_t)(kMaxQ3 + 1) * 4;
    s.lpar = (int*)(base + off);            off += (size_t)kMaxQ3 * 4;
    s.rowng = (unsigned*)(base + off);      off += (size_t)kMaxQ * kMaxQ * 4;
    s.skey = (unsigned short*)(base + off); off += (size_t)kM * 2;
    s.ng = (unsigned short*)(base + off);
    return s;
}

// shared-memory union-find over the sub-cells (hook the larger root onto
// the smaller, like the global one); volatile so that a retry re-reads
// what other threads hooked
// Paths strictly decrease and every failed CAS means another hook
// succeeded, so both loops end within kMaxQ3 steps; the caps only turn
// a corrupted forest into a reported error instead of a hang.
__device__ __forceinline__ int lfind(int* lpar_, int x, int* err)
{
    volatile int* lpar = lpar_;
    int p = lpar[x];
    for (int step = 0; p != x; ++step) {
        int gp = lpar[p];
        if (gp == p)
            return p;
        if (gp > p || step > kMaxQ3) {
            atomicOr(err, kErrInternal);
            return p;
        }
        lpar[x] = gp;
        x = gp;
        p = lpar[x];
    }
    return x;
}

__device__ __forceinline__ void lunion(int* lpar, int a, int b, int* err)
{
    for (int it = 0; it <= 2 * kMaxQ3; ++it) {
        a = lfind(lpar, a, err);
        b = lfind(lpar, b, err);
        if (a == b)
            return;
        int hi = a > b ? a : b, lo = a > b ? b : a;
        if (atomicCAS(lpar + hi, hi, lo) == hi)
            return;
    }
    atomicOr(err, kErrInternal);
}

// Load cell [c0, c0+m) into shared memory in sub-cell order, with the
// sub-cell starts.  (ox, oy, oz) = fine coordinates of the cell's corner.
// kSort: the slots are not in sub-cell order yet; they are put in it here,
// also in global memory (no other kernel or CTA reads these slots meanwhile).
template <bool kSort, int kM, int kThreads>
__device__ __forceinline__ void build_cell(const DenseSmem& S, float4* __restrict__ sorted,
                                           int* __restrict__ minorig, int c0, int m, const BoxDev& b, int ox, int oy,
                                           int oz, int* err)
{
    constexpr int kPer = kM / kThreads;
    static_assert(kPer * kThreads == kM, "particles per thread");
    const int q = b.q, q3 = q * q * q;
    for (int a = threadIdx.x; a <= q3; a += kThreads) S.sstart[a] = 0;
    __syncthreads();
    float4 p[kPer];
    int key[kPer];
#pragma unroll
    for (int r = 0; r < kPer; ++r) {
        const int k = r * kThreads + threadIdx.x;
        key[r] = -1;
        if (k < m)
            p[r] = sorted[c0 + k];
    }
#pragma unroll
    for (int r = 0; r < kPer; ++r) {
        const int k = r * kThreads + threadIdx.x;
        if (k < m) {
            int sx = fine_coord(p[r].x, b) - ox, sy = fine_coord(p[r].y, b) - oy, sz = fine_coord(p[r].z, b) - oz;
            bool ok = sx >= 0 && sx < q && sy >= 0 && sy < q && sz >= 0 && sz < q;
            if (!ok) {
                atomicOr(err, kErrInternal);
                sx = sx < 0 ? 0 : (sx >= q ? q - 1 : sx);
                sy = sy < 0 ? 0 : (sy >= q ? q - 1 : sy);
                sz = sz < 0 ? 0 : (sz >= q ? q - 1 : sz);
            }
            key[r] = (sz * q + sy) * q + sx;
            atomicAdd(S.sstart + key[r], 1);
        }
    }
    __syncthreads();
    if (threadIdx.x < 32) {            // exclusive scan of q3 + 1 counts by one warp
        int carry = 0;
        for (int base = 0; base <= q3; base += 32) {
            int i = base + threadIdx.x;
            int v = i <= q3 ? S.sstart[i] : 0;
            int x = v;
            for (int o = 1; o < 32; o <<= 1) {
                int y = __shfl_up_sync(kFull, x, o);
                if ((int)threadIdx.x >= o) x += y;
            }
            if (i <= q3) S.sstart[i] = carry + x - v;
            if (kSort && i < q3) S.lpar[i] = carry + x - v;      // cursor
            carry += __shfl_sync(kFull, x, 31);
        }
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kPer; ++r) {
        if (key[r] < 0)
            continue;
        int at = r * kThreads + threadIdx.x;
        if constexpr (kSort)
            at = atomicAdd(S.lpar + key[r], 1);
        S.P[at] = p[r];
        S.skey[at] = (unsigned short)key[r];
    }
    __syncthreads();
    if constexpr (kSort) {
        for (int k = threadIdx.x; k < m; k += kThreads) {
            const float4 v = S.P[k];
            sorted[c0 + k] = v;
            minorig[c0 + k] = __float_as_int(v.w);
        }
    }
}

// The fullest sub-cell (the smallest of several), in S.misc[1].
template <int kThreads>
__device__ __forceinline__ int fullest(const DenseSmem& S, int q3)
{
    if (threadIdx.x == 0)
        S.misc[1] = 0;
    __syncthreads();
    int best = 0;
    for (int a = threadIdx.x; a < q3; a += kThreads)
        best = max(best, ((S.sstart[a + 1] - S.sstart[a]) << 11) | (kMaxQ3 - a));
    best = (int)__reduce_max_sync(kFull, (unsigned)best);
    if ((threadIdx.x & 31) == 0)
        atomicMax(S.misc + 1, best);
    __syncthreads();
    return kMaxQ3 - (S.misc[1] & 2047);
}

// The rows of sub-cells within +-2 of fine coordinates (rx, ry, rz): lane
// l < 25 gets row (dz, dy) = (l / 5 - 2, l % 5 - 2) as a range of P, and
// whether the row holds a sub-cell outside the main group.  (ux, uy, uz) is
// the searching position inside its own fine cell and reach2 bounds the
// squared distance in fine units: sub-cells farther away are left out
// (reach2 = infinity keeps all).
__device__ __forceinline__ void window_row(const DenseSmem& S, int q, int rx, int ry, int rz, float ux, float uy,
                                           float uz, float reach2, int lane, int& start, int& count, bool& outside)
{
    start = 0;
    count = 0;
    outside = false;
    const int dz = lane / 5 - 2, dy = lane % 5 - 2;
    const int z = rz + dz, y = ry + dy;
    int x0 = max(rx - 2, 0), x1 = min(rx + 2, q - 1);
    if (lane < 25 && z >= 0 && z < q && y >= 0 && y < q && x0 <= x1) {
        const float gz = dz < 0 ? (float)(-dz - 1) + uz : (dz > 0 ? (float)(dz - 1) + (1.f - uz) : 0.f);
        const float gy = dy < 0 ? (float)(-dy - 1) + uy : (dy > 0 ? (float)(dy - 1) + (1.f - uy) : 0.f);
        const float g2 = gy * gy + gz * gz;
        if (g2 <= reach2) {
            // the ends of the row, one sub-cell at a time (at most 2 below and 2 above rx)
            while (x0 <= x1 && x0 < rx) {
                const float gx = (float)(rx - x0 - 1) + ux;
                if (gx * gx + g2 <= reach2)
                    break;
                ++x0;
            }
            while (x0 <= x1 && x1 > rx) {
                const float gx = (float)(x1 - rx - 1) + (1.f - ux);
                if (gx * gx + g2 <= reach2)
                    break;
                --x1;
            }
            if (x0 <= x1) {
                const int row = z * q + y;
                start = S.sstart[row * q + x0];
                count = S.sstart[row * q + x1 + 1] - start;
                outside = (S.rowng[row] & ((2u << x1) - (1u << x0))) != 0u;
            }
        }
    }
}

// fine coordinates of pj relative to the corner (ox, oy, oz), unwrapped
// into the window next to the cell (the box has at least 3 cells per axis)
__device__ __forceinline__ bool rel_fine(float4 pj, const BoxDev& b, int ox, int oy, int oz,
                                         int& rx, int& ry, int& rz)
{
    const int q = b.q, nf = b.nf;
    rx = fine_coord(pj.x, b) - ox;
    ry = fine_coord(pj.y, b) - oy;
    rz = fine_coord(pj.z, b) - oz;
    rx = rx < -2 ? rx + nf : (rx > q + 1 ? rx - nf : rx);
    ry = ry < -2 ? ry + nf : (ry > q + 1 ? ry - nf : ry);
    rz = rz < -2 ? rz + nf : (rz > q + 1 ? rz - nf : rz);
    return rx >= -2 && rx <= q + 1 && ry >= -2 && ry <= q + 1 && rz >= -2 && rz <= q + 1;
}

// place of x inside its fine cell
__device__ __forceinline__ float fine_frac(float x, const BoxDev& b)
{
    return __fmul_rn(x, b.inv_hf) - (float)fine_coord(x, b);
}

// gap from fine coordinate r (+ u) to [0, q)
__device__ __forceinline__ float cell_gap(int r, float u, int q)
{
    return r < 0 ? (float)(-r - 1) + (1.f - u) : (r >= q ? (float)(r - q) + u : 0.f);
}

// 32 particles outside the cell, one per lane (slot j, position pj), against
// the cell in shared memory.  S.lpar[a] = a node of the global forest in the
// group of sub-cell a, `main` that of the fullest sub-cell.  Particles out of
// the cell's reach drop out; for the others, one after the other, the warp
// tests the candidates of the window, those of the main group only while the
// particle's root differs from the group's.  Equal roots prove one group, and
// a lane whose root equals that of a lane already linked to the main group
// needs no test of its own; the unions with the main group run at the end,
// one per lane, side by side.
template <bool kVar>
__device__ __forceinline__ void link_outside(const DenseSmem& S, int* parent, const BoxDev& b, float4 pj, int j,
                                             bool valid, int ox, int oy, int oz, int main, bool single, int lane,
                                             const UfArgs& uf)
{
    const int q = b.q;
    int rx = 0, ry = 0, rz = 0;
    bool near = valid && rel_fine(pj, b, ox, oy, oz, rx, ry, rz);
    if (near) {
        const float gx = cell_gap(rx, fine_frac(pj.x, b), q), gy = cell_gap(ry, fine_frac(pj.y, b), q),
                    gz = cell_gap(rz, fine_frac(pj.z, b), q);
        near = gx * gx + gy * gy + gz * gz <= b.reach2;
    }
    if (!__any_sync(kFull, near))
        return;
    int rj = -1, rm = -2;
    if (near) {
        rj = j;
        rm = main;
        if constexpr (kVar) {
            rj = ufind<kVar>(parent, rj, uf);
            rm = ufind<kVar>(parent, rm, uf);
        } else {
            uf_find2(parent, rj, rm, uf.err);
        }
    }
    unsigned want_main = __ballot_sync(kFull, near && rj != rm);
    const unsigned want_rest = single ? 0u : __ballot_sync(kFull, near);
    bool hit_main = false;
    for (unsigned todo = want_main | want_rest; todo; todo &= want_main | want_rest) {
        const int l = __ffs(todo) - 1;
        todo &= todo - 1u;
        float4 p;
        p.x = __shfl_sync(kFull, pj.x, l);
        p.y = __shfl_sync(kFull, pj.y, l);
        p.z = __shfl_sync(kFull, pj.z, l);
        p.w = 0.f;
        const int px = __shfl_sync(kFull, rx, l), py = __shfl_sync(kFull, ry, l), pz = __shfl_sync(kFull, rz, l);
        int start, count;
        bool outside;
        window_row(S, q, px, py, pz, fine_frac(p.x, b), fine_frac(p.y, b), fine_frac(p.z, b), b.reach2, lane, start,
                   count, outside);
        bool main_open = (want_main >> l) & 1u;
        const bool rest_open = !single && __any_sync(kFull, outside);
        if (!main_open && !rest_open)
            continue;
        const int pref = warp_incl(count, lane) - count;
        const int total = __shfl_sync(kFull, pref + count, 31);
        bool linked_main = false;
        for (int cb = 0; cb < total && (main_open || rest_open); cb += kWarp) {
            const int t = cb + lane;
            const int o = owner_lane(pref, t < total ? t : total - 1);
            const int at = __shfl_sync(kFull, start, o) + (t - __shfl_sync(kFull, pref, o));
            bool hit = false;
            int node = -1;
            if (t < total) {
                node = S.lpar[S.skey[at]];
                if (node == main ? main_open : rest_open)
                    hit = linked_ool(p, S.P[at], b);
            }
            if (__any_sync(kFull, hit && node == main)) {
                linked_main = true;
                main_open = false;
            }
            // groups other than the main one: few, united at once
            for (unsigned rest = __ballot_sync(kFull, hit && node != main); rest;) {
                const int lead = __ffs(rest) - 1;
                const int group = __shfl_sync(kFull, node, lead);
                const int jl = __shfl_sync(kFull, j, l);
                if (lane == lead)
                    uunion<kVar>(parent, jl, group, uf);
                rest &= ~__ballot_sync(kFull, hit && node == group);
            }
        }
        if (linked_main) {
            if (lane == l)
                hit_main = true;
            want_main &= ~__ballot_sync(kFull, rj == __shfl_sync(kFull, rj, l));
        }
    }
    if (hit_main)
        uunion<kVar>(parent, rj, main, uf);
    __syncwarp();
}

__device__ __forceinline__ int64_t nbr_cell(const BoxDev& b, int cx, int cy, int cz, int dx, int dy,
                                            int dz)
{
    return cell_key(b, wrap_cell(cx + dx, b.nc), wrap_cell(cy + dy, b.nc), wrap_cell(cz + dz, b.nc));
}

// prefix of S.nbpref[1..26] holding counts -> exclusive starts; one warp
__device__ __forceinline__ void neighbour_prefix(const DenseSmem& S)
{
    if (threadIdx.x < 32) {
        int lane = threadIdx.x;
        int v = (lane >= 1 && lane <= 26) ? S.nbpref[lane] : 0;
        int x = v;
        for (int o = 1; o < 32; o <<= 1) {
            int y = __shfl_up_sync(kFull, x, o);
            if (lane >= o) x += y;
        }
        if (lane <= 26) S.nbpref[lane] = x;    // nbpref[0] = 0, nbpref[k] = sum of counts < k
    }
}

// the neighbour k whose particles contain flat index t
__device__ __forceinline__ int neighbour_of(const DenseSmem& S, int t)
{
    int lo = 0, hi = 25;
    while (lo < hi) {
        int mid = (lo + hi + 1) >> 1;
        if (S.nbpref[mid] <= t) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// Every particle of the neighbour table (nbj0, nbpref), 32 per warp.
template <bool kVar, int kThreads>
__device__ __forceinline__ void link_neighbours(const DenseSmem& S, const Work& w, const BoxDev& b, int ox, int oy,
                                                int oz, int main, bool single, const UfArgs& uf)
{
    const int lane = threadIdx.x & 31;
    const int total = S.nbpref[26];
    for (int base = (threadIdx.x >> 5) * kWarp; base < total; base += kThreads) {
        const int t = base + lane;
        const bool valid = t < total;
        int j = 0;
        float4 pj = make_float4(0.f, 0.f, 0.f, 0.f);
        if (valid) {
            const int k = neighbour_of(S, t);
            j = S.nbj0[k] + (t - S.nbpref[k]);
            FOF_DCHECK_SLOT(j, b, uf.err);
            pj = w.sorted[j];
        }
        link_outside<kVar>(S, w.parent, b, pj, j, valid, ox, oy, oz, main, single, lane, uf);
    }
}

template <bool kVar, int kLo, int kM, int kThreads, int kBlocks>
__global__ void __launch_bounds__(kThreads, kBlocks) k_dense_self(Geometry g, Work w, int dense_min,
                                                              UfArgs uf)
{
    // beside k_link, which links no particle of a dense cell, and beside the
    // other size class: their unions are the same atomic ones.  k_link reads the
    // records that are put in sub-cell order here, but only to see which cell they
    // are in: every record written there is of the same cell, and so is any mix
    // of two, since a cell is a product of intervals.
    pdl_join(w.status->passed_on + kPassCellOrder);
    pdl_trigger();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const DenseSmem S = carve<kM>(smem_raw);
    int* err = uf.err;
    const int lane = threadIdx.x & 31;
    const int n_dense = *w.n_dense;
    for (int it = blockIdx.x; it < n_dense; it += gridDim.x) {
        const int64_t key = w.dense_list[it];
        const int c0 = w.cell_start[key], c1 = w.cell_start[key + 1];
        const int m = c1 - c0;
        if (m <= kLo || m > kM)
            continue;                             // the other size class's cell (block-uniform)
        const BoxDev& b = g.boxes[box_of_warp(g.box_p0, g.nbox, c0, threadIdx.x & 31)];
        const int q = b.q, q3 = q * q * q;
        const float4 p0 = w.sorted[c0];
        const int cx = cell_coord(p0.x, b), cy = cell_coord(p0.y, b), cz = cell_coord(p0.z, b);
        const int ox = cx * q, oy = cy * q, oz = cz * q;
        // neighbour table, filled while the cell is built
        if (threadIdx.x < 26) {
            int k = threadIdx.x;
            int code = k < 13 ? k : k + 1;            // the 26 offsets, centre skipped
            int64_t nk = nbr_cell(b, cx, cy, cz, code % 3 - 1, (code / 3) % 3 - 1, code / 9 - 1);
            int j0 = w.cell_start[nk], j1 = w.cell_start[nk + 1];
            S.nbj0[k] = j0;
            S.nbpref[k + 1] = (j1 > j0 && !is_sub(j1 - j0, b, dense_min)) ? j1 - j0 : 0;
            if (k == 0)
                S.nbpref[0] = 0;
        }
        __syncthreads();                          // every thread has read p0 (build_cell moves the slots)
        build_cell<true, kM, kThreads>(S, w.sorted, w.minorig, c0, m, b, ox, oy, oz, err);
        neighbour_prefix(S);
        for (int a = threadIdx.x; a < q3; a += kThreads) S.lpar[a] = a;
        const int top = fullest<kThreads>(S, q3);
        // sub-cells that share a face: joined at their first linked pair
        for (int item = threadIdx.x; item < 3 * q3; item += kThreads) {
            const int a = item / 3, o = item - 3 * a;
            const int ax = a % q, ay = (a / q) % q, az = a / (q * q);
            if ((o == 0 ? ax : (o == 1 ? ay : az)) == q - 1)
                continue;
            const int bb = a + (o == 0 ? 1 : (o == 1 ? q : q * q));
            const int a0 = S.sstart[a], a1 = S.sstart[a + 1];
            const int b0 = S.sstart[bb], b1 = S.sstart[bb + 1];
            if (a0 == a1 || b0 == b1 || lfind(S.lpar, a, err) == lfind(S.lpar, bb, err))
                continue;
            bool done = false;
            for (int u = a0; u < a1 && !done; ++u) {
                const float4 pu = S.P[u];
                for (int v = b0; v < b1; ++v)
                    if (linked_ool(pu, S.P[v], b)) {
                        lunion(S.lpar, a, bb, err);
                        done = true;
                        break;
                    }
            }
        }
        if (threadIdx.x == 0)
            S.misc[0] = 0;
        for (int row = threadIdx.x; row < q * q; row += kThreads) S.rowng[row] = 0u;
        __syncthreads();
        // the sub-cells outside the fullest one's group
        int main = lfind(S.lpar, top, err);
        for (int a = threadIdx.x; a < q3; a += kThreads)
            if (S.sstart[a + 1] > S.sstart[a] && lfind(S.lpar, a, err) != main)
                S.ng[atomicAdd(S.misc, 1)] = (unsigned short)a;
        __syncthreads();
        const int n_ng = S.misc[0];
        // each of them against its whole window, one warp per sub-cell; pairs
        // of sub-cells inside the group cannot change anything
        for (int t = threadIdx.x >> 5; t < n_ng; t += kThreads / kWarp) {
            const int a = S.ng[t];
            int start, count;
            bool outside;
            window_row(S, q, a % q, (a / q) % q, a / (q * q), 0.f, 0.f, 0.f, INFINITY, lane, start, count, outside);
            const int pref = warp_incl(count, lane) - count;
            const int total = __shfl_sync(kFull, pref + count, 31);
            const int a0 = S.sstart[a], a1 = S.sstart[a + 1];
            for (int cb = 0; cb < total; cb += kWarp) {
                const int u = cb + lane;
                const int o = owner_lane(pref, u < total ? u : total - 1);
                const int at = __shfl_sync(kFull, start, o) + (u - __shfl_sync(kFull, pref, o));
                if (u < total) {
                    const int bb = S.skey[at];
                    if (lfind(S.lpar, a, err) != lfind(S.lpar, bb, err)) {
                        const float4 pv = S.P[at];
                        for (int v = a0; v < a1; ++v)
                            if (linked_ool(S.P[v], pv, b)) {
                                lunion(S.lpar, a, bb, err);
                                break;
                            }
                    }
                }
                __syncwarp();
            }
        }
        __syncthreads();
        // the cell's forest goes to global memory; roots are smallest slots
        main = lfind(S.lpar, top, err);
        int differs = 0;
        for (int t = threadIdx.x; t < n_ng; t += kThreads) {
            const int a = S.ng[t];
            if (lfind(S.lpar, a, err) != main) {
                differs = 1;
                atomicOr(S.rowng + a / q, 1u << (a % q));
            }
        }
        for (int k = threadIdx.x; k < m; k += kThreads)
            w.parent[c0 + k] = c0 + S.sstart[lfind(S.lpar, S.skey[k], err)];
        __threadfence();
        const bool single = !__syncthreads_or(differs);
        main = c0 + S.sstart[main];
        // from here on S.lpar holds each sub-cell's root slot
        for (int a = threadIdx.x; a < q3; a += kThreads) {
            const int a0 = S.sstart[a];
            if (S.sstart[a + 1] > a0)
                S.lpar[a] = single ? main : w.parent[c0 + a0];
        }
        if (threadIdx.x == 0)
            w.dense_root[c0 / dense_min] = single ? main : -1;
        __syncthreads();
        // particles of the 26 neighbours that are not subdivided, all at
        // once: every pair of them with this cell belongs to this task
        link_neighbours<kVar, kThreads>(S, w, b, ox, oy, oz, main, single, uf);
        __syncthreads();
    }
    pdl_wait();
}

template <bool kVar, int kLo, int kM, int kThreads, int kBlocks>
__global__ void __launch_bounds__(kThreads, kBlocks) k_dense_pairs(Geometry g, Work w, int dense_min,
                                                               UfArgs uf)
{
    // after dense_self; the second size class beside the first
    if (kLo == 0) {
        pdl_wait();
        pdl_pass_on(w.status->passed_on + kPassDenseOrder);
    } else {
        pdl_join(w.status->passed_on + kPassDenseOrder);
        pdl_trigger();
    }
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const DenseSmem S = carve<kM>(smem_raw);
    int* err = uf.err;
    const int n_dense = *w.n_dense;
    for (int it = blockIdx.x; it < n_dense; it += gridDim.x) {
        const int64_t key = w.dense_list[it];
        const int c0 = w.cell_start[key], c1 = w.cell_start[key + 1];
        const int m = c1 - c0;
        if (m <= kLo || m > kM)
            continue;                             // the other size class's cell (block-uniform)
        const BoxDev& b = g.boxes[box_of_warp(g.box_p0, g.nbox, c0, threadIdx.x & 31)];
        const int q = b.q, q3 = q * q * q;
        const float4 p0 = w.sorted[c0];
        const int cx = cell_coord(p0.x, b), cy = cell_coord(p0.y, b), cz = cell_coord(p0.z, b);
        const int ox = cx * q, oy = cy * q, oz = cz * q;
        const int ua = w.dense_root[c0 / dense_min];
        // the 13 forward neighbours that are subdivided and not yet joined
        if (threadIdx.x < 32) {
            int k = threadIdx.x;
            int cnt = 0;
            if (k < 13) {
                int dx, dy, dz;
                fwd_offset(k, dx, dy, dz);
                int64_t nk = nbr_cell(b, cx, cy, cz, dx, dy, dz);
                int j0 = w.cell_start[nk], j1 = w.cell_start[nk + 1];
                if (is_sub(j1 - j0, b, dense_min) && !is_big(j1 - j0, b)) {
                    int ub = w.dense_root[j0 / dense_min];
                    const bool both = ua >= 0 && ub >= 0;
                    cnt = (both && ufind<kVar>(w.parent, ua, uf) == ufind<kVar>(w.parent, ub, uf)) ? 0 : j1 - j0;
                }
                S.nbj0[k] = j0;
            }
            if (k >= 1 && k <= 26)
                S.nbpref[k] = 0;
            __syncwarp();
            if (k < 13)
                S.nbpref[k + 1] = cnt;
            if (k == 0)
                S.nbpref[0] = 0;
            __syncwarp();
            neighbour_prefix(S);
        }
        __syncthreads();
        const int total = S.nbpref[26];
        __syncthreads();                          // everyone has read the table's total
        if (total == 0)
            continue;                             // block-uniform
        build_cell<false, kM, kThreads>(S, w.sorted, w.minorig, c0, m, b, ox, oy, oz, err);
        const int top = fullest<kThreads>(S, q3);
        for (int row = threadIdx.x; row < q * q; row += kThreads) S.rowng[row] = 0u;
        for (int a = threadIdx.x; a < q3; a += kThreads)
            if (S.sstart[a + 1] > S.sstart[a])
                S.lpar[a] = ua >= 0 ? ua : ufind<kVar>(w.parent, c0 + S.sstart[a], uf);
        __syncthreads();
        const int main = S.lpar[top];
        int differs = 0;
        for (int a = threadIdx.x; a < q3; a += kThreads)
            if (S.sstart[a + 1] > S.sstart[a] && S.lpar[a] != main) {
                differs = 1;
                atomicOr(S.rowng + a / q, 1u << (a % q));
            }
        const bool single = !__syncthreads_or(differs);
        link_neighbours<kVar, kThreads>(S, w, b, ox, oy, oz, main, single, uf);
        __syncthreads();
    }
    if (kLo != 0)
        pdl_wait();
}

}  // namespace

// Up to this many particles dense cells are fewer than SMs, or a few per SM,
// and what counts is the chain of one cell: one launch with 32 warps per cell
// of either size class (dense_self + dense_pairs against the two classes of 8
// and 16 warps, us: 60,000 particles 66 and 120, 2 million 107 and 129, 3
// million 169 and 187, 4 million 178 and 163).
bool dense_one_launch(int64_t total_n)
{
    return total_n <= 3 << 20;
}

template <bool kVar, int kLo, int kM, int kThreads, int kBlocks>
cudaError_t configure_dense()
{
    cudaError_t e = cudaFuncSetAttribute(k_dense_self<kVar, kLo, kM, kThreads, kBlocks>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dense_smem_bytes<kM>());
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(k_dense_pairs<kVar, kLo, kM, kThreads, kBlocks>,
                                cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dense_smem_bytes<kM>());
}

template <bool kVar, int kLo, int kM, int kThreads, int kBlocks>
cudaError_t run_dense(const Geometry& g, const Work& w, int dense_min, const UfArgs& uf, bool pairs, cudaStream_t s)
{
    const int blocks = sm_count() * kBlocks;
    if (pairs && kLo == 0)
        return launch_next(g.total_n, k_dense_pairs<kVar, kLo, kM, kThreads, kBlocks>, blocks, kThreads,
                           dense_smem_bytes<kM>(), s, g, w, dense_min, uf);
    return launch_beside(g.total_n, pairs ? k_dense_pairs<kVar, kLo, kM, kThreads, kBlocks>
                                          : k_dense_self<kVar, kLo, kM, kThreads, kBlocks>,
                         blocks, kThreads, dense_smem_bytes<kM>(), s, g, w, dense_min, uf);
}

template <bool kVar>
cudaError_t configure_all()
{
    cudaError_t e;
    if ((e = configure_dense<kVar, 0, kDenseSmall, 256, 6>()) != cudaSuccess) return e;
    if ((e = configure_dense<kVar, kDenseSmall, kDenseMax, 512, 2>()) != cudaSuccess) return e;
    return configure_dense<kVar, 0, kDenseMax, 1024, 1>();
}

template <bool kVar>
cudaError_t run_all(const Geometry& g, const Work& w, int dense_min, const UfArgs& uf, bool pairs, cudaStream_t s)
{
    if (dense_one_launch(g.total_n))
        return run_dense<kVar, 0, kDenseMax, 1024, 1>(g, w, dense_min, uf, pairs, s);
    cudaError_t e = run_dense<kVar, 0, kDenseSmall, 256, 6>(g, w, dense_min, uf, pairs, s);
    return e != cudaSuccess ? e : run_dense<kVar, kDenseSmall, kDenseMax, 512, 2>(g, w, dense_min, uf, pairs, s);
}

int dense_launches(const Geometry& g, int dense_min)
{
    if (g.max_split_n < dense_min)
        return 0;                               // no cell can be larger than its box
    return dense_one_launch(g.total_n) ? 1 : 2;
}

cudaError_t launch_dense(const Geometry& g, const Work& w, int dense_min, const UfArgs& uf, bool pairs,
                         cudaStream_t s)
{
    if (dense_launches(g, dense_min) == 0)
        return cudaSuccess;
    // the shared-memory opt-in is per device; setting it again is harmless
    static bool configured[64] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64 || !configured[dev]) {
        if ((e = configure_all<false>()) != cudaSuccess) return e;
        if ((e = configure_all<true>()) != cudaSuccess) return e;
        if (dev >= 0 && dev < 64) configured[dev] = true;
    }
    return uf.var ? run_all<true>(g, w, dense_min, uf, pairs, s) : run_all<false>(g, w, dense_min, uf, pairs, s);
}

}  // namespace fofgpu
