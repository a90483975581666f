// Self- and pair-cell linking (the paper's "self" and "pair" tasks over
// cells, Sec. 3.1, Fig. 1), on the binned particle order.
//
// A warp takes 32 consecutive binned particles (one per lane).  For every
// particle the cell itself and its 13 forward neighbours (half of the
// periodic 26-neighbourhood) are searched, so each unordered cell pair is
// visited once; inside the own cell only partners with a larger slot are
// tested.
//
// Cells with at least team_min particles are linked by the warp as a
// team: the lanes that belong to the cell keep their current root, the
// candidates of the neighbour cells are loaded 32 at a time (coalesced
// float4) and filtered by the team's bounding box, the survivors are
// gathered in shared memory, and for up to 32 of them at once their roots
// are taken and
//   * the whole buffer is skipped when all roots on both sides agree,
//   * a pair is skipped when the member's root equals the candidate's,
// which is exact because groups only ever merge: two particles whose roots
// were once equal stay in one group.  Sparse particles search on their own.
//
// Cells that the dense kernels link (subdivided cells, fof_dense.cu) are
// skipped here, as own cells and as neighbours: every pair that involves
// one of them belongs to a dense task.  Where the box has sub-cells, a
// linked pair is at most 2 fine cells apart on each axis, so a particle
// only visits the forward neighbours across faces it lies within 2 fine
// cells of (exact pruning of the stencil).
//
// Linked pairs are merged with the CAS union of fof_internal.cuh.
#include "fof_internal.cuh"

namespace fofgpu {

namespace {

struct Cell {
    int cx, cy, cz;
};

// the cell of a window's particle (k_link: x | y << 16, z)
__device__ __forceinline__ Cell cell_at(const int4& at)
{
    return Cell{at.x & 0xffff, at.x >> 16, at.y};
}

// cell_key with the Morton spreading of the in-brick coordinates (< 16)
// read from a shared-memory table instead of computed
__device__ __forceinline__ int64_t cell_key_tab(const BoxDev& b, int cx, int cy, int cz, const uint32_t* tab)
{
    const int m = b.r - 1;
    const int64_t r3 = (int64_t)b.r * b.r * b.r;
    return b.cell0 + brick_local(b, cx, cy, cz) * r3 + (tab[cx & m] | (tab[cy & m] << 1) | (tab[cz & m] << 2));
}

__device__ __forceinline__ int64_t nbr_key_tab(const BoxDev& b, const Cell& c, int k, const uint32_t* tab)
{
    int dx, dy, dz;
    fwd_offset(k, dx, dy, dz);
    return cell_key_tab(b, wrap_cell(c.cx + dx, b.nc), wrap_cell(c.cy + dy, b.nc), wrap_cell(c.cz + dz, b.nc),
                        tab);
}

__device__ __forceinline__ int64_t nbr_key(const BoxDev& b, const Cell& c, int k)
{
    int dx, dy, dz;
    fwd_offset(k, dx, dy, dz);
    return cell_key(b, wrap_cell(c.cx + dx, b.nc), wrap_cell(c.cy + dy, b.nc),
                    wrap_cell(c.cz + dz, b.nc));
}

// Neighbour k duplicates the own cell or an earlier neighbour (only when
// fewer than 3 cells per axis).
__device__ __forceinline__ bool nbr_duplicate(const BoxDev& b, const Cell& c, int k)
{
    if (b.nc >= 3)
        return false;
    int64_t key = nbr_key(b, c, k);
    if (key == cell_key(b, c.cx, c.cy, c.cz))
        return true;
    for (int q = 0; q < k; ++q)
        if (nbr_key(b, c, q) == key)
            return true;
    return false;
}

// The forward neighbours particle p can reach.  With sub-cells (q > 1) a
// linked pair is at most 2 fine cells apart on each axis, so p needs the
// neighbour across a face only when it sits within 2 fine cells of that
// face; without sub-cells every neighbour is kept.  Bit k = fwd_offset(k).
__device__ __forceinline__ unsigned reach_mask(const float4& p, const BoxDev& b, const Cell& c)
{
    if (b.q == 1)
        return 0x1fffu;
    const int q = b.q;
    const int lx = fine_coord(p.x, b) - c.cx * q;
    const int ly = fine_coord(p.y, b) - c.cy * q;
    const int lz = fine_coord(p.z, b) - c.cz * q;
    const unsigned hx = lx >= q - 2, hy = ly >= q - 2, hz = lz >= q - 2;
    const unsigned wx = lx <= 1, wy = ly <= 1;
    // per axis, bit d+1 set when offset d in {-1, 0, +1} is reachable
    const unsigned xm = wx | 2u | (hx << 2);
    const unsigned ym = wy | 2u | (hy << 2);
    // k = 0..8: dz = +1, k = 3 (dy+1) + (dx+1); k = 9..11: dz = 0, dy = +1;
    // k = 12: dz = dy = 0, dx = +1  (the order of fwd_offset)
    unsigned m9 = ((ym & 1u) ? xm : 0u) | ((ym & 2u) ? xm << 3 : 0u) | ((ym & 4u) ? xm << 6 : 0u);
    return (hz ? m9 : 0u) | (hy ? xm << 9 : 0u) | (hx << 12);
}

// Bounding box of the team's particles.
struct TeamBox {
    float lx, ly, lz, hx, hy, hz;
};

__device__ __forceinline__ unsigned lanemask_lt()
{
    unsigned m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

// The index of the r-th (0-based) set bit of m (r < popc(m)).
__device__ __forceinline__ int nth_bit(unsigned m, int r)
{
    for (; r > 0; --r) m &= m - 1u;
    return __ffs(m) - 1;
}

// Per-warp staging of the team path: the team's members and one chunk of
// compacted candidates, in shared memory.
struct TeamStage {
    float4 mpos[32];    // member a = lane lo + a of the team: x, y, z, w = reach mask bits
    float4 cpos[32];    // candidate b of the chunk: x, y, z, w = neighbour index (13 = own cell)
    int mroot[32];      // a root of member a (possibly stale: equal roots prove one group)
    int croot[32];      // root snapshot of candidate b
    int cslot[32];      // slot of candidate b
    unsigned lmask[32]; // candidates of the chunk member a is linked to
    TeamBox box;        // the team's bounding box (kept here, not in registers)
    float4 shift[16];   // periodic shift of stream entry k's positions (k < 13)
};

constexpr int kLinkThreads = 256;
constexpr int kLinkWarps = kLinkThreads / 32;
constexpr int kLinkBlocks = 5;   // resident CTAs per SM (48 registers)
// The form that reads the union-find options at run time holds more, and spills
// at 48 (link phase, 134 million particles, with 5 and 4 CTAs: the defaults through
// it 14.9 and 14.4 ms, halving at every depth 16.2 and 15.6, no compression 17.7 and
// 17.2, random linking 15.0 and 14.5; full compression 17.6 and 18.2).
constexpr int kLinkVarBlocks = 4;
constexpr int kOwnCell = 13;     // stream index of a team's own cell (cells above kTeamSelfMax)

// The buffered candidates S.cpos/cslot[0..c) of a team against its m
// members: their roots; nothing more when all roots (members and
// candidates) agree, which is exact because groups only merge; otherwise
// the m x c pairs are tested lane-parallel (one pair per lane and step),
// skipping pairs whose roots already agree, linked pairs set bits in the
// member's link mask, and each member merges with the distinct candidate
// roots it links to.
template <bool kVar>
__device__ __forceinline__ void team_flush(TeamStage& S, int* __restrict__ parent, const BoxDev& b, int lane,
                                           int m, int first, int c, const UfArgs& uf)
{
    __syncwarp();
    int rj = -1;
    if (lane < c) {
        rj = ufind<kVar>(parent, S.cslot[lane], uf);
        S.croot[lane] = rj;
    }
    const int ref = S.mroot[0];
    const int mr = lane < m ? S.mroot[lane] : ref;
    if (__all_sync(kFull, mr == ref && (lane >= c || rj == ref)))
        return;
    __syncwarp();
    // pair t2 = a * c + bb, advanced by 32 per step without a division
    const int P = m * c;
    int a = lane / c;
    int bb = lane - a * c;
    const int qa = kWarp / c, qb = kWarp - qa * c;
    for (int t2 = lane; t2 < P; t2 += kWarp) {
        const float4 pm = S.mpos[a];
        const float4 qc = S.cpos[bb];
        const int kc = __float_as_int(qc.w);
        bool need = kc == kOwnCell ? S.cslot[bb] > first + a : ((__float_as_int(pm.w) >> kc) & 1);
        need = need && S.mroot[a] != S.croot[bb];
        if (need && linked(pm, qc, b))
            atomicOr(&S.lmask[a], 1u << bb);
        bb += qb;
        a += qa;
        if (bb >= c) {
            bb -= c;
            ++a;
        }
    }
    __syncwarp();
    if (lane < m) {
        unsigned links = S.lmask[lane];
        if (links) {
            int ri = S.mroot[lane];
            int last = -1;
            while (links) {
                const int u = __ffs(links) - 1;
                links &= links - 1u;
                const int rt = S.croot[u];
                if (rt != ri && rt != last) {
                    ri = uunion<kVar>(parent, ri, rt, uf);
                    last = rt;
                }
            }
            S.mroot[lane] = ri;
            S.lmask[lane] = 0u;
        }
    }
    __syncwarp();
}

// One team cell: its members (lanes lo .. lo+m-1 of the warp, contiguous
// slots first .. first+m-1) against every particle they can reach in the
// forward neighbour cells, as ONE stream of candidates, 32 per chunk.
// Lane k < 13 holds neighbour k's first slot and count (0 when the team does
// not reach it or the dense kernels own it); lane 13 the rest of the own
// cell when the cell is larger than kTeamSelfMax (k_team_self links the own
// pairs of smaller cells).  Candidates outside the team's bounding box + l_x
// are dropped; the survivors of successive chunks are gathered in shared
// memory (most are dropped, so a team usually fills one buffer of 32) and
// handed to team_flush when the buffer is full and at the end, so that the
// roots, pair tests and unions of several chunks take one round.
// kSplit: this warp takes chunks part, part + parts, ... of the stream.
template <bool kVar, bool kSplit>
__device__ __forceinline__ void team_cell(TeamStage& S, int* __restrict__ parent,
                                          const float4* __restrict__ sorted, const BoxDev& b, int lane,
                                          int lo, int m, int first, int j0k, int cntk,
                                          const TeamBox& tb, bool filter, int part, int parts,
                                          const UfArgs& uf)
{
    const int start_k = warp_incl(cntk, lane) - cntk;
    const int total = __shfl_sync(kFull, start_k + cntk, 31);
    int nb = 0;                                 // candidates in the buffer
    // one pass past the end of the stream flushes the rest (team_flush is
    // inlined once)
    const int step = kSplit ? parts * kWarp : kWarp;
    for (int cb = kSplit ? part * kWarp : 0; cb < total + step; cb += step) {
        const int t = cb + lane;
        bool jv = t < total;
        int k = 0;                              // last stream entry starting at or before t
#pragma unroll
        for (int half = 8; half; half >>= 1) {
            const int probe = k + half <= 13 ? k + half : 13;
            const int sm = __shfl_sync(kFull, start_k, probe);
            if (k + half <= 13 && sm <= t) k += half;
        }
        int j = __shfl_sync(kFull, j0k, k) + (t - __shfl_sync(kFull, start_k, k));
        float4 q = make_float4(0.f, 0.f, 0.f, 0.f);
        if (jv) {
            FOF_DCHECK_SLOT(j, b, uf.err);
            q = sorted[j];
            if (filter && k < kOwnCell) {
                const float4 sh = S.shift[k];
                const float xx = q.x + sh.x, yy = q.y + sh.y, zz = q.z + sh.z;
                const float gx = fmaxf(0.f, fmaxf(tb.lx - xx, xx - tb.hx));
                const float gy = fmaxf(0.f, fmaxf(tb.ly - yy, yy - tb.hy));
                const float gz = fmaxf(0.f, fmaxf(tb.lz - zz, zz - tb.hz));
                jv = gx * gx + gy * gy + gz * gz <= b.bb_reach2;
            }
        }
        const unsigned cand = __ballot_sync(kFull, jv);
        const int c = __popc(cand);
        if (nb + c > kWarp || (cb >= total && nb > 0)) {
            team_flush<kVar>(S, parent, b, lane, m, first, nb, uf);
            nb = 0;
        }
        if (jv) {
            const int r = nb + __popc(cand & lanemask_lt());
            S.cpos[r] = make_float4(q.x, q.y, q.z, __int_as_float(k));
            S.cslot[r] = j;
        }
        nb += c;
    }
}

// kSplit (small problems, of no more than two windows to a resident warp): a
// grid of one window per `parts` warps, neighbours in the grid, that all find
// its teams and their neighbour ranges and share the candidates (4,096
// particles, 8 warps and one: 23 and 36 us).  One window's chain counts there,
// so these have 64 registers (300,007 particles: 76 us, with 48: 87).
template <bool kVar, bool kSplit>
__global__ void __launch_bounds__(kLinkThreads, kSplit ? 4 : (kVar ? kLinkVarBlocks : kLinkBlocks))
    k_link(Geometry g, const float4* __restrict__ sorted, const int* __restrict__ cell_start, int* parent,
           int dense_min, int parts, int batch, Status* status, UfArgs uf)
{
    pdl_wait();
    pdl_pass_on(status->passed_on + kPassCellOrder);
    __shared__ TeamStage stage[kLinkWarps];
    __shared__ uint32_t spread_tab[16];
    if (threadIdx.x < 16)
        spread_tab[threadIdx.x] = spread3(threadIdx.x);
    __syncthreads();
    // each lane's binned record of the warp's next window, copied ahead
    // (cp.async) while the current window is linked; two buffers
    __shared__ float4 ahead[kLinkWarps][2][kWarp];
    // cell (x | y << 16, z) and box of each lane's particle, and the cell's end:
    // read back where they are needed, like the record, because registers are
    // what limits the warps per SM, and those the kernel (64 registers, 4 CTAs:
    // 35.8 ms on the 768^3 box; 48, 5, with 28 bytes spilled: 34.4; 40, 6, with 120
    // bytes: 37.0)
    __shared__ int4 where[kLinkWarps][kWarp];
    const int lane = threadIdx.x & 31;
    TeamStage& S = stage[threadIdx.x >> 5];
    float4* pf = &ahead[threadIdx.x >> 5][0][0];
    int4* at = &where[threadIdx.x >> 5][0];
    const unsigned total = (unsigned)g.total_n;         // slots fit in 31 bits
    const unsigned nwarps = (gridDim.x * kLinkWarps) / (kSplit ? parts : 1);   // a multiple of parts
    const unsigned warp = (blockIdx.x * kLinkWarps + (threadIdx.x >> 5)) / (kSplit ? parts : 1);
    const int part = kSplit ? (int)((blockIdx.x * kLinkWarps + (threadIdx.x >> 5)) % parts) : 0;
    S.lmask[lane] = 0u;
    __syncwarp();
    // Batches of windows (a power of two each): a warp's first by its number, the
    // others by a ticket drawn when the batch before is begun.  Windows of blobs
    // take ten times those of the background, and a warp sees too few of them to
    // even out (a fixed share per warp against tickets, this kernel: 2 million
    // particles 319 and 282 us, 453 million (768^3) 38.2 and 36.1 ms).
    const unsigned span = (kSplit ? 1u : (unsigned)batch) * kWarp;
    unsigned base = warp * span;
    unsigned drawn = 0u;                                // lane 0: the next batch's ticket
    if (base + lane < total)
        cp_async16(pf + lane, sorted + base + lane);
    cp_async_commit();
    if (!kSplit && lane == 0)
        drawn = atomicAdd(&status->link_ticket, 1u);

    for (int par = 0; base < total; par ^= 1) {
        const unsigned s = base + lane;
        const bool valid = s < total;
        int c0 = 0;
        bool sub = false, team = false;
        cp_async_wait_all();
        __syncwarp();                           // every lane's copy is in, and the last window's reads are done
        const float4* rec = pf + par * kWarp;
        if (valid) {
            // (with the warp's search of box_of_warp, this kernel: batch of 512
            // boxes 24.4 ms instead of 24.5, but the 768^3 box 34.2 instead of 33.9)
            const int bi = box_of(g.box_p0, g.nbox, s);
            const BoxDev& b = g.boxes[bi];
            const float4 p = rec[lane];
            const int cx = cell_coord(p.x, b), cy = cell_coord(p.y, b), cz = cell_coord(p.z, b);
            const int64_t self = cell_key_tab(b, cx, cy, cz, spread_tab);
            c0 = cell_start[self];
            const int c1 = cell_start[self + 1];
            at[lane] = make_int4(cx | (cy << 16), cz, bi, c1);
            sub = is_sub(c1 - c0, b, dense_min);
            team = !sub && (c1 - c0) >= b.team_min;
        }
        __syncwarp();
        unsigned tmask = __ballot_sync(kFull, team);

        // ---- team cells: the warp links each cell's members as a team ----
        while (tmask) {
            const int lead = __ffs(tmask) - 1;
            // (a cell that holds particles is told by its first slot)
            const int lead_c0 = __shfl_sync(kFull, c0, lead);
            const bool mine = team && c0 == lead_c0;
            const unsigned peers = __ballot_sync(kFull, mine);
            tmask &= ~peers;
            const int m = __popc(peers);          // members: lanes lead .. lead + m - 1
            const int4 lead_at = at[lead];
            const BoxDev& b = g.boxes[lead_at.z];
            const Cell tc = cell_at(lead_at);
            const float4 p = mine ? rec[lane] : make_float4(0.f, 0.f, 0.f, 0.f);
            // coordinates are finite and >= 0 (x + 0 turns -0 into +0), so
            // their bit patterns order like the values: one integer
            // reduction per bound
            TeamBox tbx;
            {
                const unsigned ux = __float_as_uint(p.x + 0.f), uy = __float_as_uint(p.y + 0.f),
                               uz = __float_as_uint(p.z + 0.f);
                const unsigned hi = 0x7f800000u;  // +inf: ignored by the minimum
                tbx.lx = __uint_as_float(__reduce_min_sync(kFull, mine ? ux : hi));
                tbx.ly = __uint_as_float(__reduce_min_sync(kFull, mine ? uy : hi));
                tbx.lz = __uint_as_float(__reduce_min_sync(kFull, mine ? uz : hi));
                tbx.hx = __uint_as_float(__reduce_max_sync(kFull, mine ? ux : 0u));
                tbx.hy = __uint_as_float(__reduce_max_sync(kFull, mine ? uy : 0u));
                tbx.hz = __uint_as_float(__reduce_max_sync(kFull, mine ? uz : 0u));
            }
            const unsigned reach = mine ? reach_mask(p, b, tc) : 0u;
            const unsigned team_reach = __reduce_or_sync(kFull, reach);
            if (mine) {
                S.mpos[lane - lead] = make_float4(p.x, p.y, p.z, __int_as_float((int)reach));
                S.mroot[lane - lead] = ufind<kVar>(parent, (int)s, uf);
            }
            const int first = (int)__shfl_sync(kFull, s, lead);
            const int cell_end = lead_at.w;
            const int cell_size = cell_end - lead_c0;
            // lane k < 13: neighbour k's range, if the team reaches it and
            // the dense kernels do not own it; lane 13: the own cell's
            // particles after the first member, for cells k_team_self skips
            int j0k = 0, cntk = 0;
            if (lane < 13 && ((team_reach >> lane) & 1u) && !nbr_duplicate(b, tc, lane)) {
                const int64_t nk = nbr_key_tab(b, tc, lane, spread_tab);
                const int j0 = cell_start[nk], j1 = cell_start[nk + 1];
                if (j1 > j0 && !is_sub(j1 - j0, b, dense_min)) {
                    j0k = j0;
                    cntk = j1 - j0;
                }
            } else if (lane == kOwnCell && cell_size > kTeamSelfMax) {
                j0k = first + 1;
                cntk = cell_end - first - 1;
            }
            if (lane < 13) {
                int dx, dy, dz;
                fwd_offset(lane, dx, dy, dz);
                S.shift[lane] = make_float4(tc.cx + dx < 0 ? -b.Lf : (tc.cx + dx >= b.nc ? b.Lf : 0.f),
                                            tc.cy + dy < 0 ? -b.Lf : (tc.cy + dy >= b.nc ? b.Lf : 0.f),
                                            tc.cz + dz >= b.nc ? b.Lf : 0.f, 0.f);
            }
            // Neighbours k < 9 lie one cell up in z.  A team cell there (sorted
            // by z bin in k_team_self) is cut to the prefix that the box filter
            // can pass: past it, the z gap to the team alone squares above
            // bb_reach2 (the filter's sum only adds non-negative terms).  A
            // slot after a probed one lies in its bin or a later one, so its
            // z is at least the probed z less the width of a bin (zb_width).
            // The cut is bracketed by two rounds of a 4-ary search: the three
            // lanes 3k, 3k+1, 3k+2 probe neighbour k's range at its quarters
            // in one round, and the cut keeps [0, hi): hi is the cell's end or
            // a probed slot past the cut, so every slot from hi on is past it
            // too (the box filter drops the few kept slots below hi).
            {
                const int gk = lane / 3, sub = lane - 3 * gk;
                const int src = gk < 9 ? gk : 0;
                const int jg = __shfl_sync(kFull, j0k, src), cg = __shfl_sync(kFull, cntk, src);
                const bool act = gk < 9 && b.nc >= 3 && cg >= kSortMin && cg >= b.team_min && cg <= kTeamSelfMax;
                const float sz = tc.cz + 1 >= b.nc ? b.Lf : 0.f;
                int lo = 0, hi = act ? cg : 0;
                for (int round = 0; round < 2 && __any_sync(kFull, lo < hi); ++round) {
                    const int len = hi - lo;
                    const int p0 = lo + len / 4, p1 = lo + len / 2, p2 = lo + (3 * len) / 4;
                    bool beyond = false;
                    if (lo < hi) {
                        const int pr = sub == 0 ? p0 : (sub == 1 ? p1 : p2);
                        const float d = __fsub_rn(__fadd_rn(__fsub_rn(sorted[jg + pr].z, b.zb_width), sz), tbx.hz);
                        beyond = d > 0.f && __fmul_rn(d, d) > b.bb_reach2;
                    }
                    const unsigned g3 = (__ballot_sync(kFull, beyond) >> (3 * src)) & 7u;
                    if (lo < hi) {
                        if (g3 & 1u) {
                            hi = p0;
                        } else if (g3 & 2u) {
                            lo = p0 + 1;
                            hi = p1;
                        } else if (g3 & 4u) {
                            lo = p1 + 1;
                            hi = p2;
                        } else {
                            lo = p2 + 1;
                        }
                    }
                }
                const int cut = __shfl_sync(kFull, hi, 3 * (lane < 9 ? lane : 0));   // lo <= answer <= hi
                if (lane < 9 && b.nc >= 3 && cntk >= kSortMin && cntk >= b.team_min && cntk <= kTeamSelfMax)
                    cntk = cut;
            }
            if (lane == 0)
                S.box = tbx;
            __syncwarp();
            team_cell<kVar, kSplit>(S, parent, sorted, b, lane, lead, m, first, j0k, cntk, S.box, b.nc >= 3, part,
                                    parts, uf);
        }

        // the next window, into the buffer that was read one window ago
        const bool last = ((base + kWarp) & (span - 1u)) == 0u;     // of its batch
        unsigned next = base + kWarp;
        if (last)
            next = kSplit ? base + nwarps * span : (nwarps + __shfl_sync(kFull, drawn, 0)) * span;
        if (next + lane < total)
            cp_async16(pf + (par ^ 1) * kWarp + lane, sorted + next + lane);
        cp_async_commit();

        // ---- sparse particles: their (particle, cell) items, then their
        // (particle, candidate) pairs, pooled across the warp ----
        const bool sparse = valid && !team && !sub;
        unsigned reach_s = 0u;
        int own_n = 0;
        if (sparse) {
            const int4 own_at = at[lane];
            const BoxDev& b = g.boxes[own_at.z];
            const Cell c = cell_at(own_at);
            reach_s = reach_mask(rec[lane], b, c);
            if (b.nc < 3)
                for (int k = 0; k < 13; ++k)
                    if (((reach_s >> k) & 1u) && nbr_duplicate(b, c, k))
                        reach_s &= ~(1u << k);
            own_n = own_at.w - (int)s - 1;
        }
        const int nit = sparse ? (own_n > 0) + __popc(reach_s) : 0;
        const int istart = warp_incl(nit, lane) - nit;
        const int T = __shfl_sync(kFull, istart + nit, 31);
        for (int ib = 0; ib < T; ib += kWarp) {
            // item ib + lane: owner o, and its candidate range [j0, j0 + cnt)
            const int t = ib + lane;
            const bool iv = t < T;
            const int o = owner_lane(istart, iv ? t : T - 1);
            const int r = t - __shfl_sync(kFull, istart, o);
            const int own_o = __shfl_sync(kFull, own_n, o);
            const unsigned reach_o = __shfl_sync(kFull, reach_s, o);
            int j0 = 0, cnt = 0;
            if (iv) {
                if (own_o > 0 && r == 0) {
                    j0 = (int)(base + o) + 1;
                    cnt = own_o;
                } else {
                    const int4 o_at = at[o];
                    const BoxDev& b = g.boxes[o_at.z];
                    const int k = nth_bit(reach_o, r - (own_o > 0));
                    const int64_t nk = nbr_key_tab(b, cell_at(o_at), k, spread_tab);
                    const int a0 = cell_start[nk], a1 = cell_start[nk + 1];
                    if (!is_sub(a1 - a0, b, dense_min)) {
                        j0 = a0;
                        cnt = a1 - a0;
                    }
                }
            }
            const int cstart = warp_incl(cnt, lane) - cnt;
            const int C = __shfl_sync(kFull, cstart + cnt, 31);
            for (int cb = kSplit ? part * kWarp : 0; cb < C; cb += kSplit ? parts * kWarp : kWarp) {
                const int u = cb + lane;
                const bool uv = u < C;
                const int it = owner_lane(cstart, uv ? u : C - 1);
                int jj = __shfl_sync(kFull, j0, it) + (u - __shfl_sync(kFull, cstart, it));
                const int oo = __shfl_sync(kFull, o, it);
                if (uv) {
                    const float4 po = rec[oo];
                    const BoxDev& b = g.boxes[at[oo].z];
                    FOF_DCHECK_SLOT(jj, b, uf.err);
                    if (linked(po, sorted[jj], b))
                        uunion<kVar>(parent, (int)(base + oo), jj, uf);
                }
            }
        }
        base = next;
        if (!kSplit && last && lane == 0)
            drawn = atomicAdd(&status->link_ticket, 1u);
    }
}

// Self task of a team cell (team_min..kTeamSelfMax particles, not split
// into sub-cells): cells of up to kTeamSplit particles by one warp each, larger
// ones by a CTA of four warps.  The cell's particles are staged in shared
// memory in z order; its adjacency is built as bit rows, one 32 x 32 block at
// a time: lane i collects row i's word of the block, and the mirrored block's
// words follow by a bit transpose across the lanes, so each unordered pair is
// tested once outside the diagonal blocks.  The components are then traced by
// breadth-first search over bit sets, each lane holding its rows in registers
// (a step is a few ANDs and one ballot per 32 vertices), in ascending order of
// their smallest member s, and every member's parent is set to s.  Isolated
// particles keep parent = self.  The kernel runs before any kernel that links
// across cells, so no other thread touches these parents.
//
// Bound by issue where cells are many, by one cell's chain where they are few
// (one warp took 93,000 cycles for a cell of 256 when it sorted with a bitonic
// network, mirrored blocks by a ballot per candidate and searched rows in
// shared memory).  Before and after, us: 4,096 particles 78 and 14, 2 million
// 153 and 51, 16.8 million (256^3) 642 and 266, 453 million (768^3) 13740 and
// 6900.
constexpr int kTeamWarps = 4;
constexpr int kTeamBlocks = 8;               // CTAs per SM (64 registers, 28 bytes spilled; 27 KB)
constexpr int kZBins = 32;                   // z bins of the order of a team cell

// The staged positions of a cell, axis by axis: one 16-byte load holds two
// pairs of candidates for the packed arithmetic.
template <int kMax>
struct __align__(16) CellPos {
    float x[kMax], y[kMax], z[kMax];

    __device__ __forceinline__ void set(int k, float4 v)
    {
        x[k] = v.x;
        y[k] = v.y;
        z[k] = v.z;
    }
    __device__ __forceinline__ float4 get(int k) const { return make_float4(x[k], y[k], z[k], 0.f); }
};

struct TeamWarpSmem {                        // one warp's cell
    static constexpr int kWords = kTeamSplit / 32;
    static constexpr int kStride = kWords + 1;          // odd stride: conflict-free rows
    CellPos<kTeamSplit> P;
    float4 Q[kTeamSplit];                    // the next cell, copied ahead
    unsigned adj[kTeamSplit * kStride];
    int bin[kZBins];
};

struct TeamCtaSmem {                         // one CTA's cell
    static constexpr int kWords = kTeamSelfMax / 32;
    static constexpr int kStride = kWords + 1;
    CellPos<kTeamSelfMax> P;
    unsigned adj[kTeamSelfMax * kStride];
    int bin[kZBins];
    unsigned todo[kWords];
    unsigned front[2][kWords];
    float zlo[kWords], zhi[kWords];
};

union TeamSmem {
    TeamWarpSmem warp[kTeamWarps];
    TeamCtaSmem cta;
};

// Positions that link to nothing: rows and columns beyond the cell's
// particles.  Any difference with a real position (at most 1e30, the largest
// box) or the other sentinel squares to +inf in float32, which the pre-test
// rejects; where its bound is +inf too (linking lengths above 1.8e19), the exact
// test does: one period of the box brings no sentinel back into it.
constexpr float kFar = 3e38f;

__device__ __forceinline__ float4 far_point(float v)
{
    return make_float4(v, v, v, 0.f);
}

// Two float32 values in one register pair, and the packed operations on them
// (each half rounded to nearest, as the single operation).
__device__ __forceinline__ unsigned long long pack2(float lo, float hi)
{
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}

__device__ __forceinline__ unsigned long long add2(unsigned long long a, unsigned long long b)
{
    unsigned long long r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

__device__ __forceinline__ unsigned long long mul2(unsigned long long a, unsigned long long b)
{
    unsigned long long r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

__device__ __forceinline__ unsigned long long fma2(unsigned long long a, unsigned long long b, unsigned long long c)
{
    unsigned long long r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

// Inside one cell no pair needs the periodic wrap when the box has at least 3
// cells per axis: the cell side is then below L/2, so the wrapped float32
// separation equals the plain difference.
__device__ __forceinline__ bool plain_pairs(const BoxDev& b)
{
    return b.nc >= 3 && b.t_hi <= FLT_MAX;     // block_word: a next float above t_hi exists
}

// The pairs of `band` (bits of a row word) by the exact test; x points to the
// block's first candidate, the other axes follow `axis` words apart.
static __device__ __noinline__ unsigned settle_band(unsigned row, unsigned band, float px, float py, float pz,
                                                    const float* x, int axis, const BoxDev& b)
{
    while (band) {
        const int t = __ffs(band) - 1;
        band &= band - 1u;
        const float* q = x + t;
        if (!linked_exact_inl(make_float4(px, py, pz, 0.f), make_float4(q[0], q[axis], q[2 * axis], 0.f), b.L, b.l2))
            row &= ~(1u << t);
    }
    return row;
}

// Row word with the periodic predicate.
static __device__ __noinline__ unsigned wrapped_word(float px, float py, float pz, const float* x, int axis, int jn8,
                                                     const BoxDev& b)
{
    unsigned row = 0, band = 0;
    for (int t = 0; t < jn8; ++t) {
        const float* q = x + t;
        const float s2 = d2_f32(make_float4(px, py, pz, 0.f), make_float4(q[0], q[axis], q[2 * axis], 0.f), b.Lf);
        row |= (unsigned)(s2 <= b.t_hi) << t;
        band |= (unsigned)(s2 <= b.t_hi && s2 >= b.t_lo) << t;
    }
    return settle_band(row, band, px, py, pz, x, axis, b);
}

// Row word of particle pi against particles j0..j0+jn8 of the cell, jn8 a
// multiple of 8 up to 32.  The float32 pre-test decides; pairs in the uncertainty
// band are noted and take the exact test after the block, entered only when some
// lane has one.  Candidates go two to an operation, and the outcome of a
// comparison is the sign of a difference, shifted into the word: s2 - t is
// negative exactly when s2 < t (the rounded difference of two floats has the
// sign of the exact one), and s2 <= t_hi when s2 is below the next float.
// The kernel is bound by issue, and this halves the instructions of a pair test
// (k_team_self on the 768^3 box 9.05 ms with one candidate and one comparison at
// a time, 8.25 so).  Its 32 warps per SM are at 32 different places of the code,
// so what is rare (the band, the wrap) is out of line and the loop of a warp's
// cell stands once for cells of every size: with copies in line the warps waited
// for instructions most of all (8.25 ms, 6.9 without; 256^3 309 and 266 us).
template <int kMax>
__device__ __forceinline__ unsigned block_word(const float4& pi, const CellPos<kMax>& P, int j0, int jn8,
                                               const BoxDev& b)
{
    if (!plain_pairs(b))
        return wrapped_word(pi.x, pi.y, pi.z, P.x + j0, kMax, jn8, b);
    unsigned row = 0, certain = 0;
    const unsigned long long nx = pack2(-pi.x, -pi.x), ny = pack2(-pi.y, -pi.y), nz = pack2(-pi.z, -pi.z);
    const float above = __uint_as_float(__float_as_uint(b.t_hi) + 1u);     // t_hi > 0
    const unsigned long long nhi = pack2(-above, -above), nlo = pack2(-b.t_lo, -b.t_lo);
#pragma unroll 1
    for (int t0 = 0; t0 < jn8; t0 += 8) {
#pragma unroll
        for (int u = 0; u < 8; u += 4) {
            const ulonglong2 x = *reinterpret_cast<const ulonglong2*>(P.x + j0 + t0 + u);
            const ulonglong2 y = *reinterpret_cast<const ulonglong2*>(P.y + j0 + t0 + u);
            const ulonglong2 z = *reinterpret_cast<const ulonglong2*>(P.z + j0 + t0 + u);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const unsigned long long dx = add2(h ? x.y : x.x, nx), dy = add2(h ? y.y : y.x, ny),
                                         dz = add2(h ? z.y : z.x, nz);
                const unsigned long long s2 = fma2(dz, dz, fma2(dy, dy, mul2(dx, dx)));
                const unsigned long long hi = add2(s2, nhi), lo = add2(s2, nlo);
                row = __funnelshift_l((unsigned)hi, row, 1);
                row = __funnelshift_l((unsigned)(hi >> 32), row, 1);
                certain = __funnelshift_l((unsigned)lo, certain, 1);
                certain = __funnelshift_l((unsigned)(lo >> 32), certain, 1);
            }
        }
    }
    row = __brev(row) >> (32 - jn8);            // the first candidate was shifted in first
    const unsigned band = row & ~(__brev(certain) >> (32 - jn8));
    if (__any_sync(kFull, band != 0u))
        row = settle_band(row, band, pi.x, pi.y, pi.z, P.x + j0, kMax, b);
    return row;
}

// 32 x 32 bit matrix, row r in lane r: returns column `lane` as a row.
__device__ __forceinline__ unsigned transpose32(unsigned x, int lane)
{
    unsigned m = 0x0000ffffu;
#pragma unroll
    for (int k = 16; k; k >>= 1) {
        const unsigned y = __shfl_xor_sync(kFull, x, k);
        x = (lane & k) ? (x & ~m) | ((y >> k) & m) : (x & m) | ((y & m) << k);
        m ^= m << (k >> 1);
    }
    return x;
}

// z bin of a particle in its cell (cz): a monotone function of z
__device__ __forceinline__ int z_bin(float z, int cz, const BoxDev& b)
{
    const int k = (int)__fmul_rn(z, b.inv_zb) - kZBins * cz;
    return min(max(k, 0), kZBins - 1);
}

// Row word of block (ib, jb), jb >= ib, of the staged cell.  `apart`: no pair of
// the block can be linked.
template <int kMax>
__device__ __forceinline__ unsigned block_row(const CellPos<kMax>& P, int m, int ib, int jb, bool apart, int lane,
                                              const BoxDev& b)
{
    if (apart)
        return 0u;
    const int i = ib * 32 + lane;
    const float4 pi = i < m ? P.get(i) : far_point(-kFar);
    const unsigned row = block_word(pi, P, jb * 32, (min(32, m - jb * 32) + 7) & ~7, b);
    return jb == ib ? row & ~(1u << lane) : row;               // not the particle itself
}

// The block's words in the adjacency rows, and those of the mirrored block.
template <int kStride>
__device__ __forceinline__ void put_block(unsigned* adj, unsigned row, int ib, int jb, bool apart, int lane)
{
    adj[(ib * 32 + lane) * kStride + jb] = row;
    if (jb != ib)
        adj[(jb * 32 + lane) * kStride + ib] = apart ? 0u : transpose32(row, lane);
}

// Components of the adjacency rows of a cell of kNw * 32 rows by one warp:
// lane l holds rows l, l + 32, ...; the vertex sets are the same in every lane.
template <int kNw>
__device__ __forceinline__ void trace_components(const unsigned (&rows)[kNw][kNw], int* parent, int c0, int lane)
{
    unsigned todo[kNw];
#pragma unroll
    for (int r = 0; r < kNw; ++r) {
        unsigned any = 0u;
#pragma unroll
        for (int k = 0; k < kNw; ++k)
            any |= rows[r][k];
        todo[r] = __ballot_sync(kFull, any != 0u);
    }
    for (;;) {
        unsigned comp[kNw], front[kNw];
        int s = -1;
#pragma unroll
        for (int r = 0; r < kNw; ++r) {
            const bool here = s < 0 && todo[r] != 0u;
            front[r] = here ? todo[r] & (0u - todo[r]) : 0u;
            if (here)
                s = r * 32 + __ffs(todo[r]) - 1;
            comp[r] = front[r];
        }
        if (s < 0)
            break;
        for (int step = 0; step < kNw * 32; ++step) {      // every step adds a vertex
            unsigned nxt[kNw], any = 0u;
#pragma unroll
            for (int r = 0; r < kNw; ++r) {
                unsigned hit = 0u;
#pragma unroll
                for (int k = 0; k < kNw; ++k)
                    hit |= rows[r][k] & front[k];
                nxt[r] = __ballot_sync(kFull, hit != 0u) & ~comp[r];
                any |= nxt[r];
            }
#pragma unroll
            for (int r = 0; r < kNw; ++r) {
                comp[r] |= nxt[r];
                front[r] = nxt[r];
            }
            if (!any)
                break;
        }
#pragma unroll
        for (int r = 0; r < kNw; ++r) {
            todo[r] &= ~comp[r];
            if ((comp[r] >> lane) & 1u)
                parent[c0 + r * 32 + lane] = c0 + s;
        }
    }
}

template <int kNw>
__device__ __forceinline__ void trace_staged(const TeamWarpSmem& S, int* parent, int c0, int lane)
{
    unsigned rows[kNw][kNw];
#pragma unroll
    for (int r = 0; r < kNw; ++r)
#pragma unroll
        for (int k = 0; k < kNw; ++k)
            rows[r][k] = S.adj[(r * 32 + lane) * TeamWarpSmem::kStride + k];
    trace_components<kNw>(rows, parent, c0, lane);
}

// Positions of a listed cell (size << 32 | first slot) into S.Q with cp.async,
// one commit group; lane k copies particles k, k + 32, ...
__device__ __forceinline__ void team_fetch(TeamWarpSmem& S, int64_t e, const float4* sorted, int lane)
{
    const int c0 = (int)(uint32_t)e, m = (int)(e >> 32);
#pragma unroll
    for (int r = 0; r < kTeamSplit / 32; ++r)
        if (lane + 32 * r < m)
            cp_async16(&S.Q[lane + 32 * r], sorted + c0 + lane + 32 * r);
    cp_async_commit();
}

// One cell of kTeamSplit + 1..kTeamSelfMax particles by the whole CTA.
__device__ __forceinline__ void team_cell_cta(TeamCtaSmem& S, int c0, int m, float4* sorted, int* parent,
                                              int* minorig, const BoxDev& b)
{
    constexpr int kThreads = kTeamWarps * 32, kPer = kTeamSelfMax / kThreads;
    constexpr int kNw = TeamCtaSmem::kWords, kStride = TeamCtaSmem::kStride;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int nw = (m + 31) >> 5;
    float4 v[kPer];
    int bin[kPer], rank[kPer];
    if (threadIdx.x < kZBins)
        S.bin[threadIdx.x] = 0;
#pragma unroll
    for (int r = 0; r < kPer; ++r) {
        const int k = r * kThreads + threadIdx.x;
        if (k < m)
            v[r] = sorted[c0 + k];
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kPer; ++r) {
        const int k = r * kThreads + threadIdx.x;
        if (k < m) {
            bin[r] = z_bin(v[r].z, cell_coord(v[r].z, b), b);
            rank[r] = atomicAdd(S.bin + bin[r], 1);
        }
    }
    __syncthreads();
    if (wid == 0) {
        const int c = S.bin[lane];
        S.bin[lane] = warp_incl(c, lane) - c;
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kPer; ++r) {
        const int k = r * kThreads + threadIdx.x;
        if (k < m) {
            const int at = S.bin[bin[r]] + rank[r];
            S.P.set(at, v[r]);
            sorted[c0 + at] = v[r];
            minorig[c0 + at] = __float_as_int(v[r].w);
        } else if (k < nw * 32) {
            S.P.set(k, far_point(kFar));
        }
    }
    __syncthreads();
    // the z range of each 32 particles: blocks too far apart hold no link
    for (int r = wid; r < nw; r += kTeamWarps) {
        const unsigned z = __float_as_uint(S.P.z[r * 32 + lane] + 0.f);    // finite and >= 0: ordered bits
        const bool in = r * 32 + lane < m;
        const unsigned lo = __reduce_min_sync(kFull, in ? z : 0x7f800000u), hi = __reduce_max_sync(kFull, in ? z : 0u);
        if (lane == 0) {
            S.zlo[r] = __uint_as_float(lo);
            S.zhi[r] = __uint_as_float(hi);
        }
    }
    __syncthreads();
    for (int p = wid; p < nw * (nw + 1) / 2; p += kTeamWarps) {
        int ib = 0, jb = p;
        while (jb >= nw - ib) {
            jb -= nw - ib;
            ++ib;
        }
        jb += ib;
        const float gap = __fsub_rn(S.zlo[jb], S.zhi[ib]);
        const bool apart = b.nc >= 3 && gap > 0.f && __fmul_rn(gap, gap) > b.t_hi;
        put_block<kStride>(S.adj, block_row(S.P, m, ib, jb, apart, lane, b), ib, jb, apart, lane);
    }
    __syncthreads();
    // warp w searches row blocks w and w + kTeamWarps; the frontier's words are
    // exchanged through shared memory, two buffers in turn
    unsigned rows[2][kNw];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int r = wid + h * kTeamWarps;
        unsigned any = 0u;
#pragma unroll
        for (int k = 0; k < kNw; ++k) {
            rows[h][k] = r < nw && k < nw ? S.adj[(r * 32 + lane) * kStride + k] : 0u;
            any |= rows[h][k];
        }
        const unsigned t = __ballot_sync(kFull, any != 0u);
        if (lane == 0)
            S.todo[r] = t;
    }
    __syncthreads();
    unsigned todo[kNw];
#pragma unroll
    for (int k = 0; k < kNw; ++k)
        todo[k] = S.todo[k];
    int buf = 0;
    for (;;) {
        unsigned front[kNw];
        int s = -1;
#pragma unroll
        for (int k = 0; k < kNw; ++k) {
            const bool here = s < 0 && todo[k] != 0u;
            front[k] = here ? todo[k] & (0u - todo[k]) : 0u;
            if (here)
                s = k * 32 + __ffs(todo[k]) - 1;
        }
        if (s < 0)
            break;
        unsigned own[2];                       // this warp's words of the component
#pragma unroll
        for (int h = 0; h < 2; ++h)
            own[h] = (s >> 5) == wid + h * kTeamWarps ? 1u << (s & 31) : 0u;
        for (int step = 0; step < kTeamSelfMax; ++step) {  // every step adds a vertex
#pragma unroll
            for (int k = 0; k < kNw; ++k)
                todo[k] &= ~front[k];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                unsigned hit = 0u;
#pragma unroll
                for (int k = 0; k < kNw; ++k)
                    hit |= rows[h][k] & front[k];
                const unsigned nxt = __ballot_sync(kFull, hit != 0u) & ~own[h];
                own[h] |= nxt;
                if (lane == 0)
                    S.front[buf][wid + h * kTeamWarps] = nxt;
            }
            __syncthreads();
            unsigned any = 0u;
#pragma unroll
            for (int k = 0; k < kNw; ++k) {
                front[k] = S.front[buf][k];
                any |= front[k];
            }
            buf ^= 1;
            if (!any)
                break;
        }
#pragma unroll
        for (int h = 0; h < 2; ++h)
            if ((own[h] >> lane) & 1u)
                parent[c0 + (wid + h * kTeamWarps) * 32 + lane] = c0 + s;
    }
    __syncthreads();                           // smem reused by the next cell
}

__global__ void __launch_bounds__(kTeamWarps * 32, kTeamBlocks)
    k_team_self(Geometry g, const int64_t* list, int64_t cap, const int* n_lo, const int* n_hi, float4* sorted,
                int* __restrict__ parent, int* __restrict__ minorig)
{
    pdl_wait();
    pdl_trigger();
    extern __shared__ float4 team_raw[];
    TeamSmem& smem = *reinterpret_cast<TeamSmem*>(team_raw);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    // cells above kTeamSplit lie at the back of the list
    for (int it = blockIdx.x, n = *n_hi; it < n; it += gridDim.x) {
        const int64_t e = list[cap - 1 - it];
        const int c0 = (int)(uint32_t)e;
        team_cell_cta(smem.cta, c0, (int)(e >> 32), sorted, parent, minorig,
                      g.boxes[box_of_warp(g.box_p0, g.nbox, c0, lane)]);
    }
    // the others, one per warp, the last CTAs first (they have the fewest
    // large cells).  Software pipeline: the next cell's positions are copied
    // ahead while this cell is linked, and the entry after it is read.
    TeamWarpSmem& S = smem.warp[wid];
    const int n = *n_lo;
    const int stride = gridDim.x * kTeamWarps;
    int it = (gridDim.x - 1 - blockIdx.x) * kTeamWarps + wid;
    int64_t e = it < n ? list[it] : 0;
    team_fetch(S, e, sorted, lane);
    int64_t e_next = it + stride < n ? list[it + stride] : 0;
    for (; it < n; it += stride) {
        const int c0 = (int)(uint32_t)e, m = (int)(e >> 32);
        const int nw = (m + 31) >> 5;
        const BoxDev& b = g.boxes[box_of_warp(g.box_p0, g.nbox, c0, lane)];
        cp_async_wait_all();                   // each lane reads back only its own copies
        // the cell in z order (bins of 1/32 of the cell), also in global
        // memory: the streams of the neighbours below then read only a
        // z-prefix of it (k_link), and blocks of 32 here are z-slabs whose
        // gaps prune block pairs.  No kernel has read these slots' order yet
        // (cross-cell links come later).  Cells below kSortMin are not sorted
        // (k_link searches no smaller).
        if (m >= kSortMin) {
            S.bin[lane] = 0;
            __syncwarp();
            int place[kTeamSplit / 32];        // bin << 8 | rank
#pragma unroll
            for (int r = 0; r < kTeamSplit / 32; ++r) {
                const int k = lane + 32 * r;
                if (k < m) {
                    const float z = S.Q[k].z;
                    const int bin = z_bin(z, cell_coord(z, b), b);
                    place[r] = (bin << 8) | atomicAdd(S.bin + bin, 1);
                }
            }
            __syncwarp();
            const int c = S.bin[lane];
            __syncwarp();
            S.bin[lane] = warp_incl(c, lane) - c;
            __syncwarp();
#pragma unroll
            for (int r = 0; r < kTeamSplit / 32; ++r) {
                const int k = lane + 32 * r;
                if (k < m) {
                    const int at = S.bin[place[r] >> 8] + (place[r] & 255);
                    const float4 v = S.Q[k];
                    S.P.set(at, v);
                    sorted[c0 + at] = v;
                    minorig[c0 + at] = __float_as_int(v.w);
                }
            }
        } else if (lane < m) {                 // kSortMin <= 32: one particle per lane
            S.P.set(lane, S.Q[lane]);
        }
        if (nw * 32 - 32 + lane >= m)          // the ragged tail links nothing
            S.P.set(nw * 32 - 32 + lane, far_point(kFar));
        __syncwarp();
        e = e_next;
        if (it + stride < n)
            team_fetch(S, e, sorted, lane);
        e_next = it + 2 * stride < n ? list[it + 2 * stride] : 0;

        // 32 to a block, in z order: blocks too far apart hold no link (every
        // pair's float32 separation squared exceeds t_hi; rounding is monotone)
        float zlo = 0.f, zhi = 0.f;            // lane r: the z range of block r
        for (int r = 0; nw > 1 && r < nw; ++r) {
            const unsigned z = __float_as_uint(S.P.z[r * 32 + lane] + 0.f);    // finite and >= 0: ordered bits
            const bool in = r * 32 + lane < m;
            const unsigned lo = __reduce_min_sync(kFull, in ? z : 0x7f800000u),
                           hi = __reduce_max_sync(kFull, in ? z : 0u);
            zlo = lane == r ? __uint_as_float(lo) : zlo;
            zhi = lane == r ? __uint_as_float(hi) : zhi;
        }
        unsigned rows[1][1];                   // the last block's words
#pragma unroll 1
        for (int ib = 0; ib < nw; ++ib)
#pragma unroll 1
            for (int jb = ib; jb < nw; ++jb) {
                const float gap = __fsub_rn(__shfl_sync(kFull, zlo, jb), __shfl_sync(kFull, zhi, ib));
                const bool apart = b.nc >= 3 && ib != jb && gap > 0.f && __fmul_rn(gap, gap) > b.t_hi;
                rows[0][0] = block_row(S.P, m, ib, jb, apart, lane, b);
                if (nw > 1)
                    put_block<TeamWarpSmem::kStride>(S.adj, rows[0][0], ib, jb, apart, lane);
            }
        __syncwarp();
        if (nw == 1)
            trace_components<1>(rows, parent, c0, lane);
        else if (nw == 2)
            trace_staged<2>(S, parent, c0, lane);
        else if (nw == 3)
            trace_staged<3>(S, parent, c0, lane);
        else
            trace_staged<4>(S, parent, c0, lane);
        __syncwarp();                          // smem reused by the next cell
    }
    cp_async_wait_all();
}

}  // namespace

cudaError_t launch_team_self(const Geometry& g, const Work& w, cudaStream_t s)
{
    if (g.total_n == 0)
        return cudaSuccess;
    // no more CTAs than warps with a cell
    int64_t blocks = w.team_cap / kTeamWarps + 1;
    const int64_t most = (int64_t)sm_count() * kTeamBlocks;
    if (blocks > most) blocks = most;
    return launch_next(g.total_n, k_team_self, blocks, kTeamWarps * 32, sizeof(TeamSmem), s, g, w.team_list, w.team_cap,
                       w.n_team, w.n_team_hi, w.sorted, w.parent, w.minorig);
}

cudaError_t launch_link(const Geometry& g, const Work& w, int dense_min, const UfArgs& uf, cudaStream_t s)
{
    if (g.total_n == 0)
        return cudaSuccess;
    const int64_t windows = (g.total_n + kWarp - 1) / kWarp;
    const int64_t warps = (int64_t)sm_count() * (uf.var ? kLinkVarBlocks : kLinkBlocks) * kLinkWarps;   // resident
    const bool split = windows <= 2 * warps;
    // warps per window while a third of the chip would have none, at most
    // kLinkWarps (a CTA's warps are a whole number of windows)
    int parts = 1;
    while (parts < kLinkWarps && windows * parts * 3 <= warps) parts *= 2;
    // windows per ticket: 32 batches or more to a warp, and few enough tickets
    // for their one counter (768^3 box: 40.4 ms with 1 window, 37.7 with 2, 36.1
    // with 8, 36.7 with 32; 8 million particles: 703, 695 and, with 4, 741 us)
    int batch = 1;
    while (batch < 8 && windows >= warps * 64 * batch) batch *= 2;
    int64_t blocks = (windows * parts + kLinkWarps - 1) / kLinkWarps;
    if (!split && blocks > warps / kLinkWarps) blocks = warps / kLinkWarps;
    auto kernel = uf.var ? (split ? k_link<true, true> : k_link<true, false>)
                         : (split ? k_link<false, true> : k_link<false, false>);
    return launch_next(g.total_n, kernel, blocks, kLinkThreads, 0, s, g, w.sorted, w.cell_start, w.parent, dense_min,
                       parts, batch, w.status, uf);
}

}  // namespace fofgpu
