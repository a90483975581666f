// Internal declarations of the GB300 Friends-of-Friends library.
//
// Device building blocks shared by the kernels:
//   * BoxDev: per-box geometry (a single box is a batch of one box);
//   * cell index of a coordinate, in float32, with a proven margin;
//   * the link predicate: a float32 pre-test whose error bound is derived in
//     fof_plan.cu (setup_box), and the exact double-precision predicate for
//     every pair the pre-test cannot settle;
//   * the concurrent union-find: Find with path halving (writes only on
//     paths of depth >= 2, paper Sec. 3.4.3) and Union by CAS hooking of the
//     larger root onto the smaller one (Sec. 3.1, Sec. 3.2), retried while
//     the hooked root changed under us, with a bounded retry count.
#pragma once

#include <cuda_runtime.h>
#include <float.h>
#include <stdint.h>

namespace fofgpu {

constexpr int kWarp = 32;
constexpr unsigned kFull = 0xffffffffu;

// device error bits (combined into the status word with atomicOr)
constexpr int kErrRange = 1;     // a coordinate outside [0, L) or not finite
constexpr int kErrTimeout = 2;   // a union ran out of CAS retries
constexpr int kErrInternal = 4;  // an internal consistency check failed
constexpr int kFindCap = 1 << 26; // steps of one Find walk (a forest path is shorter)

// Debug builds (FOF_DEBUG_CHECKS, libfof_gb300_debug.so) check every
// neighbour-candidate slot a kernel computes against its box's slot range
// before the access; a bad slot is recorded as an internal error and the
// access goes to the box's first slot instead (never a trap).
#ifdef FOF_DEBUG_CHECKS
#define FOF_DCHECK_SLOT(j, b, err)                                        \
    do {                                                                  \
        if ((int64_t)(j) < (b).p0 || (int64_t)(j) >= (b).p0 + (b).n) {   \
            atomicOr((err), kErrInternal);                                \
            (j) = (int)(b).p0;                                            \
        }                                                                 \
    } while (0)
#else
#define FOF_DCHECK_SLOT(j, b, err) \
    do {                           \
    } while (0)
#endif

struct BoxDev {
    int64_t p0;       // first particle of the box in the concatenated arrays
    int64_t n;        // particles in the box
    int64_t brick0;   // first brick of the box (concatenated brick arrays)
    int64_t cell0;    // first cell of the box (concatenated cell arrays)
    double L;         // box side
    double l2;        // l_x * l_x rounded to double once
    int32_t nb;       // bricks per axis
    int32_t r;        // cells per brick per axis (power of two)
    int32_t log2r;
    int32_t nc;       // cells per axis = nb * r
    int32_t q;        // sub-cells per cell axis (1: cells are not split)
    int32_t nf;       // fine cells per axis = nc * q
    uint32_t magic_q; // ceil(2^32 / q): g / q == __umulhi(g, magic_q) for g < 2^14
    float inv_hf;     // float32(nf / L): fine index = min(nf-1, (int)(x * inv_hf))
    float Lf;         // float32(L) for the float32 pre-test
    float xmax;       // largest float32 strictly below L (valid: 0 <= x <= xmax)
    float t_lo;       // pre-test: d2f < t_lo  => linked
    float t_hi;       // pre-test: d2f > t_hi  => not linked
    float reach2;     // (l_x / hf)^2 (1 + 2^-6): a sub-cell whose box is farther
                      // than this (in fine units, squared) holds no partner
    int32_t team_min; // occupancy from which k_link links a cell as a warp team
    float inv_zb;     // float32(32 nc / L): z bins of a cell's z order (k_team_self)
    float zb_width;   // a particle's z exceeds that of one in the same or an earlier
                      // bin of its cell by more than -zb_width
    float bb_reach2;  // (l_x + 8 L 2^-24)^2 (1 + 2^-20): squared float32 gap from a
                      // bounding box beyond which no partner lies
};

// A cell is "subdivided" (linked by the sub-cell kernels, never pair by
// pair) when its box splits cells (q > 1) and it holds at least dense_min
// particles: up to kDenseMax particles it is a dense cell, staged in shared
// memory (fof_dense.cu); above, a big cell, sorted by sub-cell in global
// memory (fof_big.cu).
constexpr int kDenseMax = 3072;   // particles of a dense cell (shared memory)
// Largest team cell whose own pairs one warp links in shared memory
// (k_team_self); larger unsplit cells link their own pairs in k_link.
constexpr int kTeamSelfMax = 256;
// Team cells up to kTeamSplit particles (one warp each in k_team_self) are
// listed from the front of the team list, larger ones (one CTA each) from its
// back.
constexpr int kTeamSplit = 128;
// Team cells from this size on are stored in z order by k_team_self, and the
// kernels that stream them from the cell below read only the z-prefix that
// can pair (768^3 box, k_team_self and k_link: from 10 on 7.05 and 33.88 ms, from
// 17 6.91 and 33.96, from 25 6.81 and 34.17; step 71.03, 70.94 and 71.08).
constexpr int kSortMin = 17;
constexpr int kMaxQ = 12;
constexpr int kMaxQ3 = kMaxQ * kMaxQ * kMaxQ;

// Per-run device status.
struct Status {
    int err;
    int pad;
    long long n_cat_total;
    int flat;                 // the forest is flattened: parent, minorig and cnt are final
    unsigned link_ticket;
    unsigned passed_on[3];    // pdl_pass_on
};

// ------------------------------------------------------------------------
// ranges of slots
// ------------------------------------------------------------------------
//
// Slots are int32 and a plan may hold 2^31 - 2 of them, so a loop that steps
// past the end of a range counts from the range's start: the slot itself has no
// room to step past.

struct SlotRange {
    int first, count;
};

// Share `rank` of `of` of the slots [first, first + count).
__host__ __device__ __forceinline__ SlotRange slot_share(int first, int count, int rank, int of)
{
    const int share = count / of + (count % of != 0);
    const int64_t at = (int64_t)rank * share;
    const int off = at < count ? (int)at : count;
    return SlotRange{first + off, count - off < share ? count - off : share};
}

// Slot `first + k` lies before `end`.
__host__ __device__ __forceinline__ bool slot_before(int first, int k, int end)
{
    return k < end - first;
}

// ------------------------------------------------------------------------
// dependent launches
// ------------------------------------------------------------------------
//
// A kernel can be launched as a programmatic dependent of the one before it in
// the stream: its CTAs may start once every CTA of that one has started and
// called pdl_trigger (or exited), which takes the launch gap, 2 to 3 us a
// kernel, off the small problems.  A kernel touches nothing that an earlier
// kernel writes before pdl_wait, which returns when the kernel before it has
// completed (and, since that one waited too, all earlier ones).
//
// A kernel that does not need the one just before it starts beside it: it calls
// pdl_wait as its last step, so that it still completes after it.  What the
// kernels before both wrote has completed by then, but only pdl_wait makes it
// visible to a grid, and this grid has not waited.  So the kernel before it
// passes on what its own wait showed it: after that wait it stores a word with
// release order and then triggers (pdl_pass_on), and the kernel beside it loads
// the word with acquire order before it reads anything (pdl_join).  Release and
// acquire are cumulative at gpu scope: every write that the storing thread could
// see comes before every read after the load.  A CTA that does not find the word
// waits at the top instead; the word starts each run at zero.  (After a plain
// launch the word is there, both waits return at once, and the order in the
// stream does the rest.)
//
// Values that an earlier kernel writes are not read through `const
// __restrict__` parameters or __ldg before a value that was read after the
// wait decides their address: the compiler takes such loads for constant
// during the kernel and may move them above the wait.
//
// Every kernel is launched so up to kDependentMax particles: above, launch gaps
// count for little, and a CTA that starts early on an SM keeps the split of its L1
// that the kernel before wanted.  Step with all launches dependent and with none but
// those beside another (at 4 million and below none at all), us: 0.5 million 227 and
// 251, 2 million 523 and 539, 4 million 896 and 915, 8 million 1585 and 1578, 16.7
// million 3015 and 2982, 67 million 11200 and 10700, 453 million 73360 and 70940.
//
// Kernels that run beside the one before them are up to kBesideMax.  The gain of
// filling that one's last SMs shrinks with the work; step with and without them, us:
// 8 million 1578 and 1642, 16.7 million 2982 and 3043, 33.5 million 5630 and 5719, 67
// million 10700 and 10910, 134 million 20760 and 20880, 453 million 70810 and 70940.

constexpr int64_t kDependentMax = 1 << 22;
constexpr int64_t kBesideMax = 1 << 26;

__device__ __forceinline__ void pdl_wait()
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

__device__ __forceinline__ void pdl_trigger()
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// The words of Status::passed_on.
enum { kPassBrickOrder, kPassCellOrder, kPassDenseOrder, kPassWords };

// By every thread of a kernel that another one may run beside, after pdl_wait.
__device__ __forceinline__ void pdl_pass_on(unsigned* word)
{
    if (threadIdx.x == 0) {                    // the trigger after the store
        if (blockIdx.x == 0)
            asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(word), "r"(1u) : "memory");
        pdl_trigger();
    }
}

// By every thread of the kernel beside it, before it reads what earlier kernels wrote.
__device__ __forceinline__ void pdl_join(const unsigned* word)
{
    unsigned there = 0u;
    if (threadIdx.x == 0)
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(there) : "l"(word) : "memory");
    if (!__syncthreads_or((int)there))
        pdl_wait();
}

// dependent: as a programmatic dependent, else a plain launch
template <class... P, class... A>
cudaError_t launch_kernel(bool dependent, void (*kernel)(P...), int64_t grid, int block, size_t smem, cudaStream_t s,
                          A... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = dependent ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

// The next kernel of a run over n particles.
template <class... P, class... A>
cudaError_t launch_next(int64_t n, void (*kernel)(P...), int64_t grid, int block, size_t smem, cudaStream_t s,
                        A... args)
{
    return launch_kernel(n <= kDependentMax, kernel, grid, block, smem, s, args...);
}

// One that runs beside the kernel before it.
template <class... P, class... A>
cudaError_t launch_beside(int64_t n, void (*kernel)(P...), int64_t grid, int block, size_t smem, cudaStream_t s,
                          A... args)
{
    return launch_kernel(n <= kBesideMax, kernel, grid, block, smem, s, args...);
}

// ------------------------------------------------------------------------
// warp helpers
// ------------------------------------------------------------------------

// Inclusive warp prefix sum.
__device__ __forceinline__ int warp_incl(int v, int lane)
{
    for (int o = 1; o < 32; o <<= 1) {
        int y = __shfl_up_sync(kFull, v, o);
        if (lane >= o) v += y;
    }
    return v;
}

// Last lane l with start(l) <= t, where `start` is a non-decreasing per-lane
// value with start(0) == 0 <= t (a binary search over the lanes; lanes
// with an empty range share their successor's start and are never chosen).
__device__ __forceinline__ int owner_lane(int start, int t)
{
    int lo = 0;
#pragma unroll
    for (int step = 16; step; step >>= 1) {      // lo + step <= 31 throughout
        const int probe = __shfl_sync(kFull, start, lo + step);
        if (probe <= t) lo += step;
    }
    return lo;
}

// 16-byte asynchronous copy global -> shared (cp.async), its commit and
// the wait for all of the thread's copies
__device__ __forceinline__ void cp_async16(void* smem, const void* gmem)
{
    const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(sa), "l"(gmem) : "memory");
}

__device__ __forceinline__ void cp_async_commit()
{
    asm volatile("cp.async.commit_group;" ::: "memory");
}

__device__ __forceinline__ void cp_async_wait_all()
{
    asm volatile("cp.async.wait_all;" ::: "memory");
}

// ------------------------------------------------------------------------
// box lookup: box index of a concatenated particle / brick index
// ------------------------------------------------------------------------

__device__ __forceinline__ int box_of(const int64_t* __restrict__ starts, int nbox, int64_t i)
{
    int lo = 0, hi = nbox - 1;
    while (lo < hi) {                 // last box with starts[b] <= i
        int mid = (lo + hi + 1) >> 1;
        if (__ldg(starts + mid) <= i) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// The same by a whole warp (i is the same in all lanes): 32 starts are compared
// at a time, where the search above is a chain of loads (9 for 512 boxes, 2
// here; batch of 512 boxes, binning, self links and outputs together 24.4 and
// 22.6 ms).
__device__ __forceinline__ int box_of_warp(const int64_t* __restrict__ starts, int nbox, int64_t i, int lane)
{
    int lo = 0;
    for (int n = nbox; n > 1;) {
        const int step = (n + 31) >> 5;
        const bool below = lane * step < n && __ldg(starts + lo + lane * step) <= i;
        const int k = max(__popc(__ballot_sync(kFull, below)) - 1, 0);
        lo += k * step;
        n = min(step, n - k * step);
    }
    return lo;
}

// The box of a warp's particles in ascending order: looked up once and kept
// until the particles pass its end.
struct BoxCursor {
    int bi = 0;
    int64_t end = 0;

    // the box of particle i; `first` is the warp's lowest, all lanes take part
    __device__ __forceinline__ int at(const int64_t* starts, int nbox, int64_t first, int64_t i, int lane)
    {
        if (nbox == 1)
            return 0;
        if (first >= end) {
            bi = box_of_warp(starts, nbox, first, lane);
            end = bi + 1 < nbox ? __ldg(starts + bi + 1) : INT64_MAX;
        }
        return i < end ? bi : box_of(starts, nbox, i);
    }
};

// ------------------------------------------------------------------------
// cells
// ------------------------------------------------------------------------

// Fine coordinate along one axis: (int)fl32(x * fl32(nf / L)), clamped so
// that every input (even an invalid one) stays inside the grid.  The cell
// coordinate is the fine one divided by q; the margins that make linked
// pairs land in adjacent cells (and sub-cells within +-2, and sub-cells
// cliques) are derived in fof_plan.cu (setup_box).
__device__ __forceinline__ int fine_coord(float x, const BoxDev& b)
{
    int c = (int)__fmul_rn(x, b.inv_hf);
    c = c < 0 ? 0 : c;
    return c > b.nf - 1 ? b.nf - 1 : c;
}

__device__ __forceinline__ int cell_coord(float x, const BoxDev& b)
{
    int g = fine_coord(x, b);
    return b.q == 1 ? g : (int)__umulhi((unsigned)g, b.magic_q);
}

__device__ __forceinline__ bool is_sub(int m, const BoxDev& b, int dense_min)
{
    return b.q > 1 && m >= dense_min;
}

__device__ __forceinline__ bool is_big(int m, const BoxDev& b)
{
    return b.q > 1 && m > kDenseMax;
}

__device__ __forceinline__ uint32_t spread3(uint32_t v)   // 5 bits -> every 3rd bit
{
    v &= 0x1fu;
    v = (v | (v << 8)) & 0x100fu;
    v = (v | (v << 4)) & 0x10c3u;
    v = (v | (v << 2)) & 0x1249u;
    return v;
}

// Morton order of a cell inside its brick (r <= 32).
__device__ __forceinline__ uint32_t local_code(int lx, int ly, int lz)
{
    return spread3((uint32_t)lx) | (spread3((uint32_t)ly) << 1) | (spread3((uint32_t)lz) << 2);
}

__device__ __forceinline__ int64_t brick_local(const BoxDev& b, int cx, int cy, int cz)
{
    int s = b.log2r;
    return ((int64_t)(cz >> s) * b.nb + (cy >> s)) * b.nb + (cx >> s);
}

// Concatenated cell index: cells are ordered brick by brick (row-major
// bricks), Morton order inside a brick.
__device__ __forceinline__ int64_t cell_key(const BoxDev& b, int cx, int cy, int cz)
{
    int m = b.r - 1;
    int64_t r3 = (int64_t)b.r * b.r * b.r;
    return b.cell0 + brick_local(b, cx, cy, cz) * r3 + local_code(cx & m, cy & m, cz & m);
}

__device__ __forceinline__ int wrap_cell(int c, int nc)
{
    return c < 0 ? c + nc : (c >= nc ? c - nc : c);
}

// The 13 forward neighbours of the half stencil: dz > 0, or dz == 0 and
// dy > 0, or dz == dy == 0 and dx > 0.  Offsets packed as (dx+1) + 3(dy+1)
// + 9(dz+1).
__device__ __forceinline__ void fwd_offset(int k, int& dx, int& dy, int& dz)
{
    // k = 0..12
    int code = k < 9 ? 18 + k : (k < 12 ? 15 + (k - 9) : 14);
    dx = code % 3 - 1;
    dy = (code / 3) % 3 - 1;
    dz = code / 9 - 1;
}

// ------------------------------------------------------------------------
// the link predicate
// ------------------------------------------------------------------------

__device__ __forceinline__ float sep_f32(float a, float b, float Lf)
{
    float d = fabsf(__fsub_rn(a, b));
    return fminf(d, __fsub_rn(Lf, d));
}

__device__ __forceinline__ float d2_f32(const float4& p, const float4& q, float Lf)
{
    float mx = sep_f32(p.x, q.x, Lf);
    float my = sep_f32(p.y, q.y, Lf);
    float mz = sep_f32(p.z, q.z, Lf);
    return __fmaf_rn(mz, mz, __fmaf_rn(my, my, __fmul_rn(mx, mx)));
}

__device__ __forceinline__ double wrap64(double d, double L)
{
    double half = 0.5 * L;
    if (d > half)
        d = __dsub_rn(d, L);
    else if (d < -half)
        d = __dadd_rn(d, L);
    return d;
}

// Exact predicate: s = (dx*dx + dy*dy) + dz*dz in IEEE double with every
// operation rounded to nearest and no contraction; linked iff s <= l2.
__device__ __forceinline__ bool linked_exact_inl(const float4& p, const float4& q, double L, double l2)
{
    double dx = wrap64(__dsub_rn((double)p.x, (double)q.x), L);
    double dy = wrap64(__dsub_rn((double)p.y, (double)q.y), L);
    double dz = wrap64(__dsub_rn((double)p.z, (double)q.z), L);
    double s = __dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy));
    s = __dadd_rn(s, __dmul_rn(dz, dz));
    return s <= l2;
}

// Out of line where register pressure matters: the band is rarely entered.
static __device__ __noinline__ bool linked_exact(float4 p, float4 q, double L, double l2)
{
    return linked_exact_inl(p, q, L, l2);
}

// Pre-test in float32, exact test only inside the uncertainty band.
__device__ __forceinline__ bool linked(const float4& p, const float4& q, const BoxDev& b)
{
    float s = d2_f32(p, q, b.Lf);
    if (s > b.t_hi)
        return false;
    if (s < b.t_lo)
        return true;
    return linked_exact_inl(p, q, b.L, b.l2);
}

// The same predicate with the band test out of line: fewer registers where
// the caller keeps much state live (the dense cell kernels).
__device__ __forceinline__ bool linked_ool(const float4& p, const float4& q, const BoxDev& b)
{
    float s = d2_f32(p, q, b.Lf);
    if (s > b.t_hi)
        return false;
    if (s < b.t_lo)
        return true;
    return linked_exact(p, q, b.L, b.l2);
}

// ------------------------------------------------------------------------
// union-find on the parent array (indices into the binned particle order)
// ------------------------------------------------------------------------

// Loads and stores at gpu scope, served by L2, so that a retry after a
// failed CAS sees the other SMs' hooks (L1 is not coherent).
__device__ __forceinline__ int ld_relaxed(const int* p)
{
    int v;
    asm volatile("ld.relaxed.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void st_relaxed(int* p, int v)
{
    asm volatile("st.relaxed.gpu.global.b32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// Find with path halving.  Every value parent[x] ever holds is an ancestor
// of x (hooks only change roots, halving only skips to a grandparent), so
// racing writes are harmless; the walk strictly decreases x and ends.  The
// step cap only guards against a corrupted forest (it reports, never hangs).
__device__ __forceinline__ int uf_find(int* parent, int x, int* err)
{
    int p = ld_relaxed(parent + x);
    for (int step = 0; p != x; ++step) {
        int gp = ld_relaxed(parent + p);
        if (gp == p)
            return p;
        if (step >= kFindCap || gp > p) {
            atomicOr(err, kErrInternal);
            return p;
        }
        st_relaxed(parent + x, gp);
        x = gp;
        p = ld_relaxed(parent + x);
    }
    return x;
}

// The Finds of x and y (the same walk and halving as uf_find), with the two
// walks interleaved: each step issues the loads of both before using
// either, so the two chains of dependent loads overlap.
__device__ __forceinline__ void uf_find2(int* parent, int& x, int& y, int* err)
{
    int px = ld_relaxed(parent + x);
    int py = ld_relaxed(parent + y);
    for (int step = 0; px != x || py != y; ++step) {
        const bool wx = px != x, wy = py != y;
        const int gx = wx ? ld_relaxed(parent + px) : px;
        const int gy = wy ? ld_relaxed(parent + py) : py;
        if (step >= kFindCap || (wx && gx > px) || (wy && gy > py)) {
            atomicOr(err, kErrInternal);
            x = px;
            y = py;
            return;
        }
        if (wx) {
            if (gx == px) {
                x = px;                        // px is the root
            } else {
                st_relaxed(parent + x, gx);
                x = gx;
                px = ld_relaxed(parent + x);
            }
        }
        if (wy) {
            if (gy == py) {
                y = py;
            } else {
                st_relaxed(parent + y, gy);
                y = gy;
                py = ld_relaxed(parent + y);
            }
        }
    }
}

// Union by root: hook the larger root onto the smaller with CAS, which only
// succeeds while the larger is still a root; otherwise re-find and retry.
// Keeps parent[x] <= x, hence no cycles.  Returns the root reached.
__device__ __forceinline__ int uf_union(int* parent, int a, int b, int cap, int* err)
{
    for (int it = 0; it < cap; ++it) {
        uf_find2(parent, a, b, err);
        if (a == b)
            return a;
        int hi = a > b ? a : b;
        int lo = a > b ? b : a;
        if (atomicCAS(parent + hi, hi, lo) == hi)
            return lo;
    }
    atomicOr(err, kErrTimeout);
    return a < b ? a : b;
}

// ------------------------------------------------------------------------
// union-find variants (measured against the default; same partition)
// ------------------------------------------------------------------------

// Arguments of every union-find call of a kernel.  `find` and `link` select
// the variants of fof.h (FOF_FIND_*, FOF_LINK_*); they are read only by the
// kernels' variant instantiation (kVar = true), so the default path carries
// no runtime switch.
struct UfArgs {
    int cap;     // CAS attempts per union
    int* err;    // status word
    int find;    // 0 halving on paths of depth >= 2, 1 halving at every depth,
                 // 2 full compression, 3 none
    int link;    // 0 hook the larger root onto the smaller, 1 randomised
    int var;     // run the variant instantiation (a variant is selected, or forced)
};

// Random priority of a root for randomised linking: the 32-bit finaliser of
// MurmurHash3, a bijection, so distinct roots never tie.
__device__ __forceinline__ uint32_t uf_priority(int x)
{
    uint32_t h = (uint32_t)x;
    h ^= h >> 16;
    h *= 0x85ebca6bu;
    h ^= h >> 13;
    h *= 0xc2b2ae35u;
    h ^= h >> 16;
    return h;
}

// Find under the selected compression.  Every value parent[x] ever holds is
// an ancestor of x in every variant, so racing writes stay harmless.  The
// ordering check (a parent never exceeds its child) holds only when roots
// hook onto smaller roots.
__device__ __forceinline__ int uf_find_var(int* parent, int x, const UfArgs& u)
{
    const bool ordered = u.link == 0;
    if (u.find == 2) {                              // full compression
        // The first walk records the nodes it passes; every one of them has
        // the root r found as an ancestor for good (trees only merge), so
        // pointing them at r is safe.  Walking the path a second time would
        // not be: other threads may have re-pointed it past r, and writing r
        // into an ancestor of r would close a cycle.
        constexpr int kPath = 16;
        int path[kPath];
        int len = 0;
        int r = x;
        int p = ld_relaxed(parent + r);
        for (int step = 0; p != r; ++step) {
            if (step >= kFindCap || (ordered && p > r)) {
                atomicOr(u.err, kErrInternal);
                return p;
            }
            if (len < kPath)
                path[len++] = r;
            r = p;
            p = ld_relaxed(parent + r);
        }
        for (int k = 0; k + 1 < len; ++k)            // the last one already points at r
            st_relaxed(parent + path[k], r);
        return r;
    }
    int p = ld_relaxed(parent + x);
    for (int step = 0; p != x; ++step) {
        const int gp = ld_relaxed(parent + p);
        if (step >= kFindCap || (ordered && gp > p)) {
            atomicOr(u.err, kErrInternal);
            return p;
        }
        if (gp == p) {
            if (u.find == 1)
                st_relaxed(parent + x, gp);         // the depth-1 rewrite (same value)
            return p;
        }
        if (u.find == 3) {                          // no compression: plain walk
            x = p;
            p = gp;
            continue;
        }
        st_relaxed(parent + x, gp);
        x = gp;
        p = ld_relaxed(parent + x);
    }
    return x;
}

__device__ __forceinline__ int uf_union_var(int* parent, int a, int b, const UfArgs& u)
{
    for (int it = 0; it < u.cap; ++it) {
        a = uf_find_var(parent, a, u);
        b = uf_find_var(parent, b, u);
        if (a == b)
            return a;
        int hi, lo;                                 // hi is hooked onto lo
        if (u.link == 1) {
            const bool a_wins = uf_priority(a) > uf_priority(b);
            lo = a_wins ? a : b;
            hi = a_wins ? b : a;
        } else {
            hi = a > b ? a : b;
            lo = a > b ? b : a;
        }
        if (atomicCAS(parent + hi, hi, lo) == hi)
            return lo;
    }
    atomicOr(u.err, kErrTimeout);
    return a < b ? a : b;
}

template <bool kVar>
__device__ __forceinline__ int ufind(int* parent, int x, const UfArgs& u)
{
    return kVar ? uf_find_var(parent, x, u) : uf_find(parent, x, u.err);
}

template <bool kVar>
__device__ __forceinline__ int uunion(int* parent, int a, int b, const UfArgs& u)
{
    return kVar ? uf_union_var(parent, a, b, u) : uf_union(parent, a, b, u.cap, u.err);
}

// ------------------------------------------------------------------------
// decoupled look-back (single-pass prefix sums over tiles)
// ------------------------------------------------------------------------

// The sum of the counts of all tiles before `tile`, whose own count is
// `mine`, by one full warp.  state[t] = flag << 32 | value, zeroed before the
// kernel: flag 1 = the tile's own count, 2 = the sum up to and including it;
// value and flag share one 64-bit word, so relaxed accesses suffice.  Tiles
// must be handed out in ascending order by a counter (every earlier tile is
// then running or done, so each wait ends); the poll cap only turns a
// corrupted state into a reported error.
__device__ __forceinline__ int lookback(unsigned long long* state, int tile, int mine, int lane, int* err)
{
    if (lane == 0) {
        const unsigned long long w = ((unsigned long long)(tile == 0 ? 2 : 1) << 32) | (unsigned)mine;
        asm volatile("st.relaxed.gpu.global.b64 [%0], %1;" ::"l"(state + tile), "l"(w) : "memory");
    }
    int before = 0;
    for (int at = tile - 1; at >= 0; at -= kWarp) {
        const int t = at - lane;
        unsigned long long w = 2ull << 32;      // before the first tile: nothing
        for (int poll = 0;; ++poll) {
            if (t >= 0)
                asm volatile("ld.relaxed.gpu.global.b64 %0, [%1];" : "=l"(w) : "l"(state + t) : "memory");
            if (__all_sync(kFull, (w >> 32) != 0ull))
                break;
            if (poll >= (1 << 22)) {
                if (lane == 0) atomicOr(err, kErrInternal);
                return 0;
            }
        }
        const unsigned full = __ballot_sync(kFull, (w >> 32) == 2ull);
        const int last = full ? __ffs(full) - 1 : kWarp - 1;    // nearest finished prefix
        before += (int)__reduce_add_sync(kFull, lane <= last ? (unsigned)w : 0u);
        if (full)
            break;
    }
    if (lane == 0 && tile > 0) {
        const unsigned long long w = (2ull << 32) | (unsigned)(before + mine);
        asm volatile("st.relaxed.gpu.global.b64 [%0], %1;" ::"l"(state + tile), "l"(w) : "memory");
    }
    return before;
}

// ------------------------------------------------------------------------
// kernel launchers (one per phase); each returns cudaGetLastError()
// ------------------------------------------------------------------------

struct Geometry {
    const BoxDev* boxes;       // [nbox]
    const int64_t* box_p0;     // [nbox] first particle of each box
    const int64_t* box_brick0; // [nbox] first brick of each box
    int nbox;
    int64_t max_split_n;       // particles of the largest box that splits cells (0: none)
    int64_t total_n;           // particles over all boxes
    int64_t total_bricks;
    int64_t total_cells;
};

struct Work {
    float4* tmp;        // [total_n] particles in brick order
    float4* sorted;     // [total_n] particles in cell order, w = box-local index
    int* parent;        // [total_n] union-find forest over cell-order slots (ranks while binning)
    int* minorig;       // [total_n] smallest box-local index per root
    int* cnt;           // [total_n] group size per root
    int* cell_start;    // [total_cells + 1]
    int* bcount;        // [total_bricks * brick_pad]
    int* bstart;        // [total_bricks + 1]
    unsigned long long* scan_state; // [scan_tiles] look-back words of the brick scan
    int* scan_ticket;   // scan tiles handed out
    int* n_heavy;       // bricks above heavy_from particles
    int* heavy_ticket;  // heavy bricks handed out
    int* heavy_list;    // [total_n / kHeavyBrick + 1] their indices
    unsigned long long* tile_state; // look-back words of the output tiles, or of the scan of their counts
    int* tile_ticket;   // tiles handed out
    int* out_cursor;    // [n_tiles] fill of each output bucket, then the tile's catalogue entries
    int* tile_off;      // [n_tiles + 1] first catalogue entry of each tile (above kDirectMax inputs)
    int64_t n_tiles;
    Status* status;     // device status
    int* group_words;   // what fof_groups counts in, cleared when it starts: n_groups, n_cat,
    int64_t n_group_words; // tile_state, out_cursor and tile_ticket
    unsigned long long* n_groups;  // [nbox]
    unsigned long long* n_cat;     // [nbox]
    int64_t* dense_list; // [dense_cap] cell keys of the subdivided cells
    int* n_dense;        // number of entries in dense_list
    int* dense_root;     // [total_n / dense_min + 1] by first slot / dense_min:
                         // root of a subdivided cell that is one group, else -1
    int64_t* big_list;   // [big_cap] cell keys of the big cells (subdivided, > kDenseMax)
    int* n_big;          // number of entries in big_list
    int64_t* team_list;  // [team_cap] team cells (team_min..kTeamSelfMax particles, not
                         // subdivided): size << 32 | first slot
    int* n_team;         // entries at the front of team_list (cells up to kTeamSplit)
    int* n_team_hi;      // entries at its back (cells above kTeamSplit)
    int64_t team_cap;    // capacity of team_list
};

// Bricks above this many particles are sorted by a cluster of CTAs (from 4,096
// on, both sort kernels: 8 million particles 236 us instead of 213, 16.7 million 392
// and 391, 453 million 9.75 ms instead of 8.93).
constexpr int kHeavyBrick = 8192;
constexpr int kBrickMax = 65535;   // particles of a brick that one CTA can sort
// Bricks whose counters a CTA of the count kernel keeps in shared memory.
constexpr int kTileBricks = 12288;
constexpr int kOutTile = 4096;  // inputs per output tile
// Largest number of inputs whose (label, size) pairs are stored straight at
// the input's index (fof_out.cu).  Outputs and catalogue straight and through
// buckets, us: 2 million 33 and 230, 8 million 132 and 361, 16.7 million 326 and 487,
// 33.5 million 843 and 640, 67 million 1840 and 1050, 453 million 13700 and 6970: the
// pairs (8 bytes each) leave L2 in between.
constexpr int64_t kDirectMax = 1 << 24;

int sm_count();

cudaError_t launch_bin_count(const float* pos, const Geometry& g, const Work& w, cudaStream_t s);
// (of a run over n particles) exclusive prefix sum of in[i * pad], i < len,
// into out[0..len]; state (scan_tiles(len) words) and ticket start at zero;
// entries above heavy_from are listed in `heavy` unless it is null
cudaError_t launch_scan(int64_t n, const int* in, int pad, int* out, int64_t len, unsigned long long* state,
                        int* ticket, int heavy_from, int* heavy, int* n_heavy, int* err, cudaStream_t s);
int heavy_from(int64_t total_n);
bool heavy_bricks(int64_t total_n);   // whether a brick can be above heavy_from
int64_t scan_tiles(int64_t len);
int brick_pad(int64_t bricks);
cudaError_t launch_bin_scatter(const float* pos, const Geometry& g, const Work& w, cudaStream_t s);
cudaError_t launch_brick_sort(const Geometry& g, const Work& w, int dense_min, cudaStream_t s);
// incremental re-binning: flags |= 1 if a particle left its cell, 2 if it left its brick
cudaError_t launch_relink_check(const float* pos, const Geometry& g, const Work& w, int* flags,
                                cudaStream_t s);
cudaError_t launch_forest_init(const Geometry& g, const Work& w, cudaStream_t s);
cudaError_t launch_dense(const Geometry& g, const Work& w, int dense_min, const UfArgs& uf, bool pairs,
                         cudaStream_t s);
int dense_launches(const Geometry& g, int dense_min);   // kernels of one launch_dense
int big_launches(const Geometry& g);                    // and of one launch_big
cudaError_t launch_link(const Geometry& g, const Work& w, int dense_min, const UfArgs& uf,
                        cudaStream_t s);
cudaError_t launch_team_self(const Geometry& g, const Work& w, cudaStream_t s);
// big cells: sort by sub-cell + own pairs (before the dense kernels), then
// their pairs with every neighbour (after them)
cudaError_t launch_big(const Geometry& g, const Work& w, int dense_min, const UfArgs& uf, bool pairs,
                       cudaStream_t s);
// size_count: 0 warp-aggregated atomics, 1 per-block shared-memory hash table
cudaError_t launch_finalize(const Geometry& g, const Work& w, const UfArgs& uf, int size_count, cudaStream_t s);
// both output kernels, and up to kDirectMax inputs the catalogue with them
cudaError_t launch_outputs(const Geometry& g, const Work& w, int32_t* ids, int32_t* sizes, int32_t min_size,
                           int2* cat, int64_t cap, cudaStream_t s);
// the catalogue's own kernels, above
cudaError_t launch_catalogue(const Geometry& g, const Work& w, const int32_t* sizes, int32_t min_size, int2* cat,
                             int64_t cap, cudaStream_t s);
int catalogue_launches(const Geometry& g);

}  // namespace fofgpu
