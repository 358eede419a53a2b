// Fluid-only ("compact") layout: the forward and adjoint steps over the
// fluid nodes alone.
//
// The step of Eq. 1-6 of arXiv 2310.00810 (and, in the adjoint, its exact
// transpose) moves Q populations in and Q out per node, so its time is set
// by the bytes it moves.  A dense layout moves solid nodes as well: in a
// Boolean sphere packing at porosity 0.45 with r = 6 the solid runs along x
// are short, nearly every 32-byte sector holds some fluid node, and skipping
// solid nodes saves almost nothing.  Here the state holds only the nf fluid
// nodes (compact index k: the interior in node order, then the columns
// x = 0 and nx - 1 in node order), and a neighbour table gives, per
// direction i >= 1, where node k pulls from:
//   nbr[(i - 1) nf + k] = compact index of x - c_i    (a fluid node)
//                       = kCmpBB                     (halfway bounce-back link)
//                       = kCmpABB                    (Eq. 6 link through x = -1/2 or nx - 1/2)
// built once from the link words.  Only the boundary columns read that table
// in the sweeps.  For the interior, 4 (Q - 1) table bytes per node would be a
// third of all traffic (32 beside the 72 population bytes of D2Q9 FP32, 72
// beside 152 on D3Q19), so their neighbours come from windows instead: 30
// columns of a row as 32 bits (fluid or not, one column more on each side)
// and the compact index of the first of them.  A node reads its 4-byte
// position (window and column) and the windows of the 3 or 9 rows around it,
// which its warp shares and the caches keep; the bits say which neighbours
// are fluid, and a population count which compact index they have.  Per
// fluid-node update the forward then moves 2 Q populations and about 5 table
// bytes, and nothing for solid nodes.  Consecutive fluid nodes of a row have
// mostly consecutive neighbours, so the loads of a warp stay nearly coalesced.
//
// Everything a node needs besides the state (position, windows, table, inlet
// density, tau) does not change during a sweep, so the kernels read it before
// they wait for the preceding launch (griddepcontrol.wait): on lattices that
// live in the L2 cache that latency hides behind the launch before.  The
// sweep's first kernel follows a copy or a memset, a full dependency.
//
// Boundary rules, collision and the adjoint algebra are the ones of step.cu
// and adjoint.cu (same helpers); only the addressing differs.  The dense
// index idx[k] recovers (x, y, z) where the rules need it: the Eq. 6 nodes
// (density and inlet-gradient slot of the row) and the conversions between
// the caller's dense arrays and the internal compact states.
//
// In-place (AA-pattern) streaming.  Slot (x, i) of a state is entry
// [i][x].  A state is stored in one of two layouts:
//   natural (N): slot (x, i) holds g_i(x);
//   swapped (W): g_i(x) sits at (x + c_i, opp(i)) where x + c_i is a fluid
//                node, else at (x, i) (the population comes back to x:
//                bounce-back, Eq. 6, the velocity inlet),
// so that in W everything node x receives sits in its own slots: direction
// i at (x, opp(i)).  A step from N gathers through the table and scatters
// its output into W (the gather step); a step from W reads and writes node
// x's own slots (the local step, no table).  In both, the slots a node
// writes are exactly the slots it reads, so each step can run in place on
// one buffer.  The adjoint (gather form) streams the other way: for lambda,
// W puts lambda_m(x) at (x - c_m, opp(m)) where x - c_m is a fluid node,
// else at (x, m), and the same two steps alternate.  A sweep stores g^t in N
// for even t and in W for odd t (lambda^t likewise), so that every other
// step of the forward and of the adjoint reads no table.  The Eq. 6 nodes
// need the velocity of their own g^{t-1}, which in place may already be
// overwritten by a neighbour: each in-place forward step keeps it per
// boundary node in a small side array (the node writes the velocity of its
// output, and reads it back at the next step).
#include <algorithm>
#include <type_traits>

#include "device.cuh"

namespace lbm {

#define LBM_CMP_TRY(expr)                 \
    do {                                  \
        lbm_status st__ = (expr);         \
        if (st__ != LBM_OK) return st__;  \
    } while (0)

namespace {

constexpr int kCmpThreads = 256;
constexpr int kScanNodes = 1024;  // nodes per block of the table-building scan (256 threads x 4)

// How a step finds what node x receives, and where it writes what x sends.
constexpr int kInGather = 0;    // from a natural state through the table (also the two-buffer pull)
constexpr int kInLocal = 1;     // from a swapped state, in x's own slots
constexpr int kOutOwn = 0;      // into x's own slots: natural layout
constexpr int kOutScatter = 1;  // through the table: swapped layout
constexpr int kOutDense = 2;    // into the caller's dense [Q][N] array

// The steps that may run in place.
template <int IN, int OUT>
constexpr bool kInPlace = IN == kInLocal || OUT == kOutScatter;

size_t a256(size_t x) { return (x + 255) & ~size_t(255); }

struct TableLayout {
    size_t inst, idx, nbr, eq6, pos, win, edge, cmap, blk, total_slot, bytes;
    long long n_win;
};

// Windows of one row and of one padded plane (a solid row on each side of
// y; D3Q19 also has a solid plane on each side of z).
int windows_per_row(const PlanInfo& p) { return (p.geo.nx + kWinCols - 1) / kWinCols; }
long long windows_per_plane(const PlanInfo& p) { return (long long)(p.geo.ny + 2) * windows_per_row(p); }

TableLayout table_layout(const PlanInfo& p, long long nf)
{
    TableLayout t;
    const long long nblk = (p.geo.N + kScanNodes - 1) / kScanNodes;
    size_t o = 0;
    t.inst = o;  // the lattice as a pack of one (BCmpInst)
    o += a256(sizeof(BCmpInst));
    t.idx = o;
    o += a256(sizeof(int32_t) * (size_t)nf);
    t.nbr = o;
    o += a256(sizeof(int32_t) * (size_t)(p.q - 1) * (size_t)nf);
    t.eq6 = o;
    o += a256(sizeof(uint32_t) * (size_t)((nf + 31) / 32));
    t.n_win = window_count(p);
    t.pos = o;
    o += a256(sizeof(uint32_t) * (size_t)nf);
    t.win = o;
    o += a256(sizeof(uint2) * (size_t)t.n_win);
    t.edge = o;
    o += a256(sizeof(int2) * (size_t)t.n_win);
    t.cmap = o;
    o += a256(sizeof(int32_t) * (size_t)p.geo.N);
    t.blk = o;
    o += a256(sizeof(int32_t) * (size_t)nblk);
    t.total_slot = o;
    o += 256;
    t.bytes = o;
    return t;
}

// --------------------------------------------------------------- the tables

__device__ __forceinline__ int block_sum_int(int v)
{
    __shared__ int s[32];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) s[threadIdx.x >> 5] = v;
    __syncthreads();
    const int nw = (blockDim.x + 31) >> 5;
    v = (int)threadIdx.x < nw ? s[threadIdx.x] : 0;
    if (threadIdx.x < 32) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    }
    return v;  // valid in thread 0
}

// Exclusive scan of one int per thread over the block (blockDim.x a multiple
// of 32, at most 1024); *total gets the block sum.
__device__ __forceinline__ int block_excl_scan(int v, int* total)
{
    __shared__ int s[32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    int inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += t;
    }
    if (lane == 31) s[w] = inc;
    __syncthreads();
    if (w == 0) {
        int x = lane < nw ? s[lane] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += t;
        }
        if (lane < nw) s[lane] = x;  // inclusive warp totals
    }
    __syncthreads();
    const int before = w > 0 ? s[w - 1] : 0;
    *total = s[nw - 1];
    __syncthreads();
    return before + inc - v;
}

// The compact order: the interior fluid nodes first, in node order, then the
// fluid nodes of the columns x = 0 and x = nx - 1 (the only ones that can
// have an Eq. 6 or velocity-inlet link), in node order.  The boundary nodes
// take a longer branch of the step and adjoint kernels; grouped, they do not
// split the warps of the interior.
__device__ __forceinline__ bool cmp_member(const uint32_t* __restrict__ link, long long n, long long N, int nx, int cls)
{
    if (n >= N || (link[n] & kLinkSolid)) return false;
    const int x = (int)(n % nx);
    return ((x == 0 || x == nx - 1) ? 1 : 0) == cls;
}

// Fluid nodes of class cls (0 interior, 1 boundary columns) per 1024-node block.
__global__ void __launch_bounds__(256) k_cmp_count(const uint32_t* __restrict__ link, long long N, int nx, int cls,
                                                   int* __restrict__ blk)
{
    const long long base = (long long)blockIdx.x * kScanNodes;
    int c = 0;
    for (int j = threadIdx.x; j < kScanNodes; j += blockDim.x)
        if (cmp_member(link, base + j, N, nx, cls)) ++c;
    c = block_sum_int(c);
    if (threadIdx.x == 0) blk[blockIdx.x] = c;
}

// In-place exclusive scan of the block counts (one block); total fluid count out.
__global__ void __launch_bounds__(1024) k_cmp_scan(int* __restrict__ blk, long long nblk, long long* __restrict__ total)
{
    long long carry = 0;
    for (long long b0 = 0; b0 < nblk; b0 += blockDim.x) {
        const long long b = b0 + threadIdx.x;
        const int v = b < nblk ? blk[b] : 0;
        int sum;
        const int ex = block_excl_scan(v, &sum);
        if (b < nblk) blk[b] = (int)(carry + ex);
        carry += sum;
    }
    if (threadIdx.x == 0) *total = carry;
}

// Dense -> compact map and the compact -> dense index of the class-cls
// nodes, in node order from compact index *base (0 for the interior, the
// interior count for the boundary columns).  The interior pass marks every
// other node -1; the boundary pass then fills its own entries.
__global__ void __launch_bounds__(256) k_cmp_index(const uint32_t* __restrict__ link, long long N, int nx, int cls,
                                                   const long long* __restrict__ base, const int* __restrict__ blk,
                                                   int32_t* __restrict__ cmap, int32_t* __restrict__ idx, long long nf)
{
    const long long n0 = (long long)blockIdx.x * kScanNodes + 4LL * threadIdx.x;
    bool fl[4];
    int c = 0;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        fl[j] = cmp_member(link, n0 + j, N, nx, cls);
        c += fl[j] ? 1 : 0;
    }
    int sum;
    long long k = (cls ? *base : 0) + (long long)blk[blockIdx.x] + block_excl_scan(c, &sum);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const long long n = n0 + j;
        if (n >= N) break;
        if (fl[j] && k >= 0 && k < nf) {
            cmap[n] = (int32_t)k;
            idx[k] = (int32_t)n;
            ++k;
        } else if (!cls) {
            cmap[n] = -1;
        }
    }
}

template <int Q>
__global__ void __launch_bounds__(256) k_cmp_nbr(const uint32_t* __restrict__ link, const int32_t* __restrict__ cmap,
                                                 const int32_t* __restrict__ idx, int32_t* __restrict__ nbr,
                                                 long long nf, Geo g)
{
    using L = Lattice<Q>;
    const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= nf) return;
    const long long n = idx[k];
    const int x = (int)(n % g.nx), y = (int)((n / g.nx) % g.ny), z = (int)(n / ((long long)g.nx * g.ny));
    const uint32_t lw = link[n];
#pragma unroll
    for (int i = 1; i < Q; ++i) {
        int32_t code;
        const int xs = x - L::c(i, 0), zs = z - L::c(i, 2);
        int ys = y - L::c(i, 1);
        if (g.periodic_y) ys = (ys + g.ny) % g.ny;  // ys is in -1..ny
        if ((lw >> i) & 1u) {
            code = kCmpBB;
        } else if (xs < 0 || xs >= g.nx) {
            code = kCmpABB;
        } else {
            // a link that is neither bounce-back nor Eq. 6 starts at a fluid node inside the lattice;
            // anything else (an inconsistent link array) is treated as bounce-back
            const bool inside = ys >= 0 && ys < g.ny && zs >= 0 && zs < g.nz;
            const long long m = ((long long)zs * g.ny + ys) * g.nx + xs;
            code = inside ? cmap[m] : kCmpBB;
            if (code < 0) code = kCmpBB;
        }
        nbr[(long long)(i - 1) * nf + k] = code;
    }
}

// One bit per compact node: set where the node has an Eq. 6 (or velocity
// inlet) link, the nodes the local step of the in-place schedule sends to
// the table path.  Bit k & 31 of word k >> 5.
template <int Q>
__global__ void __launch_bounds__(256) k_cmp_eq6_bits(const int32_t* __restrict__ nbr, long long nf,
                                                      uint32_t* __restrict__ bits)
{
    const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    bool b = false;
    if (k < nf)
        for (int i = 1; i < Q; ++i) b |= nbr[(long long)(i - 1) * nf + k] == kCmpABB;
    const unsigned w = __ballot_sync(0xffffffffu, b);
    if ((threadIdx.x & 31) == 0 && k < nf) bits[k >> 5] = w;
}

// Window g of padded row r: bit b of its word is column 30 g - 1 + b, set
// where that node is fluid; its index is such that adding the number of set
// bits below column x - 1 gives the compact index of the first interior
// fluid node of the row at or after x - 1 (the x = 0 node, whose compact
// index lies elsewhere, is counted in the bits and subtracted in the index).
// Padding rows are solid, with periodic y copies of the rows they stand for.
__global__ void __launch_bounds__(256) k_cmp_windows(const int32_t* __restrict__ cmap, Geo g, int d3, int w_row,
                                                     long long n_win, uint2* __restrict__ win, int2* __restrict__ edge)
{
    const long long w = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (w >= n_win) return;
    const int gx = (int)(w % w_row);
    const long long r = w / w_row;
    int y = (int)(r % (g.ny + 2)) - 1;
    const int z = d3 ? (int)(r / (g.ny + 2)) - 1 : 0;
    if (g.periodic_y) y = (y + g.ny) % g.ny;
    uint32_t bits = 0;
    int first = 0;
    bool have = false;
    int2 e = make_int2(-1, -1);
    if (y >= 0 && y < g.ny && z >= 0 && z < g.nz) {
        const int32_t* row = cmap + ((long long)z * g.ny + y) * g.nx;
        for (int b = 0; b < 32; ++b) {
            const int x = kWinCols * gx - 1 + b;
            if (x < 0 || x >= g.nx || row[x] < 0) continue;
            if (!have && x > 0 && x < g.nx - 1) {
                have = true;
                first = row[x] - __popc(bits);
            }
            bits |= 1u << b;
        }
        e = make_int2(row[0], row[g.nx - 1]);
    }
    win[w] = make_uint2(bits, (uint32_t)first);
    edge[w] = e;
}

// pos[k]: the window of an interior node above seven bits: its column in the
// window (0..29), and whether it lies in column 1 or nx - 2, next to a
// boundary column.  Two more codes mark the boundary columns, which go
// through the table, and a batch's padding nodes.
constexpr uint32_t kPosFirst = 1u << 5;
constexpr uint32_t kPosLast = 2u << 5;
constexpr uint32_t kPosBnd = 3u << 5;
constexpr uint32_t kPosDead = kPosBnd | 1u;
constexpr long long kMaxWindows = 1LL << 25;

__global__ void __launch_bounds__(256) k_cmp_positions(const int32_t* __restrict__ idx, Geo g, int d3, int w_row,
                                                       long long n_int, long long nf, uint32_t* __restrict__ pos)
{
    const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= nf) return;
    const unsigned n = (unsigned)idx[k], nx = (unsigned)g.nx, ny = (unsigned)g.ny;
    const unsigned row = n / nx, x = n - row * nx;
    const unsigned z = row / ny, y = row - z * ny;
    const unsigned r = (d3 ? (z + 1) * (ny + 2) : 0u) + y + 1;
    const unsigned w = r * (unsigned)w_row + x / kWinCols;
    pos[k] = k >= n_int ? kPosBnd : (w << 7) | (x == 1 ? kPosFirst : x == nx - 2 ? kPosLast : 0u) | x % kWinCols;
}

__global__ void __launch_bounds__(256) k_cmp_fill(uint32_t* __restrict__ p, long long n, uint32_t v)
{
    const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (k < n) p[k] = v;
}

// The rows a node's neighbours lie in: its own, y +- 1, and on D3Q19 those of
// z +- 1; row_of(i) is the row of direction i's source x - c_i.
template <int Q>
struct Rows {
    static constexpr int N = Q == 9 ? 3 : 9;
    static constexpr int row_of(int i) { return (1 - Lattice<Q>::c(i, 1)) + (Q == 9 ? 0 : 3 * (1 - Lattice<Q>::c(i, 2))); }
    static constexpr int dy(int r) { return r % 3 - 1; }
    static constexpr int dz(int r) { return Q == 9 ? 0 : r / 3 - 1; }
};

// An interior node's neighbours: the compact index j[i] of x - c_i where
// fluid(i), and the bits (x - 1, x, x + 1 fluid) of each row.
template <int Q>
struct Neighbours {
    uint32_t j[Q];
    uint32_t b[Rows<Q>::N];
    __device__ __forceinline__ bool fluid(int i) const
    {
        return (b[Rows<Q>::row_of(i)] & (1u << (1 - Lattice<Q>::c(i, 0)))) != 0u;
    }
};

// The windows of the rows around an interior node.
template <int Q>
struct Windows {
    uint2 q[Rows<Q>::N];
};

template <int Q>
__device__ __forceinline__ void load_windows(Windows<Q>& win, const Cmp& c, const CmpBlk& lat, uint32_t pos)
{
    using R = Rows<Q>;
    const uint2* p = c.win + (int)(pos >> 7);
#pragma unroll
    for (int r = 0; r < R::N; ++r) win.q[r] = __ldg(p + (R::dz(r) * lat.w_plane + R::dy(r) * lat.w_row));
}

template <int Q>
__device__ __forceinline__ void neighbours_of(Neighbours<Q>& nb, const Windows<Q>& win, const Cmp& c,
                                              const CmpBlk& lat, int32_t k, uint32_t pos)
{
    using L = Lattice<Q>;
    using R = Rows<Q>;
    const uint32_t s = pos & 31u, below = (1u << s) - 1u;
#pragma unroll
    for (int r = 0; r < R::N; ++r) {
        const uint2 q = win.q[r];
        const uint32_t b = q.x >> s;
        nb.b[r] = b;
        const bool own = R::dy(r) == 0 && R::dz(r) == 0;
        const uint32_t at = own ? (uint32_t)k - (b & 1u) : q.y + __popc(q.x & below);
        const uint32_t mid = at + (b & 1u);
        const uint32_t right = mid + ((b >> 1) & 1u);
#pragma unroll
        for (int i = 1; i < Q; ++i) {
            if (R::row_of(i) != r) continue;
            nb.j[i] = L::c(i, 0) == 1 ? at : (L::c(i, 0) == 0 ? mid : right);
        }
    }
    if (pos & (kPosFirst | kPosLast)) {  // a neighbour in column 0 or nx - 1
        const int2* e = c.edge + (int)(pos >> 7);
#pragma unroll
        for (int i = 1; i < Q; ++i) {
            if (L::c(i, 0) == 0) continue;
            const int2 v = __ldg(e - (L::c(i, 2) * lat.w_plane + L::c(i, 1) * lat.w_row));
            if (L::c(i, 0) == 1 && (pos & kPosFirst)) nb.j[i] = (uint32_t)v.x;
            if (L::c(i, 0) == -1 && (pos & kPosLast)) nb.j[i] = (uint32_t)v.y;
        }
    }
}

template <int Q>
__device__ __forceinline__ void window_neighbours(Neighbours<Q>& nb, const Cmp& c, const CmpBlk& lat, int32_t k,
                                                  uint32_t pos)
{
    Windows<Q> win;
    load_windows<Q>(win, c, lat, pos);
    neighbours_of<Q>(nb, win, c, lat, k, pos);
}

// Counts the interior nodes whose windows give other codes than the table
// (none, for link words of this library; a lattice with any falls back on
// the table throughout).
template <int Q>
__global__ void __launch_bounds__(256) k_cmp_window_check(Cmp c, CmpBlk lat, long long n_int,
                                                          unsigned long long* __restrict__ bad)
{
    const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n_int) return;
    Neighbours<Q> nb;
    window_neighbours<Q>(nb, c, lat, (int32_t)k, c.pos[k]);
    bool off = false;
#pragma unroll
    for (int i = 1; i < Q; ++i)
        off |= (nb.fluid(i) ? (int32_t)nb.j[i] : kCmpBB) != c.nbr[(long long)(i - 1) * c.nf + k];
    if (off) atomicAdd(bad, 1ull);
}

// ----------------------------------------------------------- the step kernels

// A boundary-column node's inlet/outlet data for Eq. 6.
struct Side {
    bool xin;
    long long row;  // z * ny + y
};

__device__ __forceinline__ Side side_of(const int32_t* __restrict__ idx, long long k, const Geo& g)
{
    const unsigned n = (unsigned)__ldg(idx + k), row = n / (unsigned)g.nx;  // N < 2^31
    Side s;
    s.xin = n == row * (unsigned)g.nx;
    s.row = row;
    return s;
}

// The side-array entry of an Eq. 6 node (three values): inlet rows first,
// then outlet rows; acc_off counts the rows of the instances before it.
template <typename T>
__device__ __forceinline__ T* side_entry(const Bc& bc, const BCmpInst& I, const Side& sd)
{
    const long long rows = (long long)I.g.ny * I.g.nz;
    return static_cast<T*>(bc.side_u) + 3 * (2 * I.acc_off + (sd.xin ? 0 : rows) + sd.row);
}

__device__ __forceinline__ bool eq6_bit(const Cmp& c, long long k)
{
    return (__ldg(c.eq6 + (k >> 5)) >> (k & 31)) & 1u;
}

template <int Q>
__device__ __forceinline__ bool load_codes(int32_t (&code)[Q], const Cmp& c, long long k)
{
    code[0] = 0;
    bool bnd = false;
#pragma unroll
    for (int i = 1; i < Q; ++i) {
        code[i] = __ldg(c.nbr + (size_t)(i - 1) * (size_t)c.nf + (int32_t)k);
        bnd |= code[i] == kCmpABB;
    }
    return bnd;
}

// A node as its kernel knows it before it touches the state.
struct Node {
    int32_t k;
    uint32_t pos;
    CmpBlk blk;      // its instance, and that one's windows per row and plane
    __device__ __forceinline__ bool live() const { return (pos & 127u) != kPosDead; }
    __device__ __forceinline__ bool bnd() const { return (pos & 127u) == kPosBnd; }
    __device__ __forceinline__ bool interior() const { return (pos & kPosBnd) != kPosBnd; }
};

// blks: a batch's entry of each 256-node block (null for a single lattice,
// which passes its own one).
__device__ __forceinline__ Node node_of(int32_t k, const Cmp& c, const CmpBlk& lat, const CmpBlk* __restrict__ blks)
{
    Node nd;
    nd.k = k;
    nd.blk = lat;
    nd.pos = kPosDead;
    if (k < (int32_t)c.nf) {
        nd.pos = __ldg(c.pos + k);
        if (blks) {
            const int4 v = __ldg(reinterpret_cast<const int4*>(blks) + k / kCmpThreads);
            nd.blk = CmpBlk{v.x, v.y, v.z, 0};
        }
    }
    return nd;
}

// What a boundary-column node knows besides: its place and wall density.
struct Wall {
    Side sd = {false, 0};
    double rw = 1.0;  // rho_w of Eq. 6
};

// A boundary-column node's neighbour codes (from the table) and wall density.
template <int Q>
__device__ __forceinline__ Wall boundary_codes(int32_t (&code)[Q], const Node& nd, const Cmp& c,
                                               const BCmpInst* __restrict__ insts, const Bc& tmpl)
{
    load_codes<Q>(code, c, nd.k);
    const BCmpInst& I = insts[nd.blk.inst];
    Wall w;
    w.sd = side_of(c.idx, nd.k, I.g);
    const double* rho_in = tmpl.rho_in + I.in_off;
    w.rw = w.sd.xin ? rho_in[I.n_in > 1 ? w.sd.row : 0] : tmpl.rho_out;
    return w;
}

// A state load.  CG: from the L2 cache, for the kernels of the in-place
// schedule and for every read-modify-write: the next launch of a sweep
// becomes resident on an SM before the current one has finished, so a line
// the current one brought into the L1 cache late can be stale for the next.
// The two-buffer pull needs no such care: a launch writes the buffer that
// the launch before it read, and the launch after it, which reads that
// buffer, starts (with an empty L1 cache) when those reads are over.
template <bool CG, typename T>
__device__ __forceinline__ T ld_state(const T* p)
{
    return CG ? __ldcg(p) : *p;
}

// What an interior node receives: from its neighbours over fluid links, else
// its own population of the opposite direction.  Every address is selected
// first (32-bit element offsets into the state) and every load issued
// unconditionally, so all Q are in flight together.
template <int Q, typename T, int IN, bool CG>
__device__ __forceinline__ void pull_interior(T (&v)[Q], const T* src, int32_t k, uint32_t NF, const Neighbours<Q>& nb)
{
    using L = Lattice<Q>;
    v[0] = ld_state<CG>(src + k);
#pragma unroll
    for (int i = 1; i < Q; ++i) {
        const uint32_t own = (uint32_t)L::opp(i) * NF + (uint32_t)k;
        const uint32_t at = IN == kInGather && nb.fluid(i) ? (uint32_t)i * NF + nb.j[i] : own;
        v[i] = ld_state<CG>(src + at);
    }
}

// The same through table codes, for the boundary columns (the populations of
// Eq. 6 links come back as they left: apply_eq6 takes them from there).
template <int Q, typename T, int IN, bool CG>
__device__ __forceinline__ void pull_links(T (&v)[Q], const T* src, int32_t k, size_t NF,
                                           const int32_t (&code)[Q])
{
    using L = Lattice<Q>;
    v[0] = ld_state<CG>(src + k);
#pragma unroll
    for (int i = 1; i < Q; ++i) {
        if (IN == kInLocal) {
            v[i] = ld_state<CG>(src + (size_t)L::opp(i) * NF + k);
        } else {
            const bool fl = code[i] >= 0;
            const T* base = src + (size_t)(fl ? i : L::opp(i)) * NF;
            v[i] = ld_state<CG>(base + (fl ? code[i] : k));
        }
    }
}

// The velocity of node k's own post-collision populations g(x), from a
// state in layout IN (natural: own slots; swapped: where x sent them).
template <int Q, typename T, int IN>
__device__ __forceinline__ void own_velocity(T (&u)[3], const T* src, int32_t k, size_t NF,
                                             const int32_t (&code)[Q])
{
    using L = Lattice<Q>;
    T loc[Q];
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        const int32_t co = IN == kInLocal && i > 0 ? code[L::opp(i)] : -1;
        const T* base = src + (size_t)(co >= 0 ? L::opp(i) : i) * NF;
        loc[i] = base[co >= 0 ? co : k];
    }
    T drho, rho;
    moments<Q, T>(loc, drho, rho, u);
}

// The Eq. 6 and velocity-inlet links of a boundary-column node, whose
// populations that came back are in v.  Its velocity comes from the side
// array in the in-place forward steps (bc.side_u), else from src.
template <int Q, typename T, int IN>
__device__ __forceinline__ void apply_eq6(T (&v)[Q], const T* src, int32_t k, const Wall& wall, size_t NF,
                                          const int32_t (&code)[Q], const Bc& bc, const BCmpInst* I, bool side)
{
    using L = Lattice<Q>;
    T u[3];
    if (side) {
        const T* e = side_entry<T>(bc, *I, wall.sd);
        u[0] = ld_state<true>(e);
        u[1] = ld_state<true>(e + 1);
        u[2] = ld_state<true>(e + 2);
    } else {
        own_velocity<Q, T, IN>(u, src, k, NF, code);
        if constexpr (IN == kInGather) {
            if (bc.uw_extrap) {
                const int32_t ke = code[inward_dir<Q>(wall.sd.xin)];
                if (ke >= 0) extrapolate_wall_velocity<Q, T>(u, src, (long long)NF, ke);
            }
        }
    }
    const T uu = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
    const T drw = T(wall.rw - 1.0), rwT = T(wall.rw);
    // Opposite links together: a node has one of each pair (nx > 1), and a warp
    // holds nodes of both sides.  These warps decide how long a small lattice's
    // step takes (64x32 FP64: 2.8 of 18.0 us per time level of a gradient
    // evaluation less than link by link here and in the adjoint).
#pragma unroll
    for (int i = 1; i < Q; ++i) {
        if (L::c(i, 0) != 1) continue;
        const int o = L::opp(i);
        const bool here = code[i] == kCmpABB;
        if (!here && code[o] != kCmpABB) continue;
        T back = here ? v[i] : v[o];
        if (here && bc.vel_inlet) {
            // velocity inlet: moving-wall bounce-back, f_i = f*_opp(i) + 6 w_i (c_i . u_in) (rho_0 = 1)
            double cu = 0.0;
#pragma unroll
            for (int a = 0; a < L::D; ++a) cu += (double)L::c(i, a) * bc.u_in[a];
            back += T(6.0 * L::w(i) * cu * bc.ramp);
        } else {
            const T cu = cdot<Q, T>(i, u);
            back = -back + T(2.0 * L::w(i)) * (drw + rwT * (T(4.5) * cu * cu - T(1.5) * uu));
        }
        if (here) v[i] = back;
        else v[o] = back;
    }
}

// What a node receives, through table codes.
template <int Q, typename T, int IN, bool CG>
__device__ __forceinline__ void pull_table(T (&v)[Q], const T* src, int32_t k, const Wall& wall, size_t NF,
                                           const int32_t (&code)[Q], const Bc& bc, const BCmpInst* I, bool side)
{
    pull_links<Q, T, IN, CG>(v, src, k, NF, code);
    bool eq6 = false;
#pragma unroll
    for (int i = 1; i < Q; ++i) eq6 |= code[i] == kCmpABB;
    if (eq6) apply_eq6<Q, T, IN>(v, src, k, wall, NF, code, bc, I, side);
}

// An opaque zero that depends on x.
template <typename T>
__device__ __forceinline__ int32_t zero_after(T x)
{
    int32_t z;
    const float f = (float)x;
    asm volatile("and.b32 %0, %1, 0;" : "=r"(z) : "r"(__float_as_int(f)));
    return z;
}

// The scattered stores of the in-place steps need the neighbours of a node
// after its collision: x + c_i for g_i (D: 1), x - c_i for lambda_i (D: -1).
// They are formed again (cache hits) from an index that depends on the
// collision's output, so that the loads stay behind it: kept in registers
// through the collision, they spill on D3Q19.
template <int Q, typename T, int D>
__device__ __forceinline__ void store_scattered(T* dst, const T (&v)[Q], const Node& nd, const Cmp& c)
{
    using L = Lattice<Q>;
    const int32_t k = nd.k + zero_after(v[Q - 1]);
    dst[k] = v[0];
    if (nd.bnd()) {
        const size_t NF = (size_t)c.nf;
        int32_t code[Q];
        load_codes<Q>(code, c, k);
#pragma unroll
        for (int i = 1; i < Q; ++i) {
            const int32_t co = code[D > 0 ? L::opp(i) : i];
            const bool fl = co >= 0;
            (dst + (size_t)(fl ? L::opp(i) : i) * NF)[fl ? co : k] = v[i];
        }
    } else {
        const uint32_t NF = (uint32_t)c.nf;
        Neighbours<Q> nb;
        window_neighbours<Q>(nb, c, nd.blk, k, nd.pos);
#pragma unroll
        for (int i = 1; i < Q; ++i) {
            const int n = D > 0 ? L::opp(i) : i;
            dst[nb.fluid(n) ? (uint32_t)L::opp(i) * NF + nb.j[n] : (uint32_t)i * NF + (uint32_t)k] = v[i];
        }
    }
}

// Stores what a node sends: into its own slots (natural), to its neighbours
// (swapped: g_i(x) to (x + c_i, opp(i)) where that node is fluid), or into
// the caller's dense array.
template <int Q, typename T, int OUT>
__device__ __forceinline__ void store_node(T* dst, const T (&v)[Q], const Node& nd, const Cmp& c, const BCmpInst* I)
{
    if (OUT == kOutScatter) {
        store_scattered<Q, T, 1>(dst, v, nd, c);
        return;
    }
    const long long n = OUT == kOutDense ? I->f_off + (long long)c.idx[nd.k] : (long long)nd.k;
    const size_t S = OUT == kOutDense ? (size_t)I->g.N : (size_t)c.nf;
#pragma unroll
    for (int i = 0; i < Q; ++i) dst[(size_t)i * S + n] = v[i];
}

// The velocity of an Eq. 6 node's output, for the next in-place step.
template <int Q, typename T>
__device__ __forceinline__ void keep_velocity(const T (&v)[Q], const Side& sd, const Bc& bc, const BCmpInst* I)
{
    T drho, rho, u[3];
    moments<Q, T>(v, drho, rho, u);
    T* e = side_entry<T>(bc, *I, sd);
    e[0] = u[0];
    e[1] = u[1];
    e[2] = u[2];
}

// The order in which the thread blocks take the node blocks: the boundary
// columns (the last ones of a lattice), whose update is the longest, first;
// then the interior, upwards or (rev) downwards.  Alternating the direction
// from launch to launch starts each launch on what the one before left in
// the L2 cache (a batch's launches carry no time level and all go upwards).
struct CmpOrder {
    unsigned n, first;  // node blocks; how many of the last come first
    int rev;
    __device__ __forceinline__ unsigned block(unsigned b) const { return b < first || rev ? n - 1 - b : b - first; }
};

// Adjoint step in the compact layout: the gather form of adjoint.cu.  The
// forward copies f*_j(x) to x + c_j, the node that pulls direction j from x;
// its compact index is the code of direction opp(j) at x (x + c_j = x - c_opp(j)).
// mu_j(x) is lambda^{t+1}_j(x + c_j) where that node is fluid, else
// lambda^{t+1}_opp(j)(x), at slot (x, opp(j)) in both layouts (with the sign
// and the velocity terms of Eq. 6 in the boundary columns).  IN gather: f^t
// and mu from the neighbours, lambda^t to OUT (own: the two-buffer pull;
// scatter: the gather step in place); IN local: both from x's own slots,
// lambda^t to its own slots.  lam_in and lam_out may be the same buffer (in
// place: each node reads all it needs before it writes the same slots).
// Every load of f^t and lambda depends only on the neighbours, so all 2 Q
// are in flight together.

// f^t and mu of an interior node.
template <int Q, typename T, bool T0, int IN, bool CG>
__device__ __forceinline__ void pull_adjoint(T (&f)[Q], T (&mu)[Q], const T* gprev, const T* lam_in, int32_t k,
                                             uint32_t NF, const Neighbours<Q>& nb)
{
    using L = Lattice<Q>;
    if (!T0) pull_interior<Q, T, IN, CG>(f, gprev, k, NF, nb);
    mu[0] = ld_state<CG>(lam_in + k);
#pragma unroll
    for (int i = 1; i < Q; ++i) {
        const int o = L::opp(i);
        const bool fl = IN == kInGather && nb.fluid(o);
        mu[i] = ld_state<CG>(lam_in + (fl ? (uint32_t)i * NF + nb.j[o] : (uint32_t)o * NF + (uint32_t)k));
    }
}

// f^t and mu of a boundary-column node, and the velocity terms G of its
// Eq. 6 links; adds its inlet gradient term (one owner per inlet node).
template <int Q, typename T, bool T0, int IN, bool CG>
__device__ __forceinline__ void pull_adjoint_table(T (&f)[Q], T (&mu)[Q], T (&G)[3], const T* gprev, const T* lam_in,
                                                   int32_t k, const Wall& wall, const int32_t (&code)[Q],
                                                   const Cmp& c, const BCmpInst* I, const Bc& tmpl,
                                                   double* __restrict__ grad_acc)
{
    using L = Lattice<Q>;
    const size_t NF = (size_t)c.nf;
    mu[0] = ld_state<CG>(lam_in + k);
#pragma unroll
    for (int i = 1; i < Q; ++i) {
        const int o = L::opp(i);
        const bool fl = IN == kInGather && code[o] >= 0;
        mu[i] = ld_state<CG>(lam_in + (size_t)(fl ? i : o) * NF + (fl ? code[o] : k));
    }
    // the segment states are read-only here: the velocity comes from gprev, not from the side array
    if (!T0) pull_table<Q, T, IN, CG>(f, gprev, k, wall, NF, code, tmpl, I, false);
    T drho, rho, u[3];
    moments<Q, T>(f, drho, rho, u);
    const T uu = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
    const T rwT = T(wall.rw);
    double sum = 0.0;
    if constexpr (std::is_same<T, double>::value) {
        // opposite links together, as in apply_eq6 (FP32 keeps the order of its sums)
#pragma unroll
        for (int i = 1; i < Q; ++i) {
            if (L::c(i, 0) != 1) continue;
            const int o = L::opp(i);
            const bool here = code[i] == kCmpABB;
            if ((!here && code[o] != kCmpABB) || (here && tmpl.vel_inlet)) continue;
            const T li = here ? mu[o] : mu[i];
            if (here) mu[o] = -li;
            else mu[i] = -li;
            const T cu = cdot<Q, T>(i, u), lw = T(2.0 * L::w(i)) * li;
            if (here) sum += lw * (T(1) + T(4.5) * cu * cu - T(1.5) * uu);
            const T lr = lw * rwT, l9 = T(9) * cu * lr, l3 = T(3) * lr;
#pragma unroll
            for (int a = 0; a < L::D; ++a) {
                G[a] -= l3 * u[a];
                if (L::c(i, a) != 0) G[a] = L::c(i, a) > 0 ? G[a] + l9 : G[a] - l9;
            }
        }
        if (wall.sd.xin) atomicAdd(grad_acc + I->acc_off + wall.sd.row, sum);
        return;
    }
#pragma unroll
    for (int j = 1; j < Q; ++j) {
        const int o = L::opp(j);
        if (L::c(o, 0) == 0 || code[o] != kCmpABB) continue;
        if (wall.sd.xin && tmpl.vel_inlet) continue;  // the velocity inlet's source is constant
        const T li = mu[j];
        mu[j] = -li;
        const T cu = cdot<Q, T>(o, u);
        const T two_w = T(2.0 * L::w(o));
        if (wall.sd.xin) sum += (double)(li * two_w * (T(1) + T(4.5) * cu * cu - T(1.5) * uu));
#pragma unroll
        for (int a = 0; a < L::D; ++a) G[a] += li * two_w * rwT * (T(9) * cu * T(L::c(o, a)) - T(3) * u[a]);
    }
    if (wall.sd.xin) atomicAdd(grad_acc + I->acc_off + wall.sd.row, sum);
}

// lambda^t of a node from f^t, mu and G (the transpose of the collision),
// stored; returns its dL/domega term.
template <int Q, typename T, int OUT, bool DENSE_ROUND>
__device__ __forceinline__ T adjoint_node(const T (&f)[Q], const T (&mu)[Q], const T (&G)[3], T* lam_out,
                                          const Node& nd, const Cmp& c, const Bc& tmpl, T omega)
{
    T drho, rho, u[3];
    moments<Q, T>(f, drho, rho, u);
    T lam[Q];
    const T dom = adjoint_collision<Q, T, DENSE_ROUND>(f, mu, drho, rho, u, G, omega, lam, tmpl);
    if (OUT == kOutScatter) {  // lambda_m(x) to (x - c_m, opp(m)) where that node is fluid
        store_scattered<Q, T, -1>(lam_out, lam, nd, c);
    } else {
        lam_out[nd.k] = lam[0];
#pragma unroll
        for (int m = 1; m < Q; ++m) (lam_out + (size_t)m * (size_t)c.nf)[nd.k] = lam[m];
    }
    return dom;
}

// One FP64 partial per warp (its sum in T, or to FP64 accuracy where wide),
// accumulated in place across time steps: no block barrier, so a warp that finishes early frees its slot at
// once instead of waiting for the slowest warp of the block.  The warp of
// compact node k owns slot k >> 5 (lane 0 holds the warp's first node).  The
// addition is a reduction at the L2 cache, whose result nothing waits for:
// each slot has one per launch, so the order of additions is the order of the
// launches.
template <typename T>
__device__ __forceinline__ void add_warp_partial(T dom, bool live, long long k, double* __restrict__ partial,
                                                 bool wide)
{
    const double dw = warp_total(dom, wide);
    if ((threadIdx.x & 31) == 0 && live) atomicAdd(partial + (k >> 5), dw);
}

// Reverse of the extrapolated Eq. 6 velocity in the compact layout: the
// per-row pass of adjoint.cu (k_adjoint_uw), with the boundary node found
// through cmap and its inward neighbour through its own table entry.
template <int Q, typename T>
__global__ void __launch_bounds__(kCmpThreads)
    k_adjoint_uw_cmp(const T* gprev, const T* lam_in, T* lam_out, Cmp c,
                     const int32_t* __restrict__ cmap, Geo g, Bc bc, double* __restrict__ grad_acc)
{
    pdl_enter();
    const long long row = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (row >= (long long)g.ny * g.nz) return;
    const size_t NF = (size_t)c.nf;
    for (int side = 0; side < 2; ++side) {
        const bool xin = side == 0;
        if (xin && bc.vel_inlet) continue;  // the velocity inlet does not use u_w
        const int32_t kb = cmap[row * g.nx + (xin ? 0 : g.nx - 1)];
        if (kb < 0) continue;
        int32_t cb[Q], ce[Q];
        load_codes<Q>(cb, c, kb);
        const int32_t ke = cb[inward_dir<Q>(xin)];
        if (ke < 0) continue;  // inward neighbour solid: u_w is the node's own velocity
        T fb[Q], fe[Q], li[Q];
        load_codes<Q>(ce, c, ke);
        Wall wb, we;  // x_b + e is a boundary node itself only where nx = 2
        wb.sd = Side{xin, row};
        we.sd = Side{!xin, row};
        wb.rw = xin ? bc.rho_in[bc.profile ? row : 0] : bc.rho_out;
        we.rw = !xin ? bc.rho_in[bc.profile ? row : 0] : bc.rho_out;
        pull_table<Q, T, kInGather, false>(fb, gprev, kb, wb, NF, cb, bc, nullptr, false);
        pull_table<Q, T, kInGather, false>(fe, gprev, ke, we, NF, ce, bc, nullptr, false);
        uint32_t eq6 = 0;
        li[0] = T(0);
#pragma unroll
        for (int i = 1; i < Q; ++i) {
            const bool on = cb[i] == kCmpABB;
            eq6 |= on ? (1u << i) : 0u;
            li[i] = on ? lam_in[(size_t)i * NF + kb] : T(0);
        }
        const T rw = T(xin ? (bc.profile ? bc.rho_in[row] : bc.rho_in[0]) : bc.rho_out);
        T db[Q], de[Q];
        const double dg = adjoint_uw_delta<Q, T>(fb, fe, li, eq6, rw, db, de);
#pragma unroll
        for (int k = 0; k < Q; ++k) {
            lam_out[(size_t)k * NF + kb] += db[k];
            lam_out[(size_t)k * NF + ke] += de[k];
        }
        if (xin) grad_acc[row] += dg;
    }
}

// --------------------------------------------- the kernels, lattices and batches
//
// The kernels below serve a single lattice and a packed batch alike.  A
// block's nodes belong to one instance (blks[block]; a single lattice passes
// no block table and is instance 0), whose entry gives its sizes, the
// offsets of its inlet data and dense arrays, and its tau.  A single lattice
// is a pack of one, so a batch instance gets bit for bit what a single plan
// computes: the same kernels run the same per-node code.

static_assert(kBatchCmpAlign == kCmpThreads, "one thread block per aligned node range of a batch instance");

// FP64 nodes hold twice the registers: half the blocks per SM.
template <typename T>
constexpr int kMinBlocks = sizeof(T) == 8 ? 2 : 4;

// What bounds these kernels.  Lattices that live in the L2 cache (up to
// about a million nodes): the chain wait, loads, arithmetic, stores of one
// launch, and in it the longest thread, a boundary-column node; its loads are
// all in flight together and its launch starts it first (D3Q19 128x64x64: a
// time step of a gradient evaluation 62.5 -> 24.1 us; the 400x160 MRT wake
// 21.5 -> 8.7 us).  Larger ones: memory, with the windows' integer work
// beside it (D3Q19 512x256x256: step 549 -> 469 us, adjoint 874 -> 833 us of
// kernel time; D2Q9: see the pipelined forms).

// One step.  MODE: stream-collide, collide-only (from the instance's dense
// [Q][N] array) or stream-only (step.cu); IN / OUT: the addressing of the
// input and output states (two-buffer pull: gather /
// own; in place: gather / scatter, then local / own; OUT dense: the caller's
// array, solid entries left to the caller).  src == dst is allowed for the
// in-place pairs: the slot sets of different nodes are disjoint, and a node
// loads every slot it owns before it stores any (each stored value depends
// on all loaded ones through the moments), so no load can see a store of the
// same launch.  The state pointers are not __restrict__: the compiler may not
// turn state loads into non-coherent ones, which could move above the wait
// for the preceding launch, or (in place) hit a line that another block has
// rewritten since.  Padding nodes of a batch are skipped: nothing ever reads
// them.
template <int Q, typename T, int MODE, int IN, int OUT, bool DENSE_ROUND>
__global__ void __launch_bounds__(kCmpThreads, kMinBlocks<T>)
    k_step_cmp(const T* src, T* dst, Cmp c, CmpBlk lat, const BCmpInst* __restrict__ insts,
               const CmpBlk* __restrict__ blks, Bc tmpl, const double* __restrict__ tau, CmpOrder ord)
{
    const int32_t k = (int32_t)(ord.block(blockIdx.x) * blockDim.x + threadIdx.x);
    const Node nd = node_of(k, c, lat, blks);
    if (!nd.live()) {
        pdl_enter();
        return;
    }
    const BCmpInst* I = insts + nd.blk.inst;
    const T omega = relaxation_rate<T>(tau[nd.blk.inst], Q == 9 && tmpl.wide);
    const bool side = tmpl.side_u != nullptr;
    T v[Q];
    Wall wall;
    if (MODE == kCollideOnly) {
        if (side && eq6_bit(c, k)) wall.sd = side_of(c.idx, k, I->g);
        pdl_enter();
        const T* s = src + I->f_off + c.idx[k];
        const size_t S = (size_t)I->g.N;
#pragma unroll
        for (int i = 0; i < Q; ++i) v[i] = s[(size_t)i * S];
    } else if (!nd.bnd()) {
        Neighbours<Q> nb;
        if (IN == kInGather) window_neighbours<Q>(nb, c, nd.blk, k, nd.pos);
        pdl_enter();
        pull_interior<Q, T, IN, kInPlace<IN, OUT>>(v, src, k, (uint32_t)c.nf, nb);
    } else {
        int32_t code[Q];
        wall = boundary_codes<Q>(code, nd, c, insts, tmpl);
        pdl_enter();
        pull_table<Q, T, IN, kInPlace<IN, OUT>>(v, src, k, wall, (size_t)c.nf, code, tmpl, I, side);
    }
    if (MODE != kStreamOnly) collide_any<Q, T, DENSE_ROUND>(v, omega, tmpl);
    store_node<Q, T, OUT>(dst, v, nd, c, I);
    if (MODE != kStreamOnly && side && (MODE == kCollideOnly || nd.bnd()) && eq6_bit(c, k))
        keep_velocity<Q, T>(v, wall.sd, tmpl, I);
}

// Pipelined forms of the two-buffer step and adjoint step, for lattices of
// several nodes per thread.  A CTA walks every gridDim.x-th node block of 128
// nodes.  Blocks that hold boundary-column (or padding) nodes come first and
// go node by node; on the others, all interior, a thread has in flight, while
// it computes a node: the populations of the next one, the windows of the one
// after, and the position of the one after that.  One node per thread leaves a
// warp three dependent trips to memory (position, windows, populations) and
// only then its arithmetic, with too few bytes in flight per SM to fill the
// memory pipe: D2Q9 4096x2048, 5.0 M fluid nodes, stream-collide 103 -> 64 us
// (340 MB of DRAM traffic, 0.79 of the measured copy bandwidth), adjoint
// 174 -> 104 us; the 64-lattice batch 178 -> 138 and 284 -> 198 us.
template <typename T>
struct PipeArgs {
    const T *src, *lam_in;  // the state pulled from (g^{t-1}); lambda^{t+1}
    T* out;
    Cmp c;
    CmpBlk lat;
    const BCmpInst* insts;
    const CmpBlk* blks;     // batches: node blocks of 256, those with boundary or padding nodes first
    Bc tmpl;
    const double* tau;
    double *grad_acc, *partial;
    CmpOrder ord;
};

constexpr int kPipeThreads = 128;

// The b-th node block in order: its first node, instance and windows.  (A
// single lattice's are the same for every block.)
template <typename T, bool BATCH>
__device__ __forceinline__ CmpBlk pipe_block(const PipeArgs<T>& A, unsigned b)
{
    if (!BATCH) return CmpBlk{A.lat.inst, A.lat.w_row, A.lat.w_plane, (int)(A.ord.block(b) * kPipeThreads)};
    const unsigned p = b < A.ord.first || !A.ord.rev ? b : A.ord.n - 1 - (b - A.ord.first);
    const int4 v = __ldg(reinterpret_cast<const int4*>(A.blks) + (p >> 1));
    return CmpBlk{v.x, v.y, v.z, v.w * kCmpThreads + (int)(p & 1u) * kPipeThreads};
}

template <int Q, typename T, bool BATCH>
struct Ahead {
    CmpBlk k1, k2, k3;   // the next node blocks; k4 follows (batches read it a step earlier)
    CmpBlk k4;
    uint32_t p1, p2, p3; // their nodes' positions
    Windows<Q> w2;
    unsigned b;          // order of k4

    __device__ __forceinline__ CmpBlk block(const PipeArgs<T>& A, unsigned at) const
    {
        return pipe_block<T, BATCH>(A, at < A.ord.n ? at : A.ord.n - 1);  // past the end: read again, not used
    }
    __device__ __forceinline__ int32_t node(const CmpBlk& k) const { return k.pad + (int32_t)threadIdx.x; }
    // the positions and windows that the first nodes' loads need, before the wait
    __device__ __forceinline__ void start(const PipeArgs<T>& A, unsigned b0)
    {
        k2 = block(A, b0);
        k3 = block(A, b0 + gridDim.x);
        b = b0 + 2 * gridDim.x;
        k4 = block(A, b);
        p2 = __ldg(A.c.pos + node(k2));
        p3 = __ldg(A.c.pos + node(k3));
        load_windows<Q>(w2, A.c, k2, p2);
    }
    // on by one node: n1's neighbours, with n2's windows and n3's position on their way
    __device__ __forceinline__ void next(const PipeArgs<T>& A, Neighbours<Q>& nb)
    {
        k1 = k2;
        p1 = p2;
        neighbours_of<Q>(nb, w2, A.c, k1, node(k1), p1);
        k2 = k3;
        p2 = p3;
        load_windows<Q>(w2, A.c, k2, p2);
        k3 = k4;
        p3 = __ldg(A.c.pos + node(k3));
        b += gridDim.x;
        k4 = block(A, b);
    }
};

// One node of a block with boundary or padding nodes.
template <int Q, typename T, bool BATCH, bool DENSE_ROUND>
__device__ __forceinline__ void pipe_step_node(const PipeArgs<T>& A, unsigned b)
{
    Node nd;
    nd.blk = pipe_block<T, BATCH>(A, b);
    nd.k = nd.blk.pad + (int32_t)threadIdx.x;
    nd.pos = nd.k < (int32_t)A.c.nf ? __ldg(A.c.pos + nd.k) : kPosDead;
    if (!nd.live()) return;
    const BCmpInst* I = A.insts + nd.blk.inst;
    T v[Q];
    if (nd.bnd()) {
        int32_t code[Q];
        const Wall wall = boundary_codes<Q>(code, nd, A.c, A.insts, A.tmpl);
        pull_table<Q, T, kInGather, false>(v, A.src, nd.k, wall, (size_t)A.c.nf, code, A.tmpl, I, false);
    } else {
        Neighbours<Q> nb;
        window_neighbours<Q>(nb, A.c, nd.blk, nd.k, nd.pos);
        pull_interior<Q, T, kInGather, false>(v, A.src, nd.k, (uint32_t)A.c.nf, nb);
    }
    collide_any<Q, T, DENSE_ROUND>(v, relaxation_rate<T>(A.tau[nd.blk.inst], Q == 9 && A.tmpl.wide), A.tmpl);
    store_node<Q, T, kOutOwn>(A.out, v, nd, A.c, I);
}

template <int Q, typename T, bool BATCH, bool DENSE_ROUND, int MINB>
__global__ void __launch_bounds__(kPipeThreads, MINB) k_step_cmp_pipe(const __grid_constant__ PipeArgs<T> A)
{
    unsigned b = blockIdx.x;
    if (b < A.ord.first) {
        pdl_enter();
        for (; b < A.ord.first; b += gridDim.x) pipe_step_node<Q, T, BATCH, DENSE_ROUND>(A, b);
        if (b >= A.ord.n) return;
    }
    Ahead<Q, T, BATCH> a;
    a.start(A, b);
    int cur = a.k2.inst;
    T omega = relaxation_rate<T>(A.tau[cur], Q == 9 && A.tmpl.wide);
    pdl_enter();
    const uint32_t NF = (uint32_t)A.c.nf;
    auto fetch = [&](T(&v)[Q]) {
        Neighbours<Q> nb;
        a.next(A, nb);
        pull_interior<Q, T, kInGather, false>(v, A.src, a.node(a.k1), NF, nb);
    };
    auto update = [&](const CmpBlk& blk, T(&v)[Q]) {
        if (BATCH && blk.inst != cur) {
            cur = blk.inst;
            omega = relaxation_rate<T>(A.tau[cur], Q == 9 && A.tmpl.wide);
        }
        collide_any<Q, T, DENSE_ROUND>(v, omega, A.tmpl);
        const int32_t k = a.node(blk);
#pragma unroll
        for (int i = 0; i < Q; ++i) (A.out + (size_t)i * (size_t)A.c.nf)[k] = v[i];
    };
    T v0[Q], v1[Q];
    fetch(v0);
    while (true) {
        CmpBlk blk = a.k1;
        if ((b += gridDim.x) >= A.ord.n) {
            update(blk, v0);
            return;
        }
        fetch(v1);
        update(blk, v0);
        blk = a.k1;
        if ((b += gridDim.x) >= A.ord.n) {
            update(blk, v1);
            return;
        }
        fetch(v0);
        update(blk, v1);
    }
}

// One node of a block with boundary or padding nodes; every thread calls it.
template <int Q, typename T, bool BATCH, bool DENSE_ROUND>
__device__ __forceinline__ void pipe_adjoint_node(const PipeArgs<T>& A, unsigned b)
{
    Node nd;
    nd.blk = pipe_block<T, BATCH>(A, b);
    nd.k = nd.blk.pad + (int32_t)threadIdx.x;
    nd.pos = nd.k < (int32_t)A.c.nf ? __ldg(A.c.pos + nd.k) : kPosDead;
    T dom = T(0);
    if (nd.live()) {
        T f[Q], mu[Q], G[3] = {T(0), T(0), T(0)};
        if (nd.bnd()) {
            int32_t code[Q];
            const Wall wall = boundary_codes<Q>(code, nd, A.c, A.insts, A.tmpl);
            pull_adjoint_table<Q, T, false, kInGather, false>(f, mu, G, A.src, A.lam_in, nd.k, wall, code, A.c,
                                                              A.insts + nd.blk.inst, A.tmpl, A.grad_acc);
        } else {
            Neighbours<Q> nb;
            window_neighbours<Q>(nb, A.c, nd.blk, nd.k, nd.pos);
            pull_adjoint<Q, T, false, kInGather, false>(f, mu, A.src, A.lam_in, nd.k, (uint32_t)A.c.nf, nb);
        }
        dom = adjoint_node<Q, T, kOutOwn, DENSE_ROUND>(f, mu, G, A.out, nd, A.c, A.tmpl, relaxation_rate<T>(A.tau[nd.blk.inst], Q == 9 && A.tmpl.wide));
    }
    add_warp_partial<T>(dom, nd.k < (int32_t)A.c.nf, nd.k, A.partial, Q == 9 && A.tmpl.wide);
}

template <int Q, typename T, bool BATCH, bool DENSE_ROUND, int MINB>
__global__ void __launch_bounds__(kPipeThreads, MINB) k_adjoint_cmp_pipe(const __grid_constant__ PipeArgs<T> A)
{
    unsigned b = blockIdx.x;
    if (b < A.ord.first) {
        pdl_enter();
        for (; b < A.ord.first; b += gridDim.x) pipe_adjoint_node<Q, T, BATCH, DENSE_ROUND>(A, b);
        if (b >= A.ord.n) return;
    }
    Ahead<Q, T, BATCH> a;
    a.start(A, b);
    int cur = a.k2.inst;
    T omega = relaxation_rate<T>(A.tau[cur], Q == 9 && A.tmpl.wide);
    pdl_enter();
    const uint32_t NF = (uint32_t)A.c.nf;
    auto fetch = [&](T(&f)[Q], T(&mu)[Q]) {
        Neighbours<Q> nb;
        a.next(A, nb);
        pull_adjoint<Q, T, false, kInGather, false>(f, mu, A.src, A.lam_in, a.node(a.k1), NF, nb);
    };
    auto update = [&](const CmpBlk& blk, T(&f)[Q], T(&mu)[Q]) {
        if (BATCH && blk.inst != cur) {
            cur = blk.inst;
            omega = relaxation_rate<T>(A.tau[cur], Q == 9 && A.tmpl.wide);
        }
        const T G[3] = {T(0), T(0), T(0)};
        Node nd;
        nd.k = a.node(blk);
        const T dom = adjoint_node<Q, T, kOutOwn, DENSE_ROUND>(f, mu, G, A.out, nd, A.c, A.tmpl, omega);
        add_warp_partial<T>(dom, true, nd.k, A.partial, Q == 9 && A.tmpl.wide);
    };
    T f0[Q], m0[Q], f1[Q], m1[Q];
    fetch(f0, m0);
    while (true) {
        CmpBlk blk = a.k1;
        if ((b += gridDim.x) >= A.ord.n) {
            update(blk, f0, m0);
            return;
        }
        fetch(f1, m1);
        update(blk, f0, m0);
        blk = a.k1;
        if ((b += gridDim.x) >= A.ord.n) {
            update(blk, f1, m1);
            return;
        }
        fetch(f0, m0);
        update(blk, f1, m1);
    }
}

// One adjoint step; the warp partials of an instance occupy slots
// [k0 / 32, (k0 + nf + 31) / 32).  lam_in == lam_out is allowed for the
// in-place pairs (as for k_step_cmp: disjoint slot sets, all loads of a node
// before its stores).
template <int Q, typename T, bool T0, int IN, int OUT, bool DENSE_ROUND>
__global__ void __launch_bounds__(kCmpThreads, kMinBlocks<T>)
    k_adjoint_cmp(const T* gprev, const T* lam_in, T* lam_out, Cmp c, CmpBlk lat,
                  const BCmpInst* __restrict__ insts, const CmpBlk* __restrict__ blks, Bc tmpl,
                  const double* __restrict__ tau, double* __restrict__ grad_acc, double* __restrict__ partial,
                  CmpOrder ord)
{
    constexpr bool CG = kInPlace<IN, OUT>;
    const int32_t k = (int32_t)(ord.block(blockIdx.x) * blockDim.x + threadIdx.x);
    const Node nd = node_of(k, c, lat, blks);
    T f[Q], mu[Q], G[3] = {T(0), T(0), T(0)};
    if (T0) {
#pragma unroll
        for (int i = 0; i < Q; ++i) f[i] = T(0);
    }
    T omega = T(0);
    if (nd.live()) omega = relaxation_rate<T>(tau[nd.blk.inst], Q == 9 && tmpl.wide);
    if (nd.interior()) {
        Neighbours<Q> nb;
        if (IN == kInGather) window_neighbours<Q>(nb, c, nd.blk, k, nd.pos);
        pdl_enter();
        pull_adjoint<Q, T, T0, IN, CG>(f, mu, gprev, lam_in, k, (uint32_t)c.nf, nb);
    } else if (nd.live()) {
        int32_t code[Q];
        const Wall wall = boundary_codes<Q>(code, nd, c, insts, tmpl);
        pdl_enter();
        pull_adjoint_table<Q, T, T0, IN, CG>(f, mu, G, gprev, lam_in, k, wall, code, c, insts + nd.blk.inst, tmpl,
                                             grad_acc);
    } else {
        pdl_enter();
    }
    T dom = T(0);
    if (nd.live()) dom = adjoint_node<Q, T, OUT, DENSE_ROUND>(f, mu, G, lam_out, nd, c, tmpl, omega);
    add_warp_partial<T>(dom, k < (int32_t)c.nf, k, partial, Q == 9 && tmpl.wide);
}

// The last launch of a sweep of a single lattice: stream-only into the
// caller's dense array, one thread per dense node, solid entries zero, so that
// every sector is written once and whole (written by compact node, after a
// memset, 512x256x256 took 1008 + 380 us).
template <int Q, typename T, int IN>
__global__ void __launch_bounds__(kCmpThreads, kMinBlocks<T>)
    k_stream_dense(const T* src, T* __restrict__ dst, Cmp c, CmpBlk lat, const BCmpInst* __restrict__ insts,
                   const int32_t* __restrict__ cmap, long long N, Bc tmpl)
{
    pdl_enter();
    const long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= N) return;
    const int32_t k = __ldg(cmap + n);
    T v[Q];
#pragma unroll
    for (int i = 0; i < Q; ++i) v[i] = T(0);
    if (k >= 0) {
        const Node nd = node_of(k, c, lat, nullptr);
        if (!nd.bnd()) {
            Neighbours<Q> nb;
            if (IN == kInGather) window_neighbours<Q>(nb, c, lat, k, nd.pos);
            pull_interior<Q, T, IN, IN == kInLocal>(v, src, k, (uint32_t)c.nf, nb);
        } else {
            int32_t code[Q];
            const Wall wall = boundary_codes<Q>(code, nd, c, insts, tmpl);
            pull_table<Q, T, IN, IN == kInLocal>(v, src, k, wall, (size_t)c.nf, code, tmpl, insts, false);
        }
    }
#pragma unroll
    for (int i = 0; i < Q; ++i) dst[(size_t)i * (size_t)N + n] = v[i];
}

// The caller's dense arrays (packed, for a batch) -> the compact state
// (ADD: added to it).  SWAP: into the swapped lambda layout (lambda_d(x) to
// (x - c_d, opp(d)) where that node is fluid), the layout of lambda^t at odd
// t in the in-place reverse sweep.
template <int Q, typename T, bool ADD, bool SWAP>
__global__ void __launch_bounds__(kCmpThreads)
    k_cmp_gather(const T* __restrict__ dense, T* __restrict__ cmp, Cmp c, const BCmpInst* __restrict__ insts,
                 const CmpBlk* __restrict__ blks)
{
    using L = Lattice<Q>;
    const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const BCmpInst I = insts[blks && k < c.nf ? blks[k / kCmpThreads].inst : 0];
    if (k >= I.k0 + I.nf) return;
    const long long n = c.idx[k];
    for (int d = 0; d < Q; ++d) {
        const T v = dense[I.f_off + (long long)d * I.g.N + n];
        long long slot = (long long)d * c.nf + k;
        if (SWAP && d > 0) {
            const int32_t co = c.nbr[(long long)(d - 1) * c.nf + k];
            if (co >= 0) slot = (long long)L::opp(d) * c.nf + co;
        }
        if (ADD) cmp[slot] += v;
        else cmp[slot] = v;
    }
}

// One instance's tables (built by compact_build) into the packed arrays:
// dense indices as they are, neighbour codes and window indices shifted by
// the instance's k0, positions by its first window w0.
__global__ void __launch_bounds__(256) k_bpack_cmp(Cmp l, int q, long long k0, long long nfp, unsigned w0,
                                                   int32_t* __restrict__ idx, int32_t* __restrict__ nbr,
                                                   uint32_t* __restrict__ pos, bool windows)
{
    const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= l.nf) return;
    idx[k0 + k] = l.idx[k];
    pos[k0 + k] = !windows || (l.pos[k] & kPosBnd) == kPosBnd ? kPosBnd : l.pos[k] + (w0 << 7);
    for (int d = 0; d < q - 1; ++d) {
        const int32_t code = l.nbr[(long long)d * l.nf + k];
        nbr[(long long)d * nfp + k0 + k] = code >= 0 ? (int32_t)(code + k0) : code;
    }
}

__global__ void __launch_bounds__(256) k_bpack_windows(Cmp l, long long n_win, int k0, uint2* __restrict__ win,
                                                       int2* __restrict__ edge)
{
    const long long w = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (w >= n_win) return;
    const uint2 q = l.win[w];
    const int2 e = l.edge[w];
    win[w] = make_uint2(q.x, q.y + (uint32_t)k0);
    edge[w] = make_int2(e.x < 0 ? e.x : e.x + k0, e.y < 0 ? e.y : e.y + k0);
}

unsigned cmp_grid(long long nf) { return (unsigned)((nf + kCmpThreads - 1) / kCmpThreads); }

// The launch of a single lattice: a pack of one (no block table).
BCmpArgs single_args(const PlanInfo& p, uint32_t* status)
{
    BCmpArgs a = {};
    a.c = p.cmp;
    a.insts = p.cmp_inst;
    a.blks = nullptr;
    a.lat = p.cmp_lat;
    a.dense_round = p.dense_round && !p.uw_extrap;
    a.n_int = (unsigned)p.cmp_int;
    a.n_blocks = cmp_grid(p.cmp.nf);
    a.q = p.q;
    a.prec = p.prec;
    a.pdl = p.pdl;
    a.status = status;
    return a;
}

// The sweeps use: stream-collide compact -> compact (two-buffer pull
// natural -> natural, or the in-place pair natural -> swapped, swapped ->
// natural); collide-only from the caller's dense array into compact;
// stream-only into the caller's dense array (batches from here, by compact
// node; single lattices through k_stream_dense).
// Threads per block of the one-node-per-thread kernels.  Below one wave small
// blocks spread the few warps evenly over the SMs (128x64 to 512x256 D2Q9:
// 64 threads 6.3 to 7.7 us per time step of a gradient evaluation, 256
// threads 6.7 to 8.4); above it 128 were fastest on D2Q9 (1024x512: 15.5 us,
// 16.7 with 256) and 256 on D3Q19 (128x64x64: 24.1 us, 24.6 with 128).  FP64
// small lattices take single warps: the SM with the most of them sets the time.
unsigned cmp_threads(int q, int prec, long long nf)
{
    if (nf < 100000) return prec == 8 ? 32 : 64;
    return q == 9 ? 128 : 256;
}

// The pipelined kernels, from 600000 nodes (6 to 8 per resident thread at 4
// and 5 CTAs on each of 152 SMs; the line lies between two measured sizes):
// D2Q9 FP32 2048x1024, 1.3 M fluid nodes, takes 58.9 us per time step of a
// gradient evaluation with them and 71.5 with one node per thread, 1024x512,
// 0.3 M, 17.6 and 16.6.  D3Q19 stays
// with one node per thread: two nodes' populations in registers leave 16
// warps per SM (512x256x256: 1829 us per step, pipelined 2085).
template <int Q, typename T>
constexpr bool kPipe = Q == 9 && std::is_same<T, float>::value;

bool pipe_step(const BCmpArgs& a) { return a.c.nf >= 600000; }

CmpOrder cmp_order(const BCmpArgs& a, unsigned threads, int t)
{
    CmpOrder o;
    o.n = (unsigned)((a.c.nf + threads - 1) / threads);
    o.first = a.blks ? 0 : o.n - a.n_int / threads;
    o.rev = t & 1;
    return o;
}

// A pipelined launch: as many CTAs as fit on the GPU at once.
template <class K, typename T>
void launch_pipe(bool pdl, K kernel, const PipeArgs<T>& A, cudaStream_t s)
{
    int dev = 0, sms = 0, per_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, kPipeThreads, 0);
    const unsigned ctas = (unsigned)(std::max(per_sm, 1) * std::max(sms, 1));
    launch_k(pdl, kernel, dim3(std::min(ctas, A.ord.n)), dim3(kPipeThreads), 0, s, A);
}

CmpOrder pipe_order(const BCmpArgs& a, int t)
{
    CmpOrder o = cmp_order(a, kPipeThreads, t);
    if (a.blks) o.first = a.n_mixed * (kBatchCmpAlign / kPipeThreads);
    return o;
}

template <int Q, typename T, bool DENSE_ROUND>
void launch_step_as(const BCmpArgs& a, int mode, const void* src, void* dst, int lin, int lout, const Bc& tmpl,
                    const double* tau, cudaStream_t s)
{
    const T* x = static_cast<const T*>(src);
    T* y = static_cast<T*>(dst);
    const unsigned threads = cmp_threads(Q, (int)sizeof(T), a.c.nf);
    const CmpOrder ord = cmp_order(a, threads, tmpl.t_level);
    const dim3 grid(ord.n), block(threads);
    const bool swap_in = lin == kLayoutSwapped, swap_out = lout == kLayoutSwapped;
    auto go = [&](auto kernel) {
        launch_k(a.pdl, kernel, grid, block, 0, s, x, y, a.c, a.lat, a.insts, a.blks, tmpl, tau, ord);
    };
    if (mode == kStreamCollide) {
        if (swap_in) {  // the local step: its interior nodes read their own slots
            go(k_step_cmp<Q, T, kStreamCollide, kInLocal, kOutOwn, DENSE_ROUND>);
            return;
        }
        if constexpr (kPipe<Q, T>) {
            if (!swap_out && pipe_step(a)) {
                constexpr int MINB = 5;
                const PipeArgs<T> A{x, nullptr, y, a.c, a.lat, a.insts, a.blks_by_class, tmpl, tau, nullptr, nullptr,
                                    pipe_order(a, tmpl.t_level)};
                if (a.blks) launch_pipe(a.pdl, k_step_cmp_pipe<Q, T, true, DENSE_ROUND, MINB>, A, s);
                else launch_pipe(a.pdl, k_step_cmp_pipe<Q, T, false, DENSE_ROUND, MINB>, A, s);
                return;
            }
        }
        if (swap_out) go(k_step_cmp<Q, T, kStreamCollide, kInGather, kOutScatter, DENSE_ROUND>);
        else go(k_step_cmp<Q, T, kStreamCollide, kInGather, kOutOwn, DENSE_ROUND>);
    } else if (mode == kCollideOnly) {
        go(k_step_cmp<Q, T, kCollideOnly, kInGather, kOutOwn, DENSE_ROUND>);
    } else {
        go(k_step_cmp<Q, T, kStreamOnly, kInGather, kOutDense, DENSE_ROUND>);
    }
}

template <int Q, typename T>
void launch_step(const BCmpArgs& a, int mode, const void* src, void* dst, int lin, int lout, const Bc& tmpl,
                 const double* tau, cudaStream_t s)
{
    if constexpr (Q == 9 && std::is_same<T, float>::value) {
        if (a.dense_round && mode != kStreamOnly) {
            launch_step_as<Q, T, true>(a, mode, src, dst, lin, lout, tmpl, tau, s);
            return;
        }
    }
    launch_step_as<Q, T, false>(a, mode, src, dst, lin, lout, tmpl, tau, s);
}

template <int Q, typename T, int IN, int OUT, bool DENSE_ROUND>
void launch_adjoint_as(const BCmpArgs& a, int t0, const T* gp, const T* li, T* lo, const Bc& tmpl, const double* tau,
                       double* grad_acc, double* partial, cudaStream_t s)
{
    const unsigned threads = cmp_threads(Q, (int)sizeof(T), a.c.nf);
    const CmpOrder ord = cmp_order(a, threads, tmpl.t_level);
    auto go = [&](auto kernel) {
        launch_k(a.pdl, kernel, dim3(ord.n), dim3(threads), 0, s, gp, li, lo, a.c, a.lat, a.insts, a.blks, tmpl,
                 tau, grad_acc, partial, ord);
    };
    if constexpr (kPipe<Q, T> && IN == kInGather && OUT == kOutOwn) {
        if (!t0 && pipe_step(a)) {
            constexpr int MINB = 4;
            const PipeArgs<T> A{gp, li, lo, a.c, a.lat, a.insts, a.blks_by_class, tmpl, tau, grad_acc, partial,
                                pipe_order(a, tmpl.t_level)};
            if (a.blks) launch_pipe(a.pdl, k_adjoint_cmp_pipe<Q, T, true, DENSE_ROUND, MINB>, A, s);
            else launch_pipe(a.pdl, k_adjoint_cmp_pipe<Q, T, false, DENSE_ROUND, MINB>, A, s);
            return;
        }
    }
    if (t0) go(k_adjoint_cmp<Q, T, true, IN, OUT, DENSE_ROUND>);
    else go(k_adjoint_cmp<Q, T, false, IN, OUT, DENSE_ROUND>);
}

// lin: the layout of g^{t-1} and lambda^{t+1} (the same in every sweep);
// lout: the layout of lambda^t.
template <int Q, typename T>
void launch_adjoint(const BCmpArgs& a, int t0, const void* gprev, const void* lam_in, void* lam_out, int lin,
                    int lout, const Bc& tmpl, const double* tau, double* grad_acc, double* partial, cudaStream_t s)
{
    const T* gp = static_cast<const T*>(gprev);
    const T* li = static_cast<const T*>(lam_in);
    T* lo = static_cast<T*>(lam_out);
    auto as = [&](auto round) {
        constexpr bool DR = decltype(round)::value;
        if (lin == kLayoutSwapped)
            launch_adjoint_as<Q, T, kInLocal, kOutOwn, DR>(a, t0, gp, li, lo, tmpl, tau, grad_acc, partial, s);
        else if (lout == kLayoutSwapped)
            launch_adjoint_as<Q, T, kInGather, kOutScatter, DR>(a, t0, gp, li, lo, tmpl, tau, grad_acc, partial, s);
        else
            launch_adjoint_as<Q, T, kInGather, kOutOwn, DR>(a, t0, gp, li, lo, tmpl, tau, grad_acc, partial, s);
    };
    if constexpr (Q == 9 && std::is_same<T, float>::value) {
        if (a.dense_round) {
            as(std::true_type{});
            return;
        }
    }
    as(std::false_type{});
}

lbm_status step_any(const BCmpArgs& a, int mode, const void* src, void* dst, const Bc& tmpl, const double* tau,
                    cudaStream_t s, int lin = kLayoutNatural, int lout = kLayoutNatural)
{
    if (a.n_blocks == 0) return LBM_OK;
    if (a.q == 9 && a.prec == 4) launch_step<9, float>(a, mode, src, dst, lin, lout, tmpl, tau, s);
    else if (a.q == 9 && a.prec == 8) launch_step<9, double>(a, mode, src, dst, lin, lout, tmpl, tau, s);
    else if (a.q == 19 && a.prec == 4) launch_step<19, float>(a, mode, src, dst, lin, lout, tmpl, tau, s);
    else if (a.q == 19 && a.prec == 8) launch_step<19, double>(a, mode, src, dst, lin, lout, tmpl, tau, s);
    else return LBM_ERR_UNSUPPORTED;
    return cuda_status(cudaGetLastError());
}

lbm_status adjoint_any(const BCmpArgs& a, int t0, const void* gprev, const void* lam_in, void* lam_out,
                       const Bc& tmpl, const double* tau, double* grad_acc, double* partial, cudaStream_t s,
                       int lin = kLayoutNatural, int lout = kLayoutNatural)
{
    if (a.n_blocks == 0) return LBM_OK;
    if (a.q == 9 && a.prec == 4)
        launch_adjoint<9, float>(a, t0, gprev, lam_in, lam_out, lin, lout, tmpl, tau, grad_acc, partial, s);
    else if (a.q == 9 && a.prec == 8)
        launch_adjoint<9, double>(a, t0, gprev, lam_in, lam_out, lin, lout, tmpl, tau, grad_acc, partial, s);
    else if (a.q == 19 && a.prec == 4)
        launch_adjoint<19, float>(a, t0, gprev, lam_in, lam_out, lin, lout, tmpl, tau, grad_acc, partial, s);
    else if (a.q == 19 && a.prec == 8)
        launch_adjoint<19, double>(a, t0, gprev, lam_in, lam_out, lin, lout, tmpl, tau, grad_acc, partial, s);
    else return LBM_ERR_UNSUPPORTED;
    return cuda_status(cudaGetLastError());
}

template <int Q, typename T>
void launch_gather(const BCmpArgs& a, const void* dense, void* compact, bool add, bool swap, cudaStream_t s)
{
    const dim3 grid(a.n_blocks), block(kCmpThreads);
    const T* d = static_cast<const T*>(dense);
    T* c = static_cast<T*>(compact);
    if (add && swap) k_cmp_gather<Q, T, true, true><<<grid, block, 0, s>>>(d, c, a.c, a.insts, a.blks);
    else if (add) k_cmp_gather<Q, T, true, false><<<grid, block, 0, s>>>(d, c, a.c, a.insts, a.blks);
    else if (swap) k_cmp_gather<Q, T, false, true><<<grid, block, 0, s>>>(d, c, a.c, a.insts, a.blks);
    else k_cmp_gather<Q, T, false, false><<<grid, block, 0, s>>>(d, c, a.c, a.insts, a.blks);
}

lbm_status gather_any(const BCmpArgs& a, const void* dense, void* compact, cudaStream_t s, bool add = false,
                      int layout = kLayoutNatural)
{
    if (a.n_blocks == 0) return LBM_OK;
    const bool swap = layout == kLayoutSwapped;
    if (a.q == 9 && a.prec == 4) launch_gather<9, float>(a, dense, compact, add, swap, s);
    else if (a.q == 9) launch_gather<9, double>(a, dense, compact, add, swap, s);
    else if (a.prec == 4) launch_gather<19, float>(a, dense, compact, add, swap, s);
    else launch_gather<19, double>(a, dense, compact, add, swap, s);
    return cuda_status(cudaGetLastError());
}

// The call's options on a batch: node-velocity Eq. 6 and BGK.
Bc batch_tmpl(const double* rho_in, double rho_out, uint32_t* status)
{
    Bc bc;
    bc.rho_in = rho_in;
    bc.profile = 0;
    bc.rho_out = rho_out;
    bc.status = status;
    return bc;
}

}  // namespace

size_t compact_table_bytes(const PlanInfo& p, long long nf) { return table_layout(p, nf).bytes; }

// 32-bit element offsets into a state, which the interior path uses
static bool windows_fit(int q, long long nf) { return (unsigned long long)q * (unsigned long long)nf < (1ull << 32); }

long long window_count(const PlanInfo& p)
{
    const long long n = windows_per_plane(p) * (p.d == 3 ? p.geo.nz + 2 : 1);
    return n < kMaxWindows ? n : 0;
}

lbm_status compact_build(const PlanInfo& p, long long nf, void* tables, Cmp* out, const int32_t** cmap_out,
                         const BCmpInst** inst_out, BCmpInst* inst_host, cudaStream_t s)
{
    const TableLayout t = table_layout(p, nf);
    unsigned char* base = static_cast<unsigned char*>(tables);
    BCmpInst* inst = reinterpret_cast<BCmpInst*>(base + t.inst);
    int32_t* idx = reinterpret_cast<int32_t*>(base + t.idx);
    int32_t* nbr = reinterpret_cast<int32_t*>(base + t.nbr);
    uint32_t* eq6 = reinterpret_cast<uint32_t*>(base + t.eq6);
    uint32_t* pos = reinterpret_cast<uint32_t*>(base + t.pos);
    uint2* win = reinterpret_cast<uint2*>(base + t.win);
    int2* edge = reinterpret_cast<int2*>(base + t.edge);
    int32_t* cmap = reinterpret_cast<int32_t*>(base + t.cmap);
    int* blk = reinterpret_cast<int*>(base + t.blk);
    long long* total = reinterpret_cast<long long*>(base + t.total_slot);
    const long long N = p.geo.N;
    const long long nblk = (N + kScanNodes - 1) / kScanNodes;
    // interior nodes, then the boundary columns (index kernels guard against counts above nf)
    const int nx = p.geo.nx;
    for (int cls = 0; cls < 2; ++cls) {
        k_cmp_count<<<(unsigned)nblk, 256, 0, s>>>(p.geo.link, N, nx, cls, blk);
        k_cmp_scan<<<1, 1024, 0, s>>>(blk, nblk, total + cls);
        k_cmp_index<<<(unsigned)nblk, 256, 0, s>>>(p.geo.link, N, nx, cls, total, blk, cmap, idx, nf);
    }
    long long got[2] = {-1, -1};
    if (cudaMemcpyAsync(got, total, sizeof(got), cudaMemcpyDeviceToHost, s) != cudaSuccess) return LBM_ERR_CUDA;
    if (cudaStreamSynchronize(s) != cudaSuccess) return LBM_ERR_CUDA;
    if (got[0] + got[1] != nf) return LBM_ERR_INVALID_ARG;
    out->nf = nf;
    out->idx = idx;
    out->nbr = nbr;
    out->eq6 = eq6;
    out->pos = pos;
    out->win = win;
    out->edge = edge;
    BCmpInst one = {};
    one.g = p.geo;
    one.k0 = 0;
    one.nf = nf;
    one.f_off = 0;
    one.in_off = 0;
    one.acc_off = 0;
    one.n_in = p.n_in;
    // without windows every node goes through the table, as the boundary columns do
    one.lat = CmpBlk{0, windows_per_row(p), (int)std::min<long long>(windows_per_plane(p), INT32_MAX), 0};
    if (nf > 0) {
        const unsigned g = cmp_grid(nf);
        if (p.q == 9) k_cmp_nbr<9><<<g, 256, 0, s>>>(p.geo.link, cmap, idx, nbr, nf, p.geo);
        else k_cmp_nbr<19><<<g, 256, 0, s>>>(p.geo.link, cmap, idx, nbr, nf, p.geo);
        if (p.q == 9) k_cmp_eq6_bits<9><<<g, 256, 0, s>>>(nbr, nf, eq6);
        else k_cmp_eq6_bits<19><<<g, 256, 0, s>>>(nbr, nf, eq6);
        k_cmp_fill<<<g, 256, 0, s>>>(pos, nf, kPosBnd);
        if (t.n_win > 0 && nx >= 4 && got[0] > 0 && windows_fit(p.q, nf)) {  // columns 1 and nx - 2 are two
            const int d3 = p.d == 3;
            k_cmp_windows<<<(unsigned)((t.n_win + 255) / 256), 256, 0, s>>>(cmap, p.geo, d3, one.lat.w_row, t.n_win, win,
                                                                            edge);
            k_cmp_positions<<<g, 256, 0, s>>>(idx, p.geo, d3, one.lat.w_row, got[0], nf, pos);
            unsigned long long* bad = reinterpret_cast<unsigned long long*>(total + 2);
            unsigned long long off = 1;
            if (cudaMemsetAsync(bad, 0, sizeof(*bad), s) != cudaSuccess) return LBM_ERR_CUDA;
            if (p.q == 9) k_cmp_window_check<9><<<g, 256, 0, s>>>(*out, one.lat, got[0], bad);
            else k_cmp_window_check<19><<<g, 256, 0, s>>>(*out, one.lat, got[0], bad);
            if (cudaMemcpyAsync(&off, bad, sizeof(off), cudaMemcpyDeviceToHost, s) != cudaSuccess) return LBM_ERR_CUDA;
            if (cudaStreamSynchronize(s) != cudaSuccess) return LBM_ERR_CUDA;
            if (off == 0) one.n_int = (int)got[0];
            else k_cmp_fill<<<g, 256, 0, s>>>(pos, nf, kPosBnd);
        }
    }
    if (cudaGetLastError() != cudaSuccess) return LBM_ERR_CUDA;
    if (inst_host) *inst_host = one;
    if (inst_out) {
        if (cudaMemcpyAsync(inst, &one, sizeof(one), cudaMemcpyHostToDevice, s) != cudaSuccess) return LBM_ERR_CUDA;
        if (cudaStreamSynchronize(s) != cudaSuccess) return LBM_ERR_CUDA;  // ends the copy of `one`
    }
    *cmap_out = cmap;
    if (inst_out) *inst_out = inst;
    return LBM_OK;
}

lbm_status step_launch_cmp(const PlanInfo& p, int mode, const void* src, void* dst, const Bc& bc,
                           const double* tau, cudaStream_t s, int lin, int lout)
{
    if (p.cmp.nf == 0) return LBM_OK;
    return step_any(single_args(p, bc.status), mode, src, dst, bc, tau, s, lin, lout);
}

template <int Q, typename T>
static void launch_stream_dense(const PlanInfo& p, const void* src, void* dst, const Bc& bc, cudaStream_t s, int lin)
{
    const dim3 grid((unsigned)((p.geo.N + kCmpThreads - 1) / kCmpThreads)), block(kCmpThreads);
    auto go = [&](auto kernel) {
        launch_k(p.pdl, kernel, grid, block, 0, s, static_cast<const T*>(src), static_cast<T*>(dst), p.cmp, p.cmp_lat,
                 p.cmp_inst, p.cmp_map, p.geo.N, bc);
    };
    if (lin == kLayoutSwapped) go(k_stream_dense<Q, T, kInLocal>);
    else go(k_stream_dense<Q, T, kInGather>);
}

lbm_status stream_dense_launch(const PlanInfo& p, const void* src, void* dst, const Bc& bc, cudaStream_t s, int lin)
{
    if (p.q == 9 && p.prec == 4) launch_stream_dense<9, float>(p, src, dst, bc, s, lin);
    else if (p.q == 9) launch_stream_dense<9, double>(p, src, dst, bc, s, lin);
    else if (p.prec == 4) launch_stream_dense<19, float>(p, src, dst, bc, s, lin);
    else launch_stream_dense<19, double>(p, src, dst, bc, s, lin);
    return cuda_status(cudaGetLastError());
}

lbm_status adjoint_launch_cmp(const PlanInfo& p, int t0, const void* gprev, const void* lam_in, void* lam_out,
                              const Bc& bc, const double* tau, double* grad_acc, double* partial, cudaStream_t s,
                              int lin, int lout)
{
    if (p.cmp.nf == 0) return LBM_OK;
    LBM_CMP_TRY(adjoint_any(single_args(p, bc.status), t0, gprev, lam_in, lam_out, bc, tau, grad_acc, partial, s,
                            lin, lout));
    if (bc.uw_extrap && !t0) {  // at t = 0 the fluid is at rest and the pass adds nothing
        // (two-buffer pull only: the in-place schedule refuses the extrapolated velocity)
        const long long rows = (long long)p.geo.ny * p.geo.nz;
        const dim3 grid((unsigned)((rows + kCmpThreads - 1) / kCmpThreads)), block(kCmpThreads);
        if (p.q == 9 && p.prec == 4)
            launch_k(p.pdl, k_adjoint_uw_cmp<9, float>, grid, block, 0, s, static_cast<const float*>(gprev),
                     static_cast<const float*>(lam_in), static_cast<float*>(lam_out), p.cmp, p.cmp_map, p.geo, bc,
                     grad_acc);
        else if (p.q == 9)
            launch_k(p.pdl, k_adjoint_uw_cmp<9, double>, grid, block, 0, s, static_cast<const double*>(gprev),
                     static_cast<const double*>(lam_in), static_cast<double*>(lam_out), p.cmp, p.cmp_map, p.geo, bc,
                     grad_acc);
        else if (p.prec == 4)
            launch_k(p.pdl, k_adjoint_uw_cmp<19, float>, grid, block, 0, s, static_cast<const float*>(gprev),
                     static_cast<const float*>(lam_in), static_cast<float*>(lam_out), p.cmp, p.cmp_map, p.geo, bc,
                     grad_acc);
        else
            launch_k(p.pdl, k_adjoint_uw_cmp<19, double>, grid, block, 0, s, static_cast<const double*>(gprev),
                     static_cast<const double*>(lam_in), static_cast<double*>(lam_out), p.cmp, p.cmp_map, p.geo, bc,
                     grad_acc);
    }
    return cuda_status(cudaGetLastError());
}

lbm_status compact_gather_launch(const PlanInfo& p, const void* dense, void* compact, cudaStream_t s, int layout)
{
    if (p.cmp.nf == 0) return LBM_OK;
    return gather_any(single_args(p, nullptr), dense, compact, s, false, layout);
}

lbm_status compact_gather_add_launch(const PlanInfo& p, const void* dense, void* compact, cudaStream_t s, int layout)
{
    if (p.cmp.nf == 0) return LBM_OK;
    return gather_any(single_args(p, nullptr), dense, compact, s, true, layout);
}

lbm_status bstep_launch_cmp(const BCmpArgs& a, int mode, const void* src, void* dst, const double* rho_in,
                            const double* tau, double rho_out, cudaStream_t s)
{
    return step_any(a, mode, src, dst, batch_tmpl(rho_in, rho_out, a.status), tau, s);
}

lbm_status badjoint_launch_cmp(const BCmpArgs& a, int t0, const void* gprev, const void* lam_in, void* lam_out,
                               const double* rho_in, const double* tau, double rho_out, double* grad_acc,
                               double* partial, cudaStream_t s)
{
    return adjoint_any(a, t0, gprev, lam_in, lam_out, batch_tmpl(rho_in, rho_out, a.status), tau, grad_acc, partial,
                       s);
}

lbm_status bgather_launch_cmp(const BCmpArgs& a, const void* dense, void* compact, cudaStream_t s)
{
    return gather_any(a, dense, compact, s);
}

lbm_status eq6_bits_launch_cmp(int q, const int32_t* nbr, long long nf, uint32_t* bits, cudaStream_t s)
{
    if (nf == 0) return LBM_OK;
    if (q == 9) k_cmp_eq6_bits<9><<<cmp_grid(nf), 256, 0, s>>>(nbr, nf, bits);
    else k_cmp_eq6_bits<19><<<cmp_grid(nf), 256, 0, s>>>(nbr, nf, bits);
    return cuda_status(cudaGetLastError());
}

lbm_status bpack_launch_cmp(const Cmp& local, int q, long long k0, long long nfp, long long n_win, long long w0,
                            bool windows, const Cmp& packed, cudaStream_t s)
{
    if (n_win > 0)  // (the packed positions start as padding: bpack_start_cmp)
        k_bpack_windows<<<(unsigned)((n_win + 255) / 256), 256, 0, s>>>(
            local, n_win, (int)k0, const_cast<uint2*>(packed.win) + w0, const_cast<int2*>(packed.edge) + w0);
    if (local.nf > 0)
        k_bpack_cmp<<<(unsigned)((local.nf + 255) / 256), 256, 0, s>>>(
            local, q, k0, nfp, (unsigned)w0, const_cast<int32_t*>(packed.idx), const_cast<int32_t*>(packed.nbr),
            const_cast<uint32_t*>(packed.pos), windows);
    return cuda_status(cudaGetLastError());
}

lbm_status bpack_start_cmp(int q, long long nfp, const Cmp& packed, cudaStream_t s)
{
    // padding nodes: bounce-back in every direction, and skipped by every kernel
    static_assert(kCmpBB == -1, "padding codes are written as all-ones bytes");
    if (nfp == 0) return LBM_OK;
    if (cudaMemsetAsync(const_cast<int32_t*>(packed.nbr), 0xFF, sizeof(int32_t) * (size_t)(q - 1) * (size_t)nfp, s) !=
        cudaSuccess)
        return LBM_ERR_CUDA;
    k_cmp_fill<<<(unsigned)((nfp + 255) / 256), 256, 0, s>>>(const_cast<uint32_t*>(packed.pos), nfp, kPosDead);
    return cuda_status(cudaGetLastError());
}

bool windows_packable(int q, long long n_win, long long nfp) { return n_win < kMaxWindows && windows_fit(q, nfp); }

}  // namespace lbm
