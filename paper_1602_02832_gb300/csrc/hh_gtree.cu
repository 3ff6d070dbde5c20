// Tree-loop step 1 on the device (Section 2): Morton octree, Barnes groups
// and interaction lists built from the synchronised particle state without
// leaving the GPU, then the particles reordered into Morton order and the
// node records written behind them.  The rules are those of the host builder
// (include/hh.h, hh_tree_build): root cube from the bounding box, 21-bit
// Morton keys, cells split while they hold more than `leaf` particles,
// pre-order cell numbering, groups = maximal cells with <= n_crit particles,
// the same opening walk.  Node moments are summed from the leaves up (the host sums in
// index order), so a node's centre of mass may differ in the last bits.
//
// CUB (shipped with the CUDA toolkit) provides the radix sort of the keys and
// the prefix sums; every other step is a kernel of this file.

#include <algorithm>
#include <cstring>
#include <functional>
#include <vector>

#include <cub/device/device_radix_sort.cuh>
#include <cub/device/device_scan.cuh>

#include "hh_ctx.h"

using namespace hh;

namespace {

constexpr int kBits = 21;
constexpr int kMaxDepth = 21;
constexpr int kWalkThreads = 128;  // threads of a walk block
constexpr int kWalkStage = 512;    // cells that it stages
constexpr int kPath = 24;  // entries of a chunk's path (at most kMaxDepth ancestors)

// ------------------------------------------------------------ small helpers
__device__ __forceinline__ unsigned long long order_bits(double v)  // monotone map double -> u64
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    return (b >> 63) ? ~b : (b | 0x8000000000000000ull);
}
__device__ __forceinline__ double from_order_bits(unsigned long long o)
{
    const unsigned long long b = (o >> 63) ? (o & 0x7fffffffffffffffull) : ~o;
    return __longlong_as_double((long long)b);
}

__device__ __forceinline__ uint64_t spread_bits(uint32_t v)
{
    uint64_t x = v & 0x1fffffu;
    x = (x | (x << 32)) & 0x001f00000000ffffull;
    x = (x | (x << 16)) & 0x001f0000ff0000ffull;
    x = (x | (x << 8)) & 0x100f00f00f00f00full;
    x = (x | (x << 4)) & 0x10c30c30c30c30c3ull;
    x = (x | (x << 2)) & 0x1249249249249249ull;
    return x;
}

// Peano-Hilbert key of a cell of the 2^21 grid (Skilling 2004): the low bit
// fields are mapped level by level into each sub-cube's frame, Gray-coded,
// and the resulting transposed index is interleaved like a Morton key.
__device__ __forceinline__ uint64_t hilbert_key(uint32_t a0, uint32_t a1, uint32_t a2)
{
    uint32_t c[3] = {a0, a1, a2};
#pragma unroll 1
    for (uint32_t q = 1u << (kBits - 1); q > 1u; q >>= 1) {
        const uint32_t p = q - 1u;
#pragma unroll
        for (int i = 0; i < 3; i++) {
            const uint32_t t = (c[0] ^ c[i]) & p;
            if (c[i] & q) {
                c[0] ^= p;
            } else {
                c[0] ^= t;
                c[i] ^= t;
            }
        }
    }
    c[1] ^= c[0];
    c[2] ^= c[1];
    uint32_t flip = 0;
    for (uint32_t q = 1u << (kBits - 1); q > 1u; q >>= 1)
        if (c[2] & q) flip ^= q - 1u;
    return (spread_bits(c[0] ^ flip) << 2) | (spread_bits(c[1] ^ flip) << 1) | spread_bits(c[2] ^ flip);
}

struct Box {
    unsigned long long lo[3], hi[3];  // order bits
    int32_t bad;                      // a particle not at the tree time
};

// Sizes the build keeps on the device, so that no step waits for the host.
struct GCounts {
    int32_t ncells, overflow, bad, G;
    int64_t L, n_tiles, total_parts;
    unsigned long long lmax;  // longest list
};

// Cell table in pre-order (a cell's subtree is the `size` cells from it on).
struct PCells {
    int32_t *begin, *end, *depth, *parent, *size;
    int32_t *arrived;  // particles below whose moments are summed
    int4 *child;       // [2 * n] children in order, -1 behind the last
    int4 *pack;        // {begin, end, FP32 bits of the reject bound, size}: what the list walk reads per cell
    float4 *cf;        // {centre of mass x, y, z in the tree's unit, accept bound}
};

enum : int { kOpen = 0, kEmitParticles = 1, kEmitNode = 2 };

// cells | groups in one word: cells below bit 34 (at most 22 per particle),
// groups above
constexpr int kCellBits = 34;

// Everything a rebuild kernel reads or writes for one simulation.  A kernel
// runs for one simulation (the record passed by value) or for many (an array
// in device memory, simulation = blockIdx.y): the same code either way.
// Scans are read relative to their first entry, so a simulation's slice of
// one scan over many simulations' arrays reads like its own scan.
struct RbSim {
    State st, alt;            // particle state and the buffer it is reordered into
    PCells P;
    GCounts *gc;
    Box *box;
    double *root_side;
    double *unit;             // power of two that brings every |coordinate| below 1
    uint64_t *key, *key2;     // particle keys, and sorted
    int32_t *idx, *perm;      // particle indices, and in key order
    int64_t *cnt, *pos;       // [n + 1] cells and groups that begin at a particle, and their exclusive scan
    int32_t *chain;           // [n] depths of the cells that begin at a particle (see k_chains)
    double *mom;              // [ncells][16] cell sums
    int32_t *g_cell;
    double *box_lo, *box_hi;  // [3][G] group boxes
    float4 *box_f;
    int64_t *ids, *ids2;
    int32_t *group_of;
    int64_t *off;             // [G + 1] list offsets
    int32_t *lidx;            // list entries
    int4 *tiles;
    int64_t *nt2, *tscan2;    // [tile counts | part counts], G + 1 each, and their scan
    int64_t *pair2, *pscan2;  // [particle | node entries per (group, chunk)], pairs + 1 each, and their scan
    int32_t *path;            // [R][kPath] ancestors of each chunk's first cell, from the root (right-aligned)
    DevScalars *ds;           // the context's device sizes (set by k_finish)
    double t, theta;
    int64_t n, pairs;
    int64_t cap_list, cap_tiles;  // entries and tiles that fit
    int32_t cap_g, cap_cells, leaf, n_crit, order, tile_i, part_len, work_item, work_split;
    int32_t seg;                 // where its particles begin among a batch's
    int32_t ncells, G;           // set by the host as they become known
    int32_t chunk, R;            // cells of a walk chunk, and chunks
};

#define RB_ARGS const RbSim one, const RbSim *many

// For many simulations a block first copies its record into shared memory:
// read from there (as from the constant bank for one), the record's fields
// can be fetched again where they are used instead of occupying registers.
template <bool kMany>
__device__ __forceinline__ const RbSim &rb_sim_of(const RbSim &one, const RbSim *many, unsigned char *sh)
{
    if (!kMany) return one;
    const uint32_t *src = reinterpret_cast<const uint32_t *>(many + blockIdx.y);
    uint32_t *dst = reinterpret_cast<uint32_t *>(sh);
    for (int i = threadIdx.x; i < int(sizeof(RbSim) / 4); i += blockDim.x) dst[i] = src[i];
    __syncthreads();
    return *reinterpret_cast<const RbSim *>(sh);
}
#define RB_SIM                                                      \
    after_previous();                                               \
    RB_RECORD
// (in front of a CUB call: its kernels are placed when this one has ended, as
// they expect of a kernel that knows nothing of dependent launches)
#define RB_SIM_BEFORE_CUB                                           \
    wait_previous();                                                \
    RB_RECORD
#define RB_RECORD                                                   \
    __shared__ __align__(16) unsigned char rb_rec_[sizeof(RbSim)]; \
    const RbSim &a = rb_sim_of<kMany>(one, many, rb_rec_)

// side of cell c: the root's, halved at each level
__device__ __forceinline__ double cell_side(const RbSim &a, int32_t c)
{
    return *a.root_side * __longlong_as_double((long long)(1023 - a.P.depth[c]) << 52);
}

template <bool kMany>
__global__ void k_box(RB_ARGS)
{
    RB_SIM;
    const State &s = a.st;
    const double t_tree = a.t;
    unsigned long long lo[3] = {~0ull, ~0ull, ~0ull}, hi[3] = {0ull, 0ull, 0ull};
    bool bad = false;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < a.n; i += (int64_t)gridDim.x * blockDim.x) {
        for (int d = 0; d < 3; d++) {
            const unsigned long long o = order_bits(s.x[d * s.cap_j + i]);
            lo[d] = o < lo[d] ? o : lo[d];
            hi[d] = o > hi[d] ? o : hi[d];
        }
        bad |= s.t[i] != t_tree;
    }
    // warp, then block reduction (blockDim.x = 256): one atomic per block and
    // bound, and none from a block that saw no particle
    __shared__ unsigned long long s_lo[8][3], s_hi[8][3];
    __shared__ int s_bad[8];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (int d = 0; d < 3; d++) {
        for (int off = 16; off > 0; off >>= 1) {
            const unsigned long long l2 = __shfl_xor_sync(0xffffffffu, lo[d], off);
            const unsigned long long h2 = __shfl_xor_sync(0xffffffffu, hi[d], off);
            lo[d] = l2 < lo[d] ? l2 : lo[d];
            hi[d] = h2 > hi[d] ? h2 : hi[d];
        }
        if (lane == 0) {
            s_lo[w][d] = lo[d];
            s_hi[w][d] = hi[d];
        }
    }
    const bool any_bad = __any_sync(0xffffffffu, bad);
    if (lane == 0) s_bad[w] = any_bad;
    __syncthreads();
    if (threadIdx.x == 0) {
        int b = 0;
        for (int k = 0; k < int(blockDim.x >> 5); k++) {
            b |= s_bad[k];
            for (int d = 0; d < 3; d++) {
                lo[d] = s_lo[k][d] < lo[d] ? s_lo[k][d] : lo[d];
                hi[d] = s_hi[k][d] > hi[d] ? s_hi[k][d] : hi[d];
            }
        }
        if (lo[0] <= hi[0])
            for (int d = 0; d < 3; d++) {
                atomicMin(&a.box->lo[d], lo[d]);
                atomicMax(&a.box->hi[d], hi[d]);
            }
        if (b) atomicExch(&a.box->bad, 1);
    }
}

template <bool kMany>
__global__ void k_keys(RB_ARGS)
{
    RB_SIM_BEFORE_CUB;
    const State &s = a.st;
    const Box *b = a.box;
    double lo[3], side = 0.0;
    for (int d = 0; d < 3; d++) {
        lo[d] = from_order_bits(b->lo[d]);
        const double ext = from_order_bits(b->hi[d]) - lo[d];
        if (ext > side) side = ext;
    }
    if (side == 0.0) side = 1.0;
    const double scale = double(1u << kBits) / side;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        *a.root_side = side;
        double xm = 0.0;  // bound on |coordinate| of every particle, node and group box
        for (int d = 0; d < 3; d++) xm = fmax(xm, fmax(fabs(lo[d]), fabs(from_order_bits(b->hi[d]))));
        int e = 0;
        if (xm > 0.0) frexp(xm, &e);
        *a.unit = ldexp(1.0, min(max(-e, -1000), 1000));
    }
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < a.n; i += (int64_t)gridDim.x * blockDim.x) {
        uint32_t u[3];
        for (int d = 0; d < 3; d++) {
            double f = floor((s.x[d * s.cap_j + i] - lo[d]) * scale);
            f = f < 0.0 ? 0.0 : f;
            f = f > double((1u << kBits) - 1u) ? double((1u << kBits) - 1u) : f;
            u[d] = uint32_t(f);
        }
        a.key[i] = a.order == HH_ORDER_HILBERT ? hilbert_key(u[0], u[1], u[2])
                                               : (spread_bits(u[0]) << 2) | (spread_bits(u[1]) << 1) | spread_bits(u[2]);
        a.idx[i] = a.seg + int32_t(i);
    }
}

// one thread per simulation
template <bool kMany>
__global__ void k_root_init(RB_ARGS)
{
    RB_SIM;
    Box *b = a.box;
    GCounts *gc = a.gc;
    for (int d = 0; d < 3; d++) {  // empty bounding box
        b->lo[d] = ~0ull;
        b->hi[d] = 0ull;
    }
    b->bad = 0;
    gc->ncells = gc->overflow = gc->bad = gc->G = 0;
    gc->lmax = 0ull;
}

// Leading octal digits that two keys share (0..21).
__device__ __forceinline__ int shared_digits(uint64_t a, uint64_t b)
{
    const uint64_t x = a ^ b;
    return x ? (__clzll((long long)x) - 1) / 3 : kMaxDepth;
}

// Whether the cell of depth d that holds sorted particles i - 1 and i has more
// than `most` particles: its first particle (or i - most, if it begins before
// that) by a binary search, then the particle `most` behind it.
__device__ __forceinline__ bool more_than(const uint64_t *key, int64_t n, int64_t i, uint64_t ki, int d, int64_t most)
{
    int64_t l = max(int64_t(0), i - most), h = i - 1;
    while (l < h) {
        const int64_t mid = (l + h) >> 1;
        if (shared_digits(key[mid], ki) >= d) h = mid;
        else l = mid + 1;
    }
    return l + most < n && shared_digits(key[l + most], ki) >= d;
}

// The cells, from the sorted keys alone.  A cell is a range of particles that
// share `depth` leading digits, and it exists when its parent holds more than
// `leaf` particles.  The cells that begin at sorted particle i are nested, so
// they are one run of depths: from one more than the digits that i shares with
// i - 1 (if the cell of that many digits, i's and i - 1's common one, is
// split) down to a leaf; the cell of depth d is split when particle i + leaf
// shares d digits too.  In pre-order the cells follow their first particle,
// then their depth: the scan of the runs' lengths gives every cell's number.
// A group (Barnes 1990: maximal cells with <= n_crit particles, or leaves)
// begins at i when the common cell of i - 1 and i has more than n_crit: it is
// the run's first cell without them.
// Splitting level by level (up to 22 launches, each with octant searches),
// sorting the cells into pre-order and selecting the groups from them took 215
// us for 262144 particles and 430 us for 32 clusters with 1k to 32k; this
// kernel, its scan and the two after it take 45 and 70 us.
// chain[i] = top | group depth << 8 | leaf depth << 16.
template <bool kMany>
__global__ void k_chains(RB_ARGS)
{
    RB_SIM_BEFORE_CUB;
    const uint64_t *key = a.key2;
    if (blockIdx.x == 0 && threadIdx.x == 0) a.cnt[a.n] = 0;  // terminal entry of the scan
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < a.n; i += (int64_t)gridDim.x * blockDim.x) {
        const uint64_t k = key[i];
        const int top = i > 0 ? shared_digits(key[i - 1], k) + 1 : 0;
        int64_t word = 0;
        if (top <= kMaxDepth) {
            const int low = i + a.leaf < a.n ? min(kMaxDepth, shared_digits(k, key[i + a.leaf]) + 1) : 0;
            if (i == 0 || low >= top || more_than(key, a.n, i, k, top - 1, a.leaf)) {
                const int leaf_d = max(low, top);
                const int big = i + a.n_crit < a.n ? shared_digits(k, key[i + a.n_crit]) + 1 : 0;
                const bool group = i == 0 || big >= top || more_than(key, a.n, i, k, top - 1, a.n_crit);
                const int group_d = min(leaf_d, max(big, top));
                word = (leaf_d - top + 1) | (int64_t(group) << kCellBits);
                a.chain[i] = top | (group_d << 8) | (leaf_d << 16);
            }
        }
        a.cnt[i] = word;
    }
}

// cells (low part) and groups (high part) before sorted particle i
__device__ __forceinline__ uint64_t before(const RbSim &a, int64_t i) { return uint64_t(a.pos[i]) - uint64_t(a.pos[0]); }
__device__ __forceinline__ int64_t cells_of(uint64_t w) { return int64_t(w & ((uint64_t(1) << kCellBits) - 1)); }

// First particle and depth of every cell, the group cells, and the sizes.  When
// the cells do not fit, none is written and both counts are zero, so that the
// kernels already queued behind this one (they run before the host reads the
// overflow and reports HH_ENOMEM) find nothing to read; group cells beyond cap_g
// are not stored, likewise.
template <bool kMany>
__global__ void k_begin_cells(RB_ARGS)
{
    RB_SIM;
    const uint64_t all = before(a, a.n);
    const int64_t ncells = cells_of(all);
    const bool overflow = ncells > a.cap_cells;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        a.gc->ncells = overflow ? 0 : int32_t(ncells);
        a.gc->overflow = overflow;
        a.gc->bad = a.box->bad;
        a.gc->G = overflow ? 0 : int32_t(all >> kCellBits);
    }
    if (overflow) return;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < a.n; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t word = a.cnt[i];
        if (word == 0) continue;
        const int32_t ch = a.chain[i], top = ch & 255;
        const uint64_t w = before(a, i);
        const int32_t p = int32_t(cells_of(w));
        for (int d = top; d <= (ch >> 16); d++) {
            a.P.begin[p + d - top] = int32_t(i);
            a.P.depth[p + d - top] = d;
        }
        if (word >> kCellBits) {
            const int32_t g = int32_t(w >> kCellBits);
            if (g < a.cap_g) a.g_cell[g] = p + ((ch >> 8) & 255) - top;
        }
    }
}

// Ends, subtree sizes, children and parents: eight lanes per cell, lane o
// finding where octant o of a split cell ends (the cell's own end is octant
// 7's) by a search that doubles its step from the cell's first particle.  A
// child that begins behind its parent's first particle is the first of the
// cells beginning there.
template <bool kMany>
__global__ void k_cells(RB_ARGS)
{
    RB_SIM;
    const uint64_t *key = a.key2;
    const int32_t n = int32_t(a.n), ncells = a.gc->ncells;
    const int lane = threadIdx.x & 31, o = lane & 7;
    const int64_t n_q = (int64_t)ncells * 8;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;  // a multiple of 32: warps stay whole
    for (int64_t q0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x - lane; q0 < n_q; q0 += stride) {
        const bool valid = q0 + lane < n_q;
        const int32_t p = int32_t((q0 + lane) >> 3);
        int32_t b = 0, d = 0, hi = 0;
        bool split = false;
        if (valid) {
            b = a.P.begin[p];
            d = a.P.depth[p];
            split = d < (a.chain[b] >> 16);
            // the first key behind octant o (a leaf: behind the cell)
            const int sh = 3 * (kBits - (split ? d + 1 : d));
            const uint64_t k = key[b];
            const uint64_t lim = (split ? ((((k >> sh) & ~uint64_t(7)) | uint64_t(o)) + 1) : ((k >> sh) + 1)) << sh;
            if (split || o == 7) {
                int32_t l = b, step = 8;
                while (n - l > step && key[l + step] < lim) {
                    l += step;
                    step *= 2;
                }
                int32_t h = n - l > step ? l + step : n;
                while (l < h) {
                    const int32_t mid = l + ((h - l) >> 1);
                    if (key[mid] < lim) l = mid + 1;
                    else h = mid;
                }
                hi = l;
            }
        }
        // children: the octants that are not empty; a lane's begins where the one before it ends
        const int prev = __shfl_up_sync(0xffffffffu, hi, 1);
        const int32_t from = o == 0 ? b : prev, end = __shfl_sync(0xffffffffu, hi, lane | 7);
        const bool has = valid && split && hi > from;
        const uint32_t oct = (__ballot_sync(0xffffffffu, has) >> (lane & 24)) & 0xffu;
        if (!valid) continue;
        int32_t *child = reinterpret_cast<int32_t *>(a.P.child) + 8 * int64_t(p);
        if (has) {
            const int32_t c = from == b ? p + 1 : int32_t(cells_of(before(a, from)));
            child[__popc(oct & ((1u << o) - 1u))] = c;
            a.P.parent[c] = p;
        }
        if (o >= __popc(oct)) child[o] = -1;
        if (o == 0) {
            a.P.end[p] = end;
            a.P.size[p] = int32_t(cells_of(before(a, end))) - p;
            a.P.arrived[p] = 0;
            if (p == 0) a.P.parent[0] = -1;
        }
    }
}

// State of the reordered particles: alt[k] = st[perm[k]] (Morton order).
template <bool kMany>
__global__ void k_permute(RB_ARGS)
{
    RB_SIM;
    const State &src = a.st;
    const State &dst = a.alt;
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < a.n; k += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = a.perm[k];
        for (int d = 0; d < 3; d++) {
            dst.x[d * dst.cap_j + k] = src.x[d * src.cap_j + i];
            dst.v[d * dst.cap_j + k] = src.v[d * src.cap_j + i];
            dst.a[d * dst.cap_j + k] = src.a[d * src.cap_j + i];
            dst.jk[d * dst.cap_j + k] = src.jk[d * src.cap_j + i];
        }
        dst.m[k] = src.m[i];
        dst.t[k] = src.t[i];
        dst.dt[k] = src.dt[i];
        a.ids2[k] = a.ids[i];
    }
}

// Mass and mass-weighted sums of x, v, a, jk of every cell's particles, in one
// pass from the leaves up.  Sixteen lanes take a leaf, lane w one of its 13
// sums (0: mass; 1 + 3k + dim: mass times x, v, a, jerk), which a single
// thread's order keeps: a leaf over its particles, a split cell over its
// children.  The lanes then add the cell's particles to its parent's arrivals;
// the last child to arrive has its lanes sum the parent and goes on, the others
// stop.  Nothing waits.  (A launch per level took 122 us for 262144 particles
// and 170 us for 32 clusters with 1k to 32k, here 94 and 106 us: FP64 sums and,
// at the top, a round trip to L2 per level.)
template <bool kMany>
__global__ void __launch_bounds__(256) k_moments(RB_ARGS)
{
    RB_SIM;
    const State &s = a.alt;  // (the reordered particles)
    const int32_t ncells = a.gc->ncells;
    const int w = threadIdx.x & 15, half = (threadIdx.x >> 4) & 1;
    const uint32_t mask = 0xffffu << (16 * half);
    const int32_t stride = int32_t(gridDim.x * blockDim.x) >> 4;
    const int field = w == 0 ? 0 : (w - 1) / 3, dim = w == 0 ? 0 : (w - 1) % 3;
    double *const f = (field == 0 ? s.x : field == 1 ? s.v : field == 2 ? s.a : s.jk) + int64_t(dim) * s.cap_j;
    for (int32_t leaf = int32_t(blockIdx.x * blockDim.x + threadIdx.x) >> 4; leaf < ncells; leaf += stride) {
        if (a.P.size[leaf] != 1) continue;
        double acc = 0.0;
        int32_t c = leaf, b = a.P.begin[leaf], e = a.P.end[leaf];
        if (w < 13)
            for (int32_t p = b; p < e; p++) {
                const double mi = s.m[p];
                acc = w == 0 ? acc + mi : fma(mi, f[p], acc);
            }
        while (true) {
            a.mom[int64_t(c) * 16 + w] = acc;
            const int32_t par = a.P.parent[c];
            bool last = false;
            __syncwarp(mask);
            if (w == 0 && par >= 0)
                last = int32_t(atom_add_acq_rel_gpu(reinterpret_cast<unsigned int *>(&a.P.arrived[par]),
                                                    (unsigned int)(e - b))) + (e - b) == a.P.end[par] - a.P.begin[par];
            if (!__shfl_sync(mask, int(last), 0, 16)) break;
            __syncwarp(mask);
            // the parent's sums
            c = par;
            b = a.P.begin[c];
            e = a.P.end[c];
            const int4 k0 = a.P.child[2 * int64_t(c)], k1 = a.P.child[2 * int64_t(c) + 1];
            const int32_t kid[8] = {k0.x, k0.y, k0.z, k0.w, k1.x, k1.y, k1.z, k1.w};
            double part[8];
#pragma unroll
            for (int k = 0; k < 8; k++) part[k] = kid[k] >= 0 ? __ldcg(&a.mom[int64_t(kid[k]) * 16 + w]) : 0.0;
            acc = 0.0;
#pragma unroll
            for (int k = 0; k < 8; k++)
                if (kid[k] >= 0) acc += part[k];
        }
    }
}

// Node records (pseudo-particles), j entry n + (pre-order number) of every
// cell: centre of mass and mass-weighted mean velocity, acceleration and jerk
// at the tree time.  And what the list walk reads of the cell: its centre in
// FP32 and the bounds on the squared distance (see decide).  A thread per cell
// (the divisions bound this kernel; sixteen lanes per cell, as the sums have
// them, leave a quarter of the lanes idle: 79 against 47 us for 112233 cells).
template <bool kMany>
__global__ void __launch_bounds__(128) k_node_records(RB_ARGS)
{
    RB_SIM;
    const State &s = a.alt;
    const int32_t ncells = a.gc->ncells;
    const double u = *a.unit;
    const float theta = float(a.theta), inv_theta = 1.0f / theta, root = float(*a.root_side * u);
    for (int32_t c = blockIdx.x * blockDim.x + threadIdx.x; c < ncells; c += gridDim.x * blockDim.x) {
        const double2 *mom = reinterpret_cast<const double2 *>(a.mom + int64_t(c) * 16);
        double sum[14];
#pragma unroll
        for (int k = 0; k < 7; k++) {
            const double2 v = mom[k];
            sum[2 * k] = v.x;
            sum[2 * k + 1] = v.y;
        }
        const double M = sum[0];
        const int64_t j = a.n + c;
        float xf[3];
#pragma unroll
        for (int d = 0; d < 3; d++) {
            const int64_t q = d * s.cap_j + j;
            const double x = sum[1 + d] / M;
            xf[d] = float(x * u);
            s.x[q] = x;
            s.v[q] = sum[4 + d] / M;
            s.a[q] = sum[7 + d] / M;
            s.jk[q] = sum[10 + d] / M;
        }
        s.m[j] = M;
        s.t[j] = a.t;
        const int32_t b = a.P.begin[c], e = a.P.end[c];
        const float side = root * __int_as_float((127 - a.P.depth[c]) << 23);
        const float far = (side * (1.0f + 0x1p-16f) + 0x1p-18f * theta) * inv_theta;
        const float near = (side * (1.0f - 0x1p-16f) - 0x1p-18f * theta) * inv_theta;
        float hi = far * far * (1.0f + 0x1p-17f), lo = near > 0.0f ? near * near * (1.0f - 0x1p-17f) : -1.0f;
        if (e - b == 1) hi = lo = __int_as_float(0x7f800000);  // a single particle always goes in as such
        a.P.cf[c] = make_float4(xf[0], xf[1], xf[2], hi);
        a.P.pack[c] = make_int4(b, e, __float_as_int(lo), a.P.size[c]);
    }
}

// Bounding box of each group's particles ([3][G] lo and hi) and the particles'
// group numbers, one warp per group (17k groups of 262144 particles: 16 us; with
// FP64 comparisons and one lane's conversions 52 us)
// (none beyond cap_g groups: the host then reports the overflow).
template <bool kMany>
__global__ void k_group_box(RB_ARGS)
{
    RB_SIM;
    const State &s = a.alt;
    const int32_t G = a.gc->G;
    if (G > a.cap_g) return;
    const int lane = threadIdx.x & 31;
    const int64_t w0 = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5, nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const double u = *a.unit;
    for (int64_t g = w0; g < G; g += nw) {
        const int32_t c = a.g_cell[g], b = a.P.begin[c], e = a.P.end[c];
        // (as ordered integers: an FP64 comparison takes the pipe 64 cycles)
        unsigned long long lo[3], hi[3];
        for (int32_t p = b + lane; p < e; p += 32) a.group_of[p] = int32_t(g);
#pragma unroll
        for (int d = 0; d < 3; d++) {
            lo[d] = hi[d] = order_bits(s.x[d * s.cap_j + min(b + lane, e - 1)]);
            for (int32_t p = b + lane + 32; p < e; p += 32) {
                const unsigned long long o = order_bits(s.x[d * s.cap_j + p]);
                lo[d] = o < lo[d] ? o : lo[d];
                hi[d] = o > hi[d] ? o : hi[d];
            }
        }
        for (int off = 16; off > 0; off >>= 1)
#pragma unroll
            for (int d = 0; d < 3; d++) {
                const unsigned long long l2 = __shfl_xor_sync(0xffffffffu, lo[d], off);
                const unsigned long long h2 = __shfl_xor_sync(0xffffffffu, hi[d], off);
                lo[d] = l2 < lo[d] ? l2 : lo[d];
                hi[d] = h2 > hi[d] ? h2 : hi[d];
            }
        if (lane < 8) {  // lanes 0..2: the lower bounds, 4..6: the upper ones
            const int d = lane & 3;
            const bool upper = lane >= 4;
            const unsigned long long o = d == 0 ? (upper ? hi[0] : lo[0]) : d == 1 ? (upper ? hi[1] : lo[1])
                                                                                  : (upper ? hi[2] : lo[2]);
            const double v = from_order_bits(o);
            if (d < 3) (upper ? a.box_hi : a.box_lo)[d * int64_t(G) + g] = v;
            reinterpret_cast<float *>(a.box_f)[8 * g + lane] = d < 3 ? float(v * u) : 0.f;
        }
    }
}

// The opening decision of cell c for group g (rules of hh_tree_build): the
// group's own cell and single particles go in as particles; a cell that does
// not contain the group goes in as a node when side < theta * (distance of its
// centre of mass to the group's box), else as particles when it is a leaf;
// everything else is opened.
//
// The distance test is screened in FP32 (FP64 throughput is low on this part),
// with two bounds on the squared distance that each cell carries (node
// records), in the tree's unit: the power of two that brings every
// |coordinate| below 1, so that no square leaves FP32's range.  Rounding centre
// and box to FP32 and taking gaps, squares and sum in FP32 moves the distance
// by less than 2^-21 + 2^-22 distance.  A cell is accepted above
// ((1 + 2^-16) side + 2^-18 theta)^2 / theta^2 (and 2^-17 more) and not accepted
// below ((1 - 2^-16) side - 2^-18 theta)^2 / theta^2 (and 2^-17 less; never when
// that difference is negative), both evaluated in FP32 to 2^-20, which covers
// those errors and the roundings of the FP64 test.  Between the bounds (and for
// any NaN) the test is redone in FP64 with the roundings of the sequential
// builder (no contraction), so the decision is always the FP64 one.  A single
// particle carries infinite bounds: it is a leaf and goes in as a particle.
// (With the two bounds instead of a square root and a tolerance per decision,
// the walk's counts of 262144 particles take 339 us, 427 before.)
struct GroupView {
    int32_t g, gc, gb, ge;
    float3 lof, hif;
};

struct CellRec {
    int4 pk;
    float4 cf;
};

__device__ __forceinline__ CellRec load_cell(const RbSim &a, int32_t c)
{
    return {__ldg(&a.P.pack[c]), __ldg(&a.P.cf[c])};
}

__device__ __forceinline__ int decide(const RbSim &a, const GroupView &G, int32_t c, const CellRec &r)
{
    if (r.pk.x <= G.gb && G.ge <= r.pk.y) return c == G.gc ? kEmitParticles : kOpen;
    const float gx = fmaxf(fmaxf(G.lof.x - r.cf.x, r.cf.x - G.hif.x), 0.f);
    const float gy = fmaxf(fmaxf(G.lof.y - r.cf.y, r.cf.y - G.hif.y), 0.f);
    const float gz = fmaxf(fmaxf(G.lof.z - r.cf.z, r.cf.z - G.hif.z), 0.f);
    const float d2f = gx * gx + gy * gy + gz * gz;
    bool accept = d2f > r.cf.w;
    if (!accept && !(d2f < __int_as_float(r.pk.z))) {
        double d2 = 0.0;
        for (int d = 0; d < 3; d++) {
            const double cm = a.st.x[d * a.st.cap_j + a.n + c];
            const double lo = a.box_lo[d * a.G + G.g], hi = a.box_hi[d * a.G + G.g];
            double gap = 0.0;
            if (cm < lo) gap = __dsub_rn(lo, cm);
            else if (cm > hi) gap = __dsub_rn(cm, hi);
            d2 = __dadd_rn(d2, __dmul_rn(gap, gap));
        }
        accept = cell_side(a, c) < __dmul_rn(a.theta, __dsqrt_rn(d2));
    }
    if (accept) return kEmitNode;
    return r.pk.w == 1 ? kEmitParticles : kOpen;  // (only a leaf is its whole subtree)
}

// The group's cell, its particle range and its FP32 box, as the list walk
// reads them (the FP64 box only where the screen cannot decide).
__device__ __forceinline__ GroupView group_view(const RbSim &a, int32_t g)
{
    GroupView V;
    V.g = g;
    V.gc = a.g_cell[g];
    const int4 pk = __ldg(&a.P.pack[V.gc]);
    V.gb = pk.x;
    V.ge = pk.y;
    const float4 l = a.box_f[2 * g], h = a.box_f[2 * g + 1];
    V.lof = make_float3(l.x, l.y, l.z);
    V.hif = make_float3(h.x, h.y, h.z);
    return V;
}

// The ancestors of each chunk's first cell, one thread per chunk: from the
// root to the parent in path[chunk][..kPath - 1], the entries before the root
// -1.  (A cell has at most kMaxDepth ancestors.)
template <bool kMany>
__global__ void k_paths(RB_ARGS)
{
    RB_SIM;
    for (int32_t k = blockIdx.x * blockDim.x + threadIdx.x; k < a.R; k += gridDim.x * blockDim.x) {
        int32_t *row = a.path + int64_t(k) * kPath;
        int32_t q = kPath;
        for (int32_t c = a.P.parent[k * a.chunk]; c >= 0 && q > 0; c = a.P.parent[c]) row[--q] = c;
        while (q > 0) row[--q] = -1;
    }
}

// The list walk, cut into chunks of `chunk` cells in pre-order: one thread per
// (group, chunk), a block taking kWalkThreads neighbouring groups (close in
// space) at one chunk, so that its lanes walk nearly the same cells, which the
// block stages first (a chunk of more than kWalkStage cells, in trees of more
// than 262144 cells, is read in place).  A thread first takes the decisions on the
// ancestors of the chunk's first cell, from the root down, until one is not
// opened: that cell is emitted by the chunk that holds it, and the walk here
// goes on behind its subtree (most chunks end there).  Then it walks the
// chunk's cells in pre-order, skipping every emitted cell's subtree.  The list
// of a group is the concatenation over the chunks: particles ascending, then
// nodes ascending, as in the sequential walk.
// The chunks around the groups' own cells take longest, so all rows of groups
// take those first (turn 0, then outwards on either side): otherwise a few of
// them run alone at the end.
// Pass 0 counts into cnt_p/cnt_n[g * R + k] (and zeroes both arrays'
// terminal entries); pass 1 writes at the scanned offsets.  cnt_n follows
// cnt_p's terminal entry, so one exclusive scan covers both (each read
// relative to its first entry).
// Bound by the decisions' latency.  Counts and entries of a rebuild of 32
// clusters with 1k to 32k particles, and of 262144 particles: a thread per
// (group, subtree of ncells / 256 cells) with a table of the topmost unopened
// cells above those subtrees, which spent most of its time on its start, 775 and
// 787 us, 583 and 730 us; a thread per chunk in launch order 180 and 308 us, 339
// and 538 us; with the staging and this order 164 and 275 us, 290 and 399 us.
// (Gathering each lane's entries into 16-byte stores, prefetching the next cell
// and more warps by fewer registers each made it slower.)
template <bool kMany, bool kWrite>
__global__ void __launch_bounds__(kWalkThreads) k_lists(RB_ARGS)
{
    if (kWrite) after_previous();
    else wait_previous();  // (the scan follows)
    RB_RECORD;
    __shared__ CellRec s_cell[kWalkStage];
    const int32_t R = a.R, n_row = (a.G + kWalkThreads - 1) / kWalkThreads;
    const int64_t n = a.n;
    int64_t *cnt_p = a.pair2, *cnt_n = a.pair2 + a.pairs + 1;
    const int64_t *scan_p = a.pscan2, *scan_n = a.pscan2 + a.pairs + 1;
    if (!kWrite && blockIdx.x == 0 && threadIdx.x == 0) cnt_p[a.pairs] = cnt_n[a.pairs] = 0;
    const int64_t pb = kWrite ? scan_p[0] : 0, nb = kWrite ? scan_n[0] : 0;
    if (kWrite && (scan_p[a.pairs] - pb) + (scan_n[a.pairs] - nb) > a.cap_list) return;  // (the host grows the lists)
    const int32_t turn = int32_t(blockIdx.x) / n_row, row = int32_t(blockIdx.x) - turn * n_row;
    if (turn >= R) return;  // (another simulation's grid)
    const int32_t g = row * kWalkThreads + int32_t(threadIdx.x);
    int32_t k = a.g_cell[min(row * kWalkThreads + kWalkThreads / 2, a.G - 1)] / a.chunk +
                ((turn & 1) ? (turn + 1) / 2 : -(turn / 2));
    if (k < 0) k += R;
    if (k >= R) k -= R;
    const int32_t first = k * a.chunk, end = min(first + a.chunk, a.ncells);
    const bool staged = a.chunk <= kWalkStage;
    if (staged)
        for (int32_t c = first + int32_t(threadIdx.x); c < end; c += kWalkThreads) s_cell[c - first] = load_cell(a, c);
    __syncthreads();
    if (g >= a.G) return;
    const int32_t *path = a.path + int64_t(k) * kPath;
    const GroupView V = group_view(a, g);
    int32_t c = first;
    for (int q = 0; q < kPath; q++) {
        const int32_t up = __ldg(&path[q]);
        if (up < 0) continue;
        const CellRec r = load_cell(a, up);
        if (decide(a, V, up, r) != kOpen) {
            c = up + r.pk.w;
            break;
        }
    }
    const int64_t q = int64_t(g) * R + k;
    int64_t wp = 0, wn = 0;
    if (kWrite && c < end) {
        wp = (scan_p[q] - pb) + (scan_n[int64_t(g) * R] - nb);
        wn = (scan_p[int64_t(g + 1) * R] - pb) + (scan_n[q] - nb);
    }
    int32_t np = 0, nn = 0;
    while (c < end) {
        const CellRec r = staged ? s_cell[c - first] : load_cell(a, c);
        const int dec = decide(a, V, c, r);
        if (dec == kEmitNode) {
            if (kWrite) a.lidx[wn++] = int32_t(n + c);
            nn++;
        } else if (dec == kEmitParticles) {
            const int32_t cnt = r.pk.y - r.pk.x;
            if (kWrite) {  // (four predicated stores a turn: half the instructions of a store a turn)
                int32_t *const o = a.lidx + wp;
                for (int32_t k = 0; k < cnt; k += 4)
#pragma unroll
                    for (int u = 0; u < 4; u++)
                        if (k + u < cnt) o[k + u] = r.pk.x + k + u;
                wp += cnt;
            }
            np += cnt;
        }
        c += dec == kOpen ? 1 : r.pk.w;
    }
    if (!kWrite) {
        cnt_p[q] = np;
        cnt_n[q] = nn;
    }
}

// off[g] = entries of all lists before group g (g = 0..G); tiles of <= tile_i
// particles per group and their list parts; the longest list
template <bool kMany>
__global__ void k_tile_counts(RB_ARGS)
{
    RB_SIM_BEFORE_CUB;
    const int32_t G = a.G, R = a.R;
    const int64_t *scan_p = a.pscan2, *scan_n = a.pscan2 + a.pairs + 1;
    const int64_t base = scan_p[0] + scan_n[0];
    int64_t *ntile = a.nt2, *nparts = a.nt2 + G + 1;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        ntile[G] = nparts[G] = 0;  // terminal entries of the scan
        a.off[G] = scan_p[a.pairs] + scan_n[a.pairs] - base;
    }
    unsigned long long lmax = 0ull;
    for (int32_t g = blockIdx.x * blockDim.x + threadIdx.x; g < G; g += gridDim.x * blockDim.x) {
        const int64_t q = int64_t(g) * R;
        const int64_t off = scan_p[q] + scan_n[q] - base;
        const int64_t L = scan_p[q + R] + scan_n[q + R] - base - off;
        a.off[g] = off;
        const int32_t c = a.g_cell[g];
        const int64_t cnt = a.P.end[c] - a.P.begin[c];
        const int64_t nt = (cnt + a.tile_i - 1) / a.tile_i;
        const int64_t parts = L > 0 ? (L + a.part_len - 1) / a.part_len : 1;
        ntile[g] = nt;
        nparts[g] = nt * parts;
        lmax = max(lmax, (unsigned long long)L);
    }
    if (lmax) atomicMax(&a.gc->lmax, lmax);
}

// tiles (none when they do not fit: the host reports it), and the list length
// and tile / work-item totals
template <bool kMany>
__global__ void k_tiles(RB_ARGS)
{
    RB_SIM;
    const int64_t *parts_off = a.tscan2 + a.G + 1;
    const int64_t t0 = a.tscan2[0], n_tiles = a.tscan2[a.G] - t0;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        a.gc->L = a.off[a.G];
        a.gc->n_tiles = n_tiles;
        a.gc->total_parts = parts_off[a.G] - parts_off[0];
    }
    if (n_tiles > a.cap_tiles) return;
    for (int32_t g = blockIdx.x * blockDim.x + threadIdx.x; g < a.G; g += gridDim.x * blockDim.x) {
        const int32_t c = a.g_cell[g];
        const int32_t b = a.P.begin[c], e = a.P.end[c];
        int64_t t = a.tscan2[g] - t0;
        for (int32_t p = b; p < e; p += a.tile_i) a.tiles[t++] = make_int4(p, min(p + a.tile_i, e), g, 0);
    }
}

// Closing step: the context's sizes on the device and, for the mixed form, the
// base records of every j entry (particles in their new order, then the new
// nodes).  Nothing when the lists or the tiles do not fit: the host then grows
// the lists and takes this step again, or fails.
template <bool kMany>
__global__ void k_finish(RB_ARGS)
{
    RB_SIM;
    const GCounts *gc = a.gc;
    if (gc->L > a.cap_list || gc->n_tiles > a.cap_tiles) return;
    const int64_t nj = a.n + gc->ncells;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        a.ds->n = a.n;
        a.ds->nj = nj;
        a.ds->n_tiles = int32_t(gc->n_tiles);
        a.ds->part_len = a.part_len;
        a.ds->work_item = a.work_item;
        a.ds->work_split = a.work_split;
    }
    if (a.st.base)
        for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < nj; q += (int64_t)gridDim.x * blockDim.x)
            refresh_base(a.st, q);
}

template <typename K, typename V>
int cub_sort_pairs(void *&tmp, size_t &tmp_bytes, const K *kin, K *kout, const V *vin, V *vout, int64_t n, int bits,
                   cudaStream_t st)
{
    size_t need = 0;
    if (cub::DeviceRadixSort::SortPairs(nullptr, need, kin, kout, vin, vout, (int)n, 0, bits, st) != cudaSuccess ||
        need == 0)
        return HH_ECUDA;
    if (need > tmp_bytes) {
        if (tmp) cudaFree(tmp);
        tmp = nullptr;
        tmp_bytes = 0;
        if (cudaMalloc(&tmp, need) != cudaSuccess) return HH_ENOMEM;
        tmp_bytes = need;
    }
    return cub::DeviceRadixSort::SortPairs(tmp, need, kin, kout, vin, vout, (int)n, 0, bits, st) == cudaSuccess
               ? HH_OK
               : HH_ECUDA;
}

template <typename T>
int cub_exclusive_sum(void *&tmp, size_t &tmp_bytes, const T *in, T *out, int64_t n, cudaStream_t st)
{
    size_t need = 0;
    if (cub::DeviceScan::ExclusiveSum(nullptr, need, in, out, (int)n, st) != cudaSuccess || need == 0) return HH_ECUDA;
    if (need > tmp_bytes) {
        if (tmp) cudaFree(tmp);
        tmp = nullptr;
        tmp_bytes = 0;
        if (cudaMalloc(&tmp, need) != cudaSuccess) return HH_ENOMEM;
        tmp_bytes = need;
    }
    return cub::DeviceScan::ExclusiveSum(tmp, need, in, out, (int)n, st) == cudaSuccess ? HH_OK : HH_ECUDA;
}

}  // namespace

// Buffers of the device builder, owned by the context (allocated on first use).
struct GTreeBuf {
    int64_t cap_n = 0, cap_c = 0;
    uint64_t *key = nullptr, *key2 = nullptr;
    int32_t *idx = nullptr, *perm = nullptr;
    Box *box = nullptr;
    double *root_side = nullptr;
    double *unit = nullptr;
    GCounts *gc = nullptr;      // device
    GCounts *gc_host = nullptr;  // pinned mirror
    float4 *box_f = nullptr;
    PCells P{};
    int64_t *cnt = nullptr, *pos = nullptr;  // [n + 1] cells and groups by first particle, and their scan
    int32_t *g_cell = nullptr;
    // [tile counts | part counts] and their one scan, each 2 (G + 1) long
    int64_t *ntile = nullptr, *tile_off = nullptr;
    double *mom = nullptr;                    // [cap_c][16] cell sums
    double *box_lo = nullptr, *box_hi = nullptr;  // [3][cap_g] group boxes
    State alt{};                 // second particle-state buffer for the reordering
    int64_t *ids = nullptr, *ids2 = nullptr;
    // (group, chunk) counts and their scans, grown on demand
    int64_t *pair_buf = nullptr;
    int64_t pair_cap = 0;
    int32_t *path_buf = nullptr;  // [R][kPath] ancestors of the chunks' first cells
    int64_t path_cap = 0;
    void *tmp = nullptr;
    size_t tmp_bytes = 0;
    std::vector<void *> all;
};

int64_t *hh_gtree_ids(GTreeBuf *g) { return g->ids; }

State hh_gtree_second(const hh_ctx *ctx) { return ctx->gtree->alt; }
int32_t *hh_gtree_flag(GTreeBuf *g) { return &g->gc->bad; }

// Ordered on the context's stream: the copy lands before the next rebuild's
// reordering kernel reads the ids (a copy on the legacy stream would not be
// ordered with a non-blocking stream).
int hh_gtree_set_ids(GTreeBuf *g, const int64_t *ids, int64_t n, cudaStream_t st)
{
    if (cudaMemcpyAsync(g->ids, ids, sizeof(int64_t) * n, cudaMemcpyHostToDevice, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
        return HH_ECUDA;
    return HH_OK;
}

// The second state set is swapped with the context's at every rebuild, so it
// is freed through its current pointers (the context frees the other set).
void hh_gtree_free(GTreeBuf *g)
{
    if (!g) return;
    for (void *p : g->all)
        if (p) cudaFree(p);
    for (double *p : {g->alt.x, g->alt.v, g->alt.a, g->alt.jk, g->alt.m, g->alt.t, g->alt.dt})
        if (p) cudaFree(p);
    if (g->tmp) cudaFree(g->tmp);
    if (g->pair_buf) cudaFree(g->pair_buf);
    if (g->path_buf) cudaFree(g->path_buf);
    if (g->gc_host) cudaFreeHost(g->gc_host);
    delete g;
}

namespace {

int gfail(hh_ctx *ctx, int code, const char *m)
{
    ctx->err = m;
    return hh_set_global_error(code, m);
}

template <typename T>
bool galloc(GTreeBuf *g, T **p, size_t count, bool track = true)
{
    if (cudaMalloc((void **)p, sizeof(T) * (count ? count : 1)) != cudaSuccess) {
        *p = nullptr;
        cudaGetLastError();
        return false;
    }
    if (track) g->all.push_back(*p);
    return true;
}

GTreeBuf *gtree_alloc(hh_ctx *ctx)
{
    GTreeBuf *g = new GTreeBuf;
    const int64_t n = ctx->cap_n, cc = ctx->cap_j;  // cells <= cap_j - n, capped by cap_j
    g->cap_n = n;
    g->cap_c = cc;
    bool ok = galloc(g, &g->key, n) && galloc(g, &g->key2, n) && galloc(g, &g->idx, n) && galloc(g, &g->perm, n) &&
              galloc(g, &g->box, 1) && galloc(g, &g->root_side, 1) && galloc(g, &g->P.begin, cc) &&
              galloc(g, &g->P.end, cc) && galloc(g, &g->P.depth, cc) && galloc(g, &g->P.parent, cc) &&
              galloc(g, &g->P.size, cc) && galloc(g, &g->P.arrived, cc) && galloc(g, &g->P.child, 2 * cc) &&
              galloc(g, &g->P.pack, cc) && galloc(g, &g->P.cf, cc) && galloc(g, &g->unit, 1) && galloc(g, &g->gc, 1) &&
              galloc(g, &g->box_f, 2 * ctx->cap_g) && galloc(g, &g->cnt, n + 1) && galloc(g, &g->pos, n + 1) &&
              galloc(g, &g->g_cell, ctx->cap_g) &&
              galloc(g, &g->mom, 16 * cc) && galloc(g, &g->box_lo, 3 * ctx->cap_g) &&
              galloc(g, &g->box_hi, 3 * ctx->cap_g) &&
              galloc(g, &g->ntile, 2 * (ctx->cap_g + 1)) && galloc(g, &g->tile_off, 2 * (ctx->cap_g + 1)) &&
              galloc(g, &g->ids, n) && galloc(g, &g->ids2, n);
    // the second state buffer mirrors the context's (same capacities)
    g->alt = ctx->st;
    g->alt.x = g->alt.v = g->alt.a = g->alt.jk = g->alt.m = g->alt.t = g->alt.dt = nullptr;
    ok = ok && galloc(g, &g->alt.x, 3 * ctx->cap_j, false) && galloc(g, &g->alt.v, 3 * ctx->cap_j, false) &&
         galloc(g, &g->alt.a, 3 * ctx->cap_j, false) && galloc(g, &g->alt.jk, 3 * ctx->cap_j, false) &&
         galloc(g, &g->alt.m, ctx->cap_j, false) && galloc(g, &g->alt.t, ctx->cap_j, false) &&
         galloc(g, &g->alt.dt, n, false);
    if (ok && cudaHostAlloc((void **)&g->gc_host, sizeof(GCounts), cudaHostAllocDefault) != cudaSuccess) {
        cudaGetLastError();
        g->gc_host = nullptr;
        ok = false;
    }
    if (!ok) {
        hh_gtree_free(g);
        return nullptr;
    }
    return g;
}

int64_t gtree_bytes(const hh_ctx *ctx)
{
    const int64_t n = ctx->cap_n, cc = ctx->cap_j, G = ctx->cap_g + 1;
    return n * (8 * 2 + 4 * 2 + 8 * 2) + (n + 1) * 8 * 2 + cc * (4 * 6 + 32 + 32 + 16 * 8) +
           G * (4 + 8 * 4 + 6 * 8 + 32) + ctx->cap_j * 8 * (12 + 2) + n * 8;
}

}  // namespace

namespace {

// The record of one simulation for the rebuild kernels, with the buffers of
// its context and of its device builder; sizes and scratch pointers are
// filled in as the build goes.
RbSim rb_sim(hh_ctx *ctx, GTreeBuf *g, double t)
{
    RbSim a{};
    a.st = ctx->st;
    a.alt = g->alt;
    a.P = g->P;
    a.gc = g->gc;
    a.box = g->box;
    a.root_side = g->root_side;
    a.unit = g->unit;
    a.key = g->key;
    a.key2 = g->key2;
    a.idx = g->idx;
    a.perm = g->perm;
    a.cnt = g->cnt;
    a.pos = g->pos;
    a.chain = g->idx;  // (the sort's input, not used after it)
    a.mom = g->mom;
    a.g_cell = g->g_cell;
    a.box_lo = g->box_lo;
    a.box_hi = g->box_hi;
    a.box_f = g->box_f;
    a.ids = g->ids;
    a.ids2 = g->ids2;
    a.group_of = ctx->group_of;
    a.off = ctx->off;
    a.lidx = ctx->idx;
    a.cap_list = ctx->cap_list;
    a.tiles = ctx->tiles;
    a.cap_tiles = ctx->cap_tiles;
    a.nt2 = g->ntile;
    a.tscan2 = g->tile_off;
    a.pair2 = g->pair_buf;
    a.pscan2 = nullptr;
    a.path = g->path_buf;
    a.t = t;
    a.theta = ctx->cfg.theta;
    a.n = ctx->n;
    a.cap_g = ctx->cap_g;
    a.cap_cells = int32_t(std::min<int64_t>(ctx->cap_j - ctx->n, INT32_MAX));
    a.leaf = ctx->cfg.leaf;
    a.n_crit = ctx->cfg.n_crit;
    a.order = ctx->cfg.order;
    a.tile_i = ctx->tile_i;
    a.part_len = ctx->part_len;
    a.ds = ctx->ds;
    a.work_item = ctx->cfg.work_item;
    a.work_split = ctx->cfg.work_split;
    return a;
}

// After the reordering the context's state and the builder's second buffer
// trade places.
void swap_state(hh_ctx *ctx, GTreeBuf *g)
{
    std::swap(ctx->st.x, g->alt.x);
    std::swap(ctx->st.v, g->alt.v);
    std::swap(ctx->st.a, g->alt.a);
    std::swap(ctx->st.jk, g->alt.jk);
    std::swap(ctx->st.m, g->alt.m);
    std::swap(ctx->st.t, g->alt.t);
    std::swap(ctx->st.dt, g->alt.dt);
    std::swap(g->ids, g->ids2);
    ctx->ids_on_device = true;  // (whether the build succeeds or not)
    ctx->ids_on_both = false;
}

int gtree_prepare(hh_ctx *ctx)
{
    // A non-sticky error left pending by earlier runtime calls would make the
    // library calls below report failure; every call here is checked itself.
    cudaGetLastError();
    if (!ctx->gtree) {
        ctx->gtree = gtree_alloc(ctx);
        if (!ctx->gtree) return gfail(ctx, HH_ENOMEM, "hh_rebuild: device tree buffers do not fit");
        ctx->device_bytes += gtree_bytes(ctx);
        // particle ids live on the device from now on
        if (hh_gtree_set_ids(ctx->gtree, ctx->ids.data(), ctx->n, ctx->stream) != HH_OK)
            return gfail(ctx, HH_ECUDA, "hh_rebuild: id upload failed");
    }
    return HH_OK;
}

// Grows a device buffer to at least `need` elements (its contents are not kept).
template <typename T>
bool grow(T *&p, int64_t &cap, int64_t need)
{
    if (need <= cap) return true;
    if (p) cudaFree(p);
    p = nullptr;
    cap = 0;
    if (cudaMalloc((void **)&p, sizeof(T) * size_t(need)) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    cap = need;
    return true;
}

int grow_list(hh_ctx *ctx, int64_t L)
{
    if (L <= ctx->cap_list) return HH_OK;  // the list buffer grows by a quarter beyond the need
    const int64_t cap = L + L / 4 + 1024;
    int32_t *idx = nullptr;
    if (cudaMalloc(&idx, sizeof(int32_t) * cap) != cudaSuccess) {
        cudaGetLastError();
        return gfail(ctx, HH_ENOMEM, "hh_rebuild: lists do not fit in device memory");
    }
    cudaFree(ctx->idx);
    ctx->idx = idx;
    ctx->device_bytes += (cap - ctx->cap_list) * int64_t(sizeof(int32_t));
    ctx->cap_list = cap;
    return HH_OK;
}

// Cells of a walk chunk: small enough that all (group, chunk) threads fill the
// chip, large enough that a thread's start (its group's record, the path, one
// pair of counts) is spread over many cells, and at most about 512 chunks per
// tree, so that the pair counts stay linear in the groups.  Rebuild of 32
// clusters with 1k to 32k particles at 32, 128, 256, 512 cells: 2.45, 2.35,
// 2.40, 2.41 ms; of 262144 particles at 128, 256, 512: 1.92, 1.92, 1.85 ms.
int32_t walk_chunk(double group_cells, int32_t max_cells)
{
    int32_t c = 32;
    while (c < 512 && group_cells / (2.0 * c) >= 600e3) c *= 2;
    while (c < max_cells / 512) c *= 2;
    return c;
}

// blocks of the walk: one per (kWalkThreads groups, chunk)
int64_t walk_blocks(int32_t G, int32_t R) { return int64_t(R) * ((G + kWalkThreads - 1) / kWalkThreads); }

}  // namespace

// Called by hh_rebuild when the context builds on the device.
int hh_rebuild_device(hh_ctx *ctx, double t)
{
    int rc = gtree_prepare(ctx);
    if (rc) return rc;
    cudaStream_t st = ctx->stream;
    const int64_t n = ctx->n;
    GTreeBuf *g = ctx->gtree;
    // element-wise kernels: a thread per particle at most (they stride over
    // cells, groups and particles alike), so a small tree launches few blocks
    const int grid = int(std::max<int64_t>(1, std::min<int64_t>(ctx->elem_grid, (n + 255) / 256)));
    // (those with 8 or 16 lanes per cell, or a warp per group: about four
    // lanes per particle)
    const int grid8 = int(std::max<int64_t>(1, std::min<int64_t>(2 * ctx->elem_grid, (4 * n + 255) / 256)));
    int64_t launches = 0;
    RbSim a = rb_sim(ctx, g, t);
    // Sizes stay on the device (GCounts) and the host reads them twice: after
    // the tree and the groups, and at the end.
    auto read_counts = [&]() {
        cudaMemcpyAsync(g->gc_host, g->gc, sizeof(GCounts), cudaMemcpyDeviceToHost, st);
        return cudaStreamSynchronize(st) == cudaSuccess;
    };
    // 1. bounding box, synchronisation check, keys, sort
    launch_after(k_root_init<false>, dim3(1), dim3(1), st, true, a, nullptr);
    launch_after(k_box<false>, dim3(grid), dim3(256), st, true, a, nullptr);
    launch_after(k_keys<false>, dim3(grid), dim3(256), st, true, a, nullptr);
    launches += 3;
    {
        size_t need = 0;
        if (cub::DeviceRadixSort::SortPairs(nullptr, need, g->key, g->key2, g->idx, g->perm, (int)n, 0, 63, st) !=
                cudaSuccess ||
            need == 0)
            return gfail(ctx, HH_ECUDA, "hh_rebuild: key sort size query failed");
        if (need > g->tmp_bytes) {
            if (g->tmp) cudaFree(g->tmp);
            g->tmp = nullptr;
            if (cudaMalloc(&g->tmp, need) != cudaSuccess) return gfail(ctx, HH_ENOMEM, "hh_rebuild: sort buffer");
            g->tmp_bytes = need;
        }
        if (cub::DeviceRadixSort::SortPairs(g->tmp, need, g->key, g->key2, g->idx, g->perm, (int)n, 0, 63, st) !=
            cudaSuccess)
            return gfail(ctx, HH_ECUDA, "hh_rebuild: key sort failed");
    }
    // 2. cells and groups, particles into Morton order and node records, group
    //    boxes: all into the builder's buffers, which become the context's when
    //    the tree is known to fit
    launch_after(k_chains<false>, dim3(grid), dim3(256), st, true, a, nullptr);
    if ((rc = cub_exclusive_sum(g->tmp, g->tmp_bytes, a.cnt, a.pos, n + 1, st)))
        return gfail(ctx, rc, "hh_rebuild: scan failed");
    launch_after(k_begin_cells<false>, dim3(grid), dim3(256), st, true, a, nullptr);
    launch_after(k_cells<false>, dim3(grid8), dim3(256), st, true, a, nullptr);
    launch_after(k_permute<false>, dim3(grid), dim3(256), st, true, a, nullptr);
    launch_after(k_moments<false>, dim3(grid8), dim3(256), st, true, a, nullptr);
    launch_after(k_node_records<false>, dim3(grid), dim3(128), st, true, a, nullptr);
    launch_after(k_group_box<false>, dim3(grid8), dim3(256), st, true, a, nullptr);
    launches += 7;
    if (!read_counts()) return gfail(ctx, HH_ECUDA, "hh_rebuild: tree build failed");
    if (g->gc_host->bad) return gfail(ctx, HH_ESTATE, "hh_rebuild: particles are not synchronised at t");
    if (g->gc_host->overflow)
        return gfail(ctx, HH_ENOMEM, "hh_rebuild: tree exceeds nj_max (more cells than room for nodes)");
    const int32_t ncells = g->gc_host->ncells;
    a.ncells = ncells;
    swap_state(ctx, g);
    a.st = ctx->st;
    a.alt = g->alt;
    a.ids = g->ids;
    a.ids2 = g->ids2;
    const int32_t G = g->gc_host->G;
    if (G > ctx->cap_g) return gfail(ctx, HH_ENOMEM, "hh_rebuild: more groups than groups_max");
    a.G = G;
    // 3. per-(group, chunk) list counts, one scan, offsets, tiles, write
    a.chunk = walk_chunk(double(G) * ncells, ncells);
    a.R = (ncells + a.chunk - 1) / a.chunk;
    if (!grow(g->path_buf, g->path_cap, int64_t(a.R) * kPath))
        return gfail(ctx, HH_ENOMEM, "hh_rebuild: list walk table does not fit");
    a.path = g->path_buf;
    launch_after(k_paths<false>, dim3((a.R + 127) / 128), dim3(128), st, true, a, nullptr);
    const int64_t pairs = int64_t(G) * a.R;
    if (2 * (pairs + 1) >= int64_t(INT32_MAX))  // (one scan covers both count arrays)
        return gfail(ctx, HH_ENOMEM, "hh_rebuild: too many (group, chunk) pairs");
    if (!grow(g->pair_buf, g->pair_cap, 4 * (pairs + 1)))
        return gfail(ctx, HH_ENOMEM, "hh_rebuild: list count buffers do not fit");
    a.pairs = pairs;
    a.pair2 = g->pair_buf;
    a.pscan2 = g->pair_buf + 2 * (pairs + 1);
    const int64_t lgrid = walk_blocks(G, a.R);
    launch_after(k_lists<false, false>, dim3(unsigned(lgrid)), dim3(kWalkThreads), st, true, a, nullptr);
    if ((rc = cub_exclusive_sum(g->tmp, g->tmp_bytes, a.pair2, a.pscan2, 2 * (pairs + 1), st)))  // cnt_p, cnt_n at once
        return gfail(ctx, rc, "hh_rebuild: scan failed");
    // 4. tiles and their work-item capacity (from the list lengths), entries and
    //    closing step: the host reads the sizes after all of it, and takes the
    //    last two again if the lists had to grow
    launch_after(k_tile_counts<false>, dim3(grid), dim3(256), st, true, a, nullptr);
    if ((rc = cub_exclusive_sum(g->tmp, g->tmp_bytes, g->ntile, g->tile_off, 2 * (int64_t(G) + 1), st)))
        return gfail(ctx, rc, "hh_rebuild: scan failed");
    launch_after(k_tiles<false>, dim3(grid), dim3(256), st, true, a, nullptr);
    launches += 4;
    int64_t L = 0, n_tiles = 0;
    const int fgrid = int(std::min<int64_t>(ctx->elem_grid, (n + ncells + 255) / 256));
    for (int pass = 0; pass < 2; pass++) {
        launch_after(k_lists<false, true>, dim3(unsigned(lgrid)), dim3(kWalkThreads), st, true, a, nullptr);
        launch_after(k_finish<false>, dim3(fgrid), dim3(256), st, true, a, nullptr);
        launches += 2;
        if (!read_counts()) return gfail(ctx, HH_ECUDA, "hh_rebuild: list count failed");
        L = g->gc_host->L;
        n_tiles = g->gc_host->n_tiles;
        if (n_tiles > ctx->cap_tiles) return gfail(ctx, HH_ENOMEM, "hh_rebuild: too many tiles");
        if (L <= ctx->cap_list) break;
        if ((rc = grow_list(ctx, L))) return rc;
        a.lidx = ctx->idx;
        a.cap_list = ctx->cap_list;
    }
    const cudaError_t ce = cudaGetLastError();
    if (ce != cudaSuccess) return gfail(ctx, HH_ECUDA, cudaGetErrorString(ce));
    hh_count_launches(launches);  // kernels of this file; the radix sort and the scans are CUB's
    ctx->nj = n + ncells;
    ctx->n_groups = G;
    ctx->list_len = L;
    ctx->n_tiles = int32_t(n_tiles);
    return hh_finish_device_rebuild(ctx, g->gc_host->total_parts, int64_t(g->gc_host->lmax));
}

// ---------------------------------------------------------------- many at once
// Scratch of the batched rebuild: the simulations' records (one region per
// stage, so that a record is never rewritten while its copy to the device may
// be pending), their counts, the segment offsets of the sorts, and the arrays
// that the sorts and scans run over as one (each simulation a slice).
struct RbScratch {
    cudaStream_t stream = nullptr;
    RbSim *h_sims = nullptr, *d_sims = nullptr;  // [kStages][cap_sims]
    GCounts *h_gc = nullptr, *d_gc = nullptr;     // [cap_sims], by the simulation's slot
    int32_t *h_seg = nullptr, *d_seg = nullptr;   // [cap_sims + 1] particle segments
    int64_t cap_sims = 0;
    uint64_t *key = nullptr, *key2 = nullptr;
    int32_t *idx = nullptr, *perm = nullptr;
    int64_t cap_key = 0, cap_key2 = 0, cap_idx = 0, cap_perm = 0;
    int64_t *cnt = nullptr, *pos = nullptr;
    int64_t cap_cnt = 0, cap_pos = 0;
    int64_t *pair2 = nullptr, *pscan2 = nullptr;
    int64_t cap_pair2 = 0, cap_pscan2 = 0;
    int32_t *path = nullptr;
    int64_t cap_path = 0;
    int64_t *nt2 = nullptr, *tscan2 = nullptr;
    int64_t cap_nt2 = 0, cap_tscan2 = 0;
    void *tmp = nullptr;
    size_t tmp_bytes = 0;
};

namespace {

constexpr int kStages = 4;  // the records of stages 0..3 (after each read of the counts, and as groups are known)

void rb_free_sims(RbScratch *r)
{
    for (void *p : {(void *)r->d_sims, (void *)r->d_gc, (void *)r->d_seg})
        if (p) cudaFree(p);
    for (void *p : {(void *)r->h_sims, (void *)r->h_gc, (void *)r->h_seg})
        if (p) cudaFreeHost(p);
    r->d_sims = r->h_sims = nullptr;
    r->d_gc = r->h_gc = nullptr;
    r->d_seg = r->h_seg = nullptr;
    r->cap_sims = 0;
}

bool rb_reserve_sims(RbScratch *r, int64_t k)
{
    if (k <= r->cap_sims) return true;
    rb_free_sims(r);
    const int64_t cap = k + k / 2 + 8;
    if (cudaMalloc(&r->d_sims, sizeof(RbSim) * kStages * cap) != cudaSuccess ||
        cudaMalloc(&r->d_gc, sizeof(GCounts) * cap) != cudaSuccess ||
        cudaMalloc(&r->d_seg, sizeof(int32_t) * (cap + 1)) != cudaSuccess ||
        cudaHostAlloc((void **)&r->h_sims, sizeof(RbSim) * kStages * cap, cudaHostAllocDefault) != cudaSuccess ||
        cudaHostAlloc((void **)&r->h_gc, sizeof(GCounts) * cap, cudaHostAllocDefault) != cudaSuccess ||
        cudaHostAlloc((void **)&r->h_seg, sizeof(int32_t) * (cap + 1), cudaHostAllocDefault) != cudaSuccess) {
        cudaGetLastError();
        rb_free_sims(r);
        return false;
    }
    r->cap_sims = cap;
    return true;
}

// grows a scratch array (a quarter beyond the need)
template <typename T>
bool rb_grow(T *&p, int64_t &cap, int64_t need)
{
    return need <= cap || grow(p, cap, need + need / 4 + 1024);
}

// The simulation (segment) of each sorted particle, then, once they are in
// simulation order again, each one's index within its simulation and its key.
__global__ void k_sim_of(const int32_t *seg, int k, const int32_t *part, uint32_t *sim, int32_t n)
{
    for (int32_t j = blockIdx.x * blockDim.x + threadIdx.x; j < n; j += gridDim.x * blockDim.x) {
        const int32_t p = part[j];
        int l = 0, h = k - 1;  // the last segment that begins at or before p
        while (l < h) {
            const int mid = (l + h + 1) >> 1;
            if (__ldg(&seg[mid]) <= p) l = mid;
            else h = mid - 1;
        }
        sim[j] = uint32_t(l);
    }
}

__global__ void k_sim_order(const int32_t *seg, const uint32_t *sim, const int32_t *part, const uint64_t *key,
                            int32_t *perm, uint64_t *key2, int32_t n)
{
    for (int32_t j = blockIdx.x * blockDim.x + threadIdx.x; j < n; j += gridDim.x * blockDim.x) {
        const int32_t p = part[j];
        perm[j] = p - seg[sim[j]];
        key2[j] = key[p];
    }
}

}  // namespace

RbScratch *hh_rb_scratch_create()
{
    RbScratch *r = new RbScratch;
    if (cudaStreamCreateWithFlags(&r->stream, cudaStreamNonBlocking) != cudaSuccess) {
        cudaGetLastError();
        delete r;
        return nullptr;
    }
    return r;
}

void hh_rb_scratch_free(RbScratch *r)
{
    if (!r) return;
    cudaStreamSynchronize(r->stream);
    rb_free_sims(r);
    for (void *p : {(void *)r->key, (void *)r->key2, (void *)r->idx, (void *)r->perm, (void *)r->cnt, (void *)r->pos,
                    (void *)r->pair2, (void *)r->pscan2, (void *)r->path, (void *)r->nt2, (void *)r->tscan2, r->tmp})
        if (p) cudaFree(p);
    cudaStreamDestroy(r->stream);
    delete r;
}

// Rebuilds k contexts on the device at once: every step of hh_rebuild_device
// runs as one launch over all of them (simulation = blockIdx.y), the key sort
// and each scan as one over all simulations' arrays (a simulation reads its
// slice of a scan relative to its first entry).  Each context gets the tree, groups, lists and node records it
// would get alone.  rcs[s] receives context s's result; a context that fails
// leaves the build at that point and the others go on.
int hh_rebuild_device_many(hh_ctx *const *ctxs, const double *ts, int k, int *rcs, RbScratch *r)
{
    if (k < 1 || !r) return HH_EINVAL;
    cudaStream_t st = r->stream;
    if (!rb_reserve_sims(r, k)) return HH_ENOMEM;
    std::vector<int> act, slot;  // contexts still in the build, and their count slots
    for (int s = 0; s < k; s++) {
        rcs[s] = gtree_prepare(ctxs[s]);
        if (rcs[s] == HH_OK && cudaStreamSynchronize(ctxs[s]->stream) != cudaSuccess)
            rcs[s] = gfail(ctxs[s], HH_ECUDA, "hh_rebuild: context stream failed");
        if (rcs[s] == HH_OK) act.push_back(s);
    }
    if (act.empty()) return HH_OK;
    // (the largest first: the blocks that take longest do not start last)
    std::stable_sort(act.begin(), act.end(), [&](int p, int q) { return ctxs[p]->n > ctxs[q]->n; });
    const int K0 = int(act.size());
    int stage = 0;
    auto H = [&](int q) -> RbSim & { return r->h_sims[stage * r->cap_sims + q]; };
    auto D = [&]() { return r->d_sims + stage * r->cap_sims; };
    auto upload = [&]() {
        return cudaMemcpyAsync(D(), &H(0), sizeof(RbSim) * act.size(), cudaMemcpyHostToDevice, st) == cudaSuccess;
    };
    auto read_counts = [&]() {
        return cudaMemcpyAsync(r->h_gc, r->d_gc, sizeof(GCounts) * K0, cudaMemcpyDeviceToHost, st) == cudaSuccess &&
               cudaStreamSynchronize(st) == cudaSuccess;
    };
    auto cnt = [&](size_t q) -> const GCounts & { return r->h_gc[slot[q]]; };
    // the next stage's records: those of the contexts for which keep(q) holds
    auto next_stage = [&](const std::function<bool(size_t)> &keep) {
        size_t w = 0;
        RbSim *src = r->h_sims + stage * r->cap_sims, *dst = r->h_sims + (stage + 1) * r->cap_sims;
        for (size_t q = 0; q < act.size(); q++)
            if (keep(q)) {
                dst[w] = src[q];
                act[w] = act[q];
                slot[w++] = slot[q];
            }
        act.resize(w);
        slot.resize(w);
        stage++;
    };
    auto fail_all = [&](int code, const char *m) {
        for (int s : act) rcs[s] = gfail(ctxs[s], code, m);
        act.clear();
        return HH_OK;
    };
    // exclusive prefix of the particle counts as segment offsets
    auto segments = [&](int64_t *total) {
        int64_t acc = 0;
        for (size_t q = 0; q < act.size(); q++) {
            r->h_seg[q] = int32_t(acc);
            acc += ctxs[act[q]]->n;
            if (acc >= int64_t(INT32_MAX)) return false;
        }
        r->h_seg[act.size()] = int32_t(acc);
        *total = acc;
        return cudaMemcpyAsync(r->d_seg, r->h_seg, sizeof(int32_t) * (act.size() + 1), cudaMemcpyHostToDevice, st) ==
               cudaSuccess;
    };
    // blocks per simulation of the element-wise kernels (they stride over
    // cells, groups and particles alike): a thread per particle of the
    // largest one, but no more than about twice the threads the SMs hold in
    // all
    int64_t launches = 0, gx = 1;
    for (int s : act) gx = std::max<int64_t>(gx, std::min<int64_t>(ctxs[s]->elem_grid, (ctxs[s]->n + 255) / 256));
    // (those with 8 or 16 lanes per cell, or a warp per group)
    const int64_t gx8 = std::max<int64_t>(
        1, std::min<int64_t>(4 * gx, 8 * int64_t(ctxs[act[0]]->elem_grid) / int64_t(act.size())));
    gx = std::max<int64_t>(1, std::min<int64_t>(gx, 2 * int64_t(ctxs[act[0]]->elem_grid) / int64_t(act.size())));
    // 1. bounding boxes, keys, sort
    int64_t tot = 0;
    if (!segments(&tot)) return fail_all(HH_ENOMEM, "hh_rebuild: batch too large");
    if (!rb_grow(r->key, r->cap_key, tot) || !rb_grow(r->key2, r->cap_key2, tot) || !rb_grow(r->idx, r->cap_idx, tot) ||
        !rb_grow(r->perm, r->cap_perm, tot) || !rb_grow(r->cnt, r->cap_cnt, tot + K0) ||
        !rb_grow(r->pos, r->cap_pos, tot + K0))
        return fail_all(HH_ENOMEM, "hh_rebuild: batch key buffers do not fit");
    for (size_t q = 0; q < act.size(); q++) {
        hh_ctx *ctx = ctxs[act[q]];
        GTreeBuf *g = ctx->gtree;
        RbSim &a = H(int(q));
        a = rb_sim(ctx, g, ts[act[q]]);
        const int64_t o = r->h_seg[q];
        a.gc = r->d_gc + q;
        a.key = r->key + o;
        a.key2 = r->key2 + o;
        a.idx = r->idx + o;
        a.seg = int32_t(o);
        a.perm = r->perm + o;
        a.chain = a.idx;  // (the sort's input, not used after it)
        a.cnt = r->cnt + o + int64_t(q);  // (a terminal entry each)
        a.pos = r->pos + o + int64_t(q);
        slot.push_back(int(q));
    }
    if (!upload()) return fail_all(HH_ECUDA, "hh_rebuild: batch upload failed");
    const dim3 g1 = dim3(unsigned(gx), unsigned(K0)), one1(1, unsigned(K0)), g8 = dim3(unsigned(gx8), unsigned(K0));
    launch_after(k_root_init<true>, one1, dim3(1), st, true, RbSim{}, D());
    launch_after(k_box<true>, g1, dim3(256), st, true, RbSim{}, D());
    launch_after(k_keys<true>, g1, dim3(256), st, true, RbSim{}, D());
    launches += 3;
    // one stable sort of all keys, then one by simulation (a segmented sort
    // gives each simulation one block: a rebuild of 32 clusters with 1k to 32k
    // particles then takes 2.01 ms, this way 1.70 ms)
    int rc = cub_sort_pairs(r->tmp, r->tmp_bytes, r->key, r->key2, r->idx, r->perm, tot, 63, st);
    if (rc) return fail_all(rc, "hh_rebuild: batch key sort failed");
    if (K0 > 1) {
        uint32_t *sim = reinterpret_cast<uint32_t *>(r->cnt), *sim2 = sim + tot;  // (not yet in use)
        const unsigned sgrid = unsigned(std::min<int64_t>((tot + 255) / 256, int64_t(ctxs[act[0]]->elem_grid)));
        int bits = 1;
        while ((1 << bits) < K0) bits++;
        k_sim_of<<<sgrid, 256, 0, st>>>(r->d_seg, K0, r->perm, sim, int32_t(tot));
        if ((rc = cub_sort_pairs(r->tmp, r->tmp_bytes, sim, sim2, r->perm, r->idx, tot, bits, st)))
            return fail_all(rc, "hh_rebuild: batch key sort failed");
        k_sim_order<<<sgrid, 256, 0, st>>>(r->d_seg, sim2, r->idx, r->key, r->perm, r->key2, int32_t(tot));
        launches += 2;
    }
    // 2. cells and groups, reordering, node records, group boxes, all into the
    //    builders' buffers
    launch_after(k_chains<true>, g1, dim3(256), st, true, RbSim{}, D());
    if ((rc = cub_exclusive_sum(r->tmp, r->tmp_bytes, r->cnt, r->pos, tot + K0, st)))
        return fail_all(rc, "hh_rebuild: batch scan failed");
    launch_after(k_begin_cells<true>, g1, dim3(256), st, true, RbSim{}, D());
    launch_after(k_cells<true>, g8, dim3(256), st, true, RbSim{}, D());
    launch_after(k_permute<true>, g1, dim3(256), st, true, RbSim{}, D());
    launch_after(k_moments<true>, g8, dim3(256), st, true, RbSim{}, D());
    launch_after(k_node_records<true>, g1, dim3(128), st, true, RbSim{}, D());
    launch_after(k_group_box<true>, g8, dim3(256), st, true, RbSim{}, D());
    launches += 7;
    if (!read_counts()) return fail_all(HH_ECUDA, "hh_rebuild: tree build failed");
    next_stage([&](size_t q) {
        if (cnt(q).bad) {
            rcs[act[q]] = gfail(ctxs[act[q]], HH_ESTATE, "hh_rebuild: particles are not synchronised at t");
            return false;
        }
        if (cnt(q).overflow) {
            rcs[act[q]] =
                gfail(ctxs[act[q]], HH_ENOMEM, "hh_rebuild: tree exceeds nj_max (more cells than room for nodes)");
            return false;
        }
        return true;
    });
    if (act.empty()) return HH_OK;
    for (size_t q = 0; q < act.size(); q++) {  // the reordered state becomes the context's
        hh_ctx *ctx = ctxs[act[q]];
        GTreeBuf *g = ctx->gtree;
        swap_state(ctx, g);
        RbSim &a = H(int(q));
        a.st = ctx->st;
        a.alt = g->alt;
        a.ids = g->ids;
        a.ids2 = g->ids2;
        a.ncells = cnt(q).ncells;
    }
    next_stage([&](size_t q) {
        if (cnt(q).G > ctxs[act[q]]->cap_g) {
            rcs[act[q]] = gfail(ctxs[act[q]], HH_ENOMEM, "hh_rebuild: more groups than groups_max");
            return false;
        }
        return true;
    });
    if (act.empty()) return HH_OK;
    // 3. per-(group, chunk) list counts (one scan), offsets, tiles (one scan)
    int64_t t_path = 0, t_pair = 0, t_nt = 0, lgrid = 1;
    int32_t max_cells = 0, max_R = 1;
    double group_cells = 0.0;
    for (size_t q = 0; q < act.size(); q++) {
        group_cells += double(cnt(q).G) * cnt(q).ncells;
        max_cells = std::max(max_cells, cnt(q).ncells);
    }
    const int32_t chunk = walk_chunk(group_cells, max_cells);
    for (size_t q = 0; q < act.size(); q++) {
        RbSim &a = H(int(q));
        a.G = cnt(q).G;
        a.chunk = chunk;
        a.R = (a.ncells + a.chunk - 1) / a.chunk;
        a.pairs = int64_t(a.G) * a.R;
        a.path = reinterpret_cast<int32_t *>(t_path);  // offsets for now
        a.pair2 = reinterpret_cast<int64_t *>(t_pair);
        a.nt2 = reinterpret_cast<int64_t *>(t_nt);
        t_path += int64_t(a.R) * kPath;
        t_pair += 2 * (a.pairs + 1);
        t_nt += 2 * (int64_t(a.G) + 1);
        max_R = std::max(max_R, a.R);
        lgrid = std::max<int64_t>(lgrid, walk_blocks(a.G, a.R));
    }
    if (t_pair >= int64_t(INT32_MAX) || t_nt >= int64_t(INT32_MAX))  // (one CUB scan each)
        return fail_all(HH_ENOMEM, "hh_rebuild: too many (group, chunk) pairs in one batch");
    if (!rb_grow(r->path, r->cap_path, t_path) || !rb_grow(r->pair2, r->cap_pair2, t_pair) ||
        !rb_grow(r->pscan2, r->cap_pscan2, t_pair) || !rb_grow(r->nt2, r->cap_nt2, t_nt) ||
        !rb_grow(r->tscan2, r->cap_tscan2, t_nt))
        return fail_all(HH_ENOMEM, "hh_rebuild: batch list buffers do not fit");
    for (size_t q = 0; q < act.size(); q++) {
        RbSim &a = H(int(q));
        const int64_t o_path = reinterpret_cast<int64_t>(a.path), o_pair = reinterpret_cast<int64_t>(a.pair2),
                      o_nt = reinterpret_cast<int64_t>(a.nt2);
        a.path = r->path + o_path;
        a.pair2 = r->pair2 + o_pair;
        a.pscan2 = r->pscan2 + o_pair;
        a.nt2 = r->nt2 + o_nt;
        a.tscan2 = r->tscan2 + o_nt;
    }
    const int K3 = int(act.size());
    const dim3 g3 = dim3(unsigned(gx), unsigned(K3)), one3(1, unsigned(K3));
    const dim3 lg3 = dim3(unsigned(lgrid), unsigned(K3));
    if (!upload()) return fail_all(HH_ECUDA, "hh_rebuild: batch upload failed");
    launch_after(k_paths<true>, dim3(unsigned((max_R + 127) / 128), unsigned(K3)), dim3(128), st, true, RbSim{}, D());
    launch_after(k_lists<true, false>, lg3, dim3(kWalkThreads), st, true, RbSim{}, D());
    if ((rc = cub_exclusive_sum(r->tmp, r->tmp_bytes, r->pair2, r->pscan2, t_pair, st)))
        return fail_all(rc, "hh_rebuild: batch scan failed");
    launch_after(k_tile_counts<true>, g3, dim3(256), st, true, RbSim{}, D());
    if ((rc = cub_exclusive_sum(r->tmp, r->tmp_bytes, r->nt2, r->tscan2, t_nt, st)))
        return fail_all(rc, "hh_rebuild: batch scan failed");
    launch_after(k_tiles<true>, g3, dim3(256), st, true, RbSim{}, D());
    // 4. entries and closing step, again for the contexts whose lists had to
    //    grow; then per context on the host: work-item capacity and sizes
    int64_t fx = 1;
    for (size_t q = 0; q < act.size(); q++)
        fx = std::max<int64_t>(
            fx, std::min<int64_t>(ctxs[act[q]]->elem_grid, (ctxs[act[q]]->n + cnt(q).ncells + 255) / 256));
    auto entries = [&]() {
        const unsigned k = unsigned(act.size());
        launch_after(k_lists<true, true>, dim3(unsigned(lgrid), k), dim3(kWalkThreads), st, true, RbSim{}, D());
        launch_after(k_finish<true>, dim3(unsigned(fx), k), dim3(256), st, true, RbSim{}, D());
        launches += 2;
    };
    entries();
    launches += 4;
    if (!read_counts()) return fail_all(HH_ECUDA, "hh_rebuild: list count failed");
    const std::vector<int> all_act = act, all_slot = slot;
    std::vector<char> done(all_act.size(), 0);  // (by position in all_act)
    next_stage([&](size_t q) {
        hh_ctx *ctx = ctxs[act[q]];
        if (cnt(q).n_tiles > ctx->cap_tiles) {
            rcs[act[q]] = gfail(ctx, HH_ENOMEM, "hh_rebuild: too many tiles");
            return false;
        }
        if (cnt(q).L <= ctx->cap_list) {
            done[q] = 1;
            return false;
        }
        if ((rcs[act[q]] = grow_list(ctx, cnt(q).L)) != HH_OK) return false;
        done[q] = 1;
        return true;
    });
    if (!act.empty()) {
        for (size_t q = 0; q < act.size(); q++) {
            H(int(q)).lidx = ctxs[act[q]]->idx;
            H(int(q)).cap_list = ctxs[act[q]]->cap_list;
        }
        if (!upload()) return fail_all(HH_ECUDA, "hh_rebuild: batch upload failed");
        entries();
    }
    const cudaError_t ce = cudaGetLastError();
    const bool ok = ce == cudaSuccess && cudaStreamSynchronize(st) == cudaSuccess;
    for (size_t q = 0; q < all_act.size(); q++) {
        if (!done[q]) continue;
        hh_ctx *ctx = ctxs[all_act[q]];
        const GCounts &c = r->h_gc[all_slot[q]];
        if (!ok) {
            rcs[all_act[q]] = gfail(ctx, HH_ECUDA, "hh_rebuild: batch build failed");
            continue;
        }
        ctx->nj = ctx->n + c.ncells;
        ctx->n_groups = c.G;
        ctx->list_len = c.L;
        ctx->n_tiles = int32_t(c.n_tiles);
        rcs[all_act[q]] = hh_finish_device_rebuild(ctx, c.total_parts, int64_t(c.lmax));
    }
    hh_count_launches(launches);  // kernels of this file; the sorts and scans are CUB's
    return HH_OK;
}
