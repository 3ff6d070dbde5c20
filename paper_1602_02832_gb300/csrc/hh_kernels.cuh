// Device code of the list-driven Hermite hot path (sm_103a).
//
// One block step (Section 2, tree-loop steps 2-7) is three kernels:
//   k_predict  every j entry (particles and tree nodes) to the block time
//              (GRAPE predictor; step 4), written as packed records;
//              and, with one ballot per static i tile, appends the work
//              items (tile, list part) of tiles with active particles
//              (t_i + dt_i == t_next, step 2);
//   k_force    CTAs pull work items from a queue and sum acc / jerk / pot
//              over the item's part of the group's list (steps 4a + 5);
//   k_correct  4th-order Hermite corrector + Aarseth block step (step 6),
//              and the min over t_i + dt_i that starts the next step.
// No kernel waits on another CTA; there are no spin loops.
#pragma once

#include <cstdint>
#include <type_traits>
#include <cuda_runtime.h>

#include "hh_pair64.cuh"

namespace hh {

constexpr int kThreads = 128;  // threads per force CTA (4 warps)
constexpr int kMaxTileI = 32;  // particles per static i tile (one ballot)
constexpr int kFold = 16;     // FP32 terms per thread between compensated folds

// ---------------------------------------------------------------- scalars
struct DevScalars {
    unsigned long long tmin[2];  // min(t_i + dt_i) as positive-double bit patterns
    double t_end;                // loop bound of hh_advance
    int32_t done;                // set once the next block time exceeds t_end
    int32_t err;                 // device-detected error (HH_* code), 0 = none
    alignas(8) uint32_t n_items;  // work items of this step
    uint32_t slot_ctr;           // partial-sum slots handed out this step (one 64-bit word with n_items)
    uint32_t work;               // force work-queue head
    int32_t part_len;            // shortest list part (a multiple of the staging chunk)
    int32_t work_item;           // target interactions per work item (0: every part is part_len long)
    int32_t work_split;          // > 0: work_item applies only to batched steps with this many active particles
    uint32_t slot_par[2];        // the same for the batched loop, by step parity
    int32_t n_act_last;          // active particles of the last corrected step
    int64_t n;                   // particles
    int64_t nj;                  // j entries
    int32_t n_tiles;             // static i tiles
    int32_t pad0;
    unsigned long long block_steps, particle_steps, interactions;
    unsigned long long list_steps;  // batched steps that predicted only their list parts' entries
    unsigned long long na_hist[32];  // active i tiles summed over block steps, by n_a - 1
    // block-step levels (level k <=> dt = 2^-k), kept by the batched loop
    int32_t lvl_cnt[32];          // particles per level
    unsigned long long t_cur_bits;  // latest block time (max t_i), positive-double bits
};

// Block-step control passed by value to every kernel of a step.
struct StepCtl {
    int32_t mode;       // 0: active = {t_i + dt_i == t_next}; 1: marked; 2: all particles
    int32_t slot_cur;   // tmin slot holding this step's time (mode 0)
    int32_t slot_next;  // tmin slot that receives the next step's time (mode 0)
    int32_t part_shift; // list parts of tile_j << part_shift entries (modes 1 and 2)
    double t_arg;       // step time for modes 1 and 2
};

// ---------------------------------------------------------------- records
// Predicted j record, plain form: (x, y, z, m), (vx, vy, vz, -) in FP64; the
// last word holds the mass's bits for the integer pair term (mass_bits).
struct __align__(32) RecF64 {
    double4 xm;
    double4 v;
};
// Predicted j record, mixed form: position as an unevaluated float pair
// x = hi + lo (|lo| <= ulp(hi)/2), velocity and mass in FP32.
struct __align__(16) RecMix {
    float4 hm;  // (x_hi, y_hi, z_hi, m)
    float4 lo;  // (x_lo, y_lo, z_lo, 0)
    float4 v;   // (vx, vy, vz, -): the last word holds the entry's index
};

// Mixed form: per j entry, the FP32 quantities the predictor needs,
// refreshed whenever the entry's FP64 state changes (upload, correction):
// position as a float pair, velocity, a/2 and jerk/6.
struct __align__(16) BaseMix {
    float4 hm;  // (x_hi, y_hi, z_hi, m)
    float4 lo;  // (x_lo, y_lo, z_lo, 0)
    float4 v;   // (vx, vy, vz, 0)
    float4 a2;  // a / 2
    float4 j6;  // jerk / 6
};

struct State {
    double *x, *v, *a, *jk;  // [3][cap_j]
    BaseMix *base;           // [cap_j] mixed form only (else nullptr)
    double *m, *t;           // [cap_j]
    double *dt;              // [cap_n]
    double *acc1, *jerk1, *pot1;  // [3][cap_n], [cap_n]: last force results
    int32_t *mark;           // [cap_n]
    int64_t cap_j, cap_n;
};

// One work item: a part of one i tile's interaction list.  It carries the
// tile record and the group's list range, so a worker reads one record before
// it can load particles and list indices.
struct __align__(16) WorkItem {
    int32_t tile;      // static tile index
    int32_t part_sim;  // list part | simulation << 16
    uint32_t mask;     // active lanes of the tile
    int32_t slot;      // first partial-sum slot of the tile's parts (0 with one part)
    int32_t p_begin, p_end;  // the tile's particles
    int32_t n_parts;         // parts of its list
    int32_t part_len;               // list entries per part of this tile (the last part may be shorter)
    int64_t gb, ge;    // the group's list [gb, ge) in idx
};

__device__ __forceinline__ WorkItem make_item(int tile, int part_sim, uint32_t mask, int slot, const int4 td, int64_t gb,
                                              int64_t ge, int part_len, int n_parts)
{
    WorkItem w;
    w.tile = tile;
    w.part_sim = part_sim;
    w.mask = mask;
    w.slot = slot;
    w.p_begin = td.x;
    w.p_end = td.y;
    w.n_parts = n_parts;
    w.part_len = part_len;
    w.gb = gb;
    w.ge = ge;
    return w;
}

// Programmatic dependent launch: a kernel launched so (launch_after) may have
// its blocks placed while the kernel before it in the stream still runs.
// after_previous: the first thing such a kernel does; returns when that kernel
// has ended and its writes are visible (at once in an ordinary launch), then
// lets the kernel behind it be placed in turn.  wait_previous: only the first, for
// kernels in front of launches that are not this library's.  (The four launches of an
// evaluation, behind a prediction: 24 particles of 16384 through host arrays
// 52.4 us before, 44.6 us; 4096 x 4096 mixed 48.7, now 43.0 us.)
__device__ __forceinline__ void wait_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void after_previous()
{
    wait_previous();
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// Launches a kernel that begins with after_previous() (hh_kernels.cuh), so that
// its start overlaps the end of the kernel before it in the stream (after =
// false: an ordinary launch).
template <typename... KArgs, typename... Args>
inline cudaError_t launch_after(void (*kernel)(KArgs...), dim3 grid, dim3 block, cudaStream_t st, bool after, const Args &...args)
{
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.stream = st;
    cfg.attrs = &attr;
    cfg.numAttrs = after ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, KArgs(args)...);
}

struct Lists {
    const int64_t *off;
    const int32_t *idx;
    const int4 *tiles;  // static i tiles: (p_begin, p_end, group, first part slot)
    WorkItem *items;    // this step's work
    void *partials;     // per (tile part, i slot) sums of split lists [part slots][32]
    int32_t *tile_cnt;  // arrivals per tile (reset by the last arriver)
    const int32_t *i_map;  // optional: i slot position -> j index (kMapI kernels only)
};

struct Params {
    double eps2, eta, eta_s, dt_min, dt_max;
    double unit;  // 1.0, as a value the compiler cannot see (pair_diff)
};

__device__ __forceinline__ double bits_to_time(unsigned long long b) { return __longlong_as_double((long long)b); }

// Time of this step; false if the step is a no-op (loop finished).
__device__ __forceinline__ bool step_time(const DevScalars *ds, const StepCtl &c, double *t)
{
    if (c.mode != 0) {
        *t = c.t_arg;
        return true;
    }
    if (*(volatile const int32_t *)&ds->done) return false;
    double tn = bits_to_time(*(volatile const unsigned long long *)&ds->tmin[c.slot_cur]);
    if (!(tn <= ds->t_end)) return false;
    *t = tn;
    return true;
}

__device__ __forceinline__ bool is_active(const State &s, const StepCtl &c, int64_t p, double tnow)
{
    if (c.mode == 0) return s.t[p] + s.dt[p] == tnow;
    if (c.mode == 1) return s.mark[p] != 0;
    return true;
}

// Largest power of two <= x for positive normal x: clear the mantissa.
__device__ __forceinline__ double pow2_floor(double x)
{
    return __longlong_as_double(__double_as_longlong(x) & (long long)0xFFF0000000000000ull);
}

// ------------------------------------------------------- tile selection
// Step 2 on the device: for each static i tile (<= 32 consecutive particles
// of one group) one warp ballots the tile's active particles; a tile with
// any active particle appends one work item per part of its group's list.
// Item order may vary between runs; results do not depend on it.
// Warp-collective: appends one work item per part of tile `tile`'s list.
// List entries per work item for a tile with n_a active particles: about
// `work` interactions per item (n_a x part length), never shorter than
// pj_min, a multiple of pj_min.  Items of equal cost keep the SMs evenly
// loaded; the length depends only on n_a, so results stay deterministic.
__device__ __forceinline__ int part_len_for(int n_a, int pj_min, int work)
{
    if (work <= 0) return pj_min;
    const int want = (work + n_a - 1) / n_a;
    const int k = (want + pj_min - 1) / pj_min;
    return (k < 1 ? 1 : k) * pj_min;
}

// (A list's length fits 32 bits: a 64-bit division would take a microsecond of
// a step's chain.)
__device__ __forceinline__ int parts_of(int64_t len, int pj)
{
    return len > 0 ? (int)(((uint32_t)len + (uint32_t)pj - 1u) / (uint32_t)pj) : 1;
}

// Warp-collective: appends one work item per part of tile `tile`'s list;
// item = (tile, part | sim << 16, active mask, first partial-sum slot, part
// length).  `work` is the equal-cost target of this step (0: parts of pj_min).
// slot_ctr = nullptr: the slots' counter is the word behind n_items (DevScalars).
__device__ __forceinline__ void append_tile_items(int tile, const int4 td, int64_t gb, int64_t ge, uint32_t mask,
                                                  int pj_min, int work, uint32_t *n_items, uint32_t *slot_ctr, WorkItem *items,
                                                  int sim, unsigned long long *na_hist, uint32_t *max_chunks = nullptr)
{
    const int lane = threadIdx.x & 31;
    const int64_t len = ge - gb;
    const int pj = part_len_for(__popc(mask), pj_min, work);
    const int n_parts = parts_of(len, pj);
    int base = 0, slot = 0;
    if (lane == 0) {
        if (slot_ctr) {
            base = (int)atomicAdd(n_items, (uint32_t)n_parts);
            slot = n_parts > 1 ? (int)atomicAdd(slot_ctr, (uint32_t)n_parts) : 0;
        } else {  // the slots are the word behind the items: one atomic for both (50001 of 200003 particles: 590 -> 580 us)
            const unsigned long long both = atomicAdd(reinterpret_cast<unsigned long long *>(n_items),
                                                      (unsigned long long)(uint32_t)n_parts * (n_parts > 1 ? 0x100000001ull : 1ull));
            base = (int)(uint32_t)both;
            slot = n_parts > 1 ? (int)(both >> 32) : 0;
        }
        atomicAdd(&na_hist[__popc(mask) - 1], 1ull);
        // (with max_chunks: the longest part so far, in 32-entry chunks)
        if (max_chunks) atomicMax(max_chunks, (uint32_t)((min((int64_t)pj, len) + 31) / 32));
    }
    base = __shfl_sync(0xffffffffu, base, 0);
    slot = __shfl_sync(0xffffffffu, slot, 0);
    for (int q = lane; q < n_parts; q += 32) items[base + q] = make_item(tile, q | (sim << 16), mask, slot, td, gb, ge, pj, n_parts);
}

__device__ __forceinline__ void select_tiles(const State &s, const Lists &L, DevScalars *ds, const StepCtl &c,
                                             double tnow)
{
    const int lane = threadIdx.x & 31;
    const int64_t warp0 = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const int n_tiles = ds->n_tiles;
    // (this loop does not count a step's active particles first, so a
    // work_item limited to large steps, work_split > 0, is not used here)
    const int work = ds->work_split > 0 ? 0 : ds->work_item;
    const int pj = work > 0 ? ds->part_len : ds->part_len << c.part_shift;
    for (int64_t tile = warp0; tile < n_tiles; tile += nwarps) {
        const int4 td = L.tiles[tile];
        const int64_t p = td.x + lane;
        const bool act = (p < td.y) && is_active(s, c, p, tnow);
        const uint32_t mask = __ballot_sync(0xffffffffu, act);
        if (mask == 0u) continue;
        append_tile_items((int)tile, td, L.off[td.z], L.off[td.z + 1], mask, pj, work, &ds->n_items, nullptr, L.items,
                          0, ds->na_hist);
    }
}

static __global__ void k_select(State s, Lists L, DevScalars *ds, StepCtl c)
{
    after_previous();
    double tnow;
    if (c.mode == 1 && *(volatile const int32_t *)&ds->err) return;  // (k_mark_begin found a bad index)
    if (!step_time(ds, c, &tnow)) return;
    select_tiles(s, L, ds, c, tnow);
}

// -------------------------------------------------------------- predictor
// x + v D + a D^2/2 + jk D^3/6 and v + a D + jk D^2/2, in Horner form.
// Taylor predictor of one component over D (Section 2, step 3).
__device__ __forceinline__ void predict_xv(double D, double x, double v, double a, double j, double &xp, double &vp)
{
    const double h = 0.5 * D, th = D * (1.0 / 3.0);
    xp = x + D * (v + h * (a + th * j));
    vp = v + D * (a + h * j);
}

template <typename Rec>
__device__ __forceinline__ void store_rec(Rec *out, int64_t e, const double xp[3], const double vp[3], double m);

template <>
__device__ __forceinline__ void store_rec<RecF64>(RecF64 *out, int64_t e, const double xp[3], const double vp[3],
                                                 double m)
{
    RecF64 r;
    r.xm = make_double4(xp[0], xp[1], xp[2], m);
    r.v = make_double4(vp[0], vp[1], vp[2], __longlong_as_double((long long)mass_bits(m)));
    out[e] = r;
}

template <>
__device__ __forceinline__ void store_rec<RecMix>(RecMix *out, int64_t e, const double xp[3], const double vp[3],
                                                 double m)
{
    float hi[3], lo[3];
#pragma unroll
    for (int d = 0; d < 3; d++) {
        hi[d] = __double2float_rn(xp[d]);
        lo[d] = __double2float_rn(xp[d] - (double)hi[d]);
    }
    RecMix r;
    r.hm = make_float4(hi[0], hi[1], hi[2], __double2float_rn(m));
    r.lo = make_float4(lo[0], lo[1], lo[2], 0.f);
    r.v = make_float4(__double2float_rn(vp[0]), __double2float_rn(vp[1]), __double2float_rn(vp[2]),
                      __int_as_float((int)e));
    out[e] = r;
}

// (float)x and (float)(x - (double)(float)x), both to nearest, on the bits: a
// conversion between FP64 and FP32 takes 64 cycles of the FP64 pipe, and the
// corrector refreshes its particles' base records with ten of them.  Numbers
// outside [2^-70, 2^127) take the conversions.
__device__ __forceinline__ uint32_t f32_rn_bits(uint32_t hi, uint32_t lo, int &rem)
{
    const uint32_t t = __funnelshift_l(lo, hi & 0x7fffffffu, 3) - (896u << 23);  // truncated
    const uint32_t r = lo & 0x1fffffffu;
    const uint32_t up = (r + (t & 1u)) > 0x10000000u ? 1u : 0u;
    rem = (int)r - (int)(up << 29);
    return t + up;
}
__device__ __forceinline__ bool f32_in_range(uint32_t hi)
{
    return ((hi >> 20) & 0x7ffu) - (1023u - 70u) < 70u + 127u;
}
__device__ __forceinline__ float f32_rn(double x)
{
    const uint32_t hi = f64_hi(x);
    if (!f32_in_range(hi)) return __double2float_rn(x);
    int rem;
    return __uint_as_float(f32_rn_bits(hi, f64_lo(x), rem) | (hi & 0x80000000u));
}
__device__ __forceinline__ void f32_pair(double x, float &h, float &l)
{
    const uint32_t hi = f64_hi(x);
    if (!f32_in_range(hi)) {
        h = __double2float_rn(x);
        l = __double2float_rn(x - (double)h);
        return;
    }
    int rem;
    h = __uint_as_float(f32_rn_bits(hi, f64_lo(x), rem) | (hi & 0x80000000u));
    // rem 2^(e - 52), |rem| <= 2^28: one rounding, then an exact scaling
    const float scale = __uint_as_float((((hi >> 20) & 0x7ffu) - 1023u - 52u + 127u) << 23 | (hi & 0x80000000u));
    l = __int2float_rn(rem) * scale;
}

// FP32 copy of entry e's FP64 state for the mixed predictor, one component
// (d = 0, 1, 2) from the values x, v, a, jk of that component; the mass m goes
// with component 0.
__device__ __forceinline__ void refresh_base_values(const State &s, int64_t e, int d, double x, double v, double a,
                                                    double jk, double m)
{
    float hi, lo;
    f32_pair(x, hi, lo);
    const float vf = f32_rn(v);
    const float a2 = 0.5f * f32_rn(a);
    const float j6 = f32_rn(jk) * (1.0f / 6.0f);
    float *b = reinterpret_cast<float *>(&s.base[e]);  // hm, lo, v, a2, j6: float4 each
    b[0 + d] = hi;
    b[4 + d] = lo;
    b[8 + d] = vf;
    b[12 + d] = a2;
    b[16 + d] = j6;
    if (d == 0) {
        b[3] = f32_rn(m);
        b[7] = b[11] = b[15] = b[19] = 0.f;
    }
}

// The same from the state arrays.
__device__ __forceinline__ void refresh_base_component(const State &s, int64_t e, int d)
{
    refresh_base_values(s, e, d, s.x[d * s.cap_j + e], s.v[d * s.cap_j + e], s.a[d * s.cap_j + e],
                        s.jk[d * s.cap_j + e], d == 0 ? s.m[e] : 0.0);
}

// All components by one thread: five 16-byte stores instead of twenty of four
// bytes (374377 entries: 33 us before, 17 us now).
__device__ __forceinline__ void refresh_base(const State &s, int64_t e)
{
    float hi[3], lo[3], v[3], a2[3], j6[3];
#pragma unroll
    for (int d = 0; d < 3; d++) {
        f32_pair(s.x[d * s.cap_j + e], hi[d], lo[d]);
        v[d] = f32_rn(s.v[d * s.cap_j + e]);
        a2[d] = 0.5f * f32_rn(s.a[d * s.cap_j + e]);
        j6[d] = f32_rn(s.jk[d * s.cap_j + e]) * (1.0f / 6.0f);
    }
    float4 *b = reinterpret_cast<float4 *>(&s.base[e]);  // hm, lo, v, a2, j6
    b[0] = make_float4(hi[0], hi[1], hi[2], f32_rn(s.m[e]));
    b[1] = make_float4(lo[0], lo[1], lo[2], 0.f);
    b[2] = make_float4(v[0], v[1], v[2], 0.f);
    b[3] = make_float4(a2[0], a2[1], a2[2], 0.f);
    b[4] = make_float4(j6[0], j6[1], j6[2], 0.f);
}

// Mixed predictor: the FP64 base position (as a float pair) plus an FP32
// increment D (v + D (a/2 + D jerk/6)), added with TwoSum; v + D (a + D jerk/2)
// in FP32.  D = t - t_e is exact in FP32 (a multiple of dt_min below dt_tree).
__device__ __forceinline__ RecMix mix_from_base(const BaseMix &b, float D, int64_t e)
{
    const float hx[3] = {b.hm.x, b.hm.y, b.hm.z}, lx[3] = {b.lo.x, b.lo.y, b.lo.z};
    const float vv[3] = {b.v.x, b.v.y, b.v.z}, aa[3] = {b.a2.x, b.a2.y, b.a2.z}, jj[3] = {b.j6.x, b.j6.y, b.j6.z};
    float ho[3], lo[3], vo[3];
#pragma unroll
    for (int d = 0; d < 3; d++) {
        const float dx = D * fmaf(D, fmaf(D, jj[d], aa[d]), vv[d]);
        const float sum = __fadd_rn(hx[d], dx);
        const float bb = __fsub_rn(sum, hx[d]);
        const float err = __fadd_rn(__fsub_rn(hx[d], __fsub_rn(sum, bb)), __fsub_rn(dx, bb));
        ho[d] = sum;
        lo[d] = __fadd_rn(lx[d], err);
        vo[d] = fmaf(D, fmaf(D, 3.f * jj[d], 2.f * aa[d]), vv[d]);
    }
    RecMix r;
    r.hm = make_float4(ho[0], ho[1], ho[2], b.hm.w);
    r.lo = make_float4(lo[0], lo[1], lo[2], 0.f);
    r.v = make_float4(vo[0], vo[1], vo[2], __int_as_float((int)e));
    return r;
}

// Inputs of one entry's prediction, loaded ahead of its arithmetic so that a
// thread can keep several entries' loads in flight (pred_load, then
// pred_store).
template <typename Rec>
struct PredIn;
template <>
struct PredIn<RecF64> {
    double t, m, x[3], v[3], a[3], j[3];
};
template <>
struct PredIn<RecMix> {
    double t;
    BaseMix b;
};

template <typename Rec>
__device__ __forceinline__ void pred_load(const State &s, int64_t e, PredIn<Rec> &in);
template <>
__device__ __forceinline__ void pred_load<RecF64>(const State &s, int64_t e, PredIn<RecF64> &in)
{
    in.t = s.t[e];
    in.m = s.m[e];
#pragma unroll
    for (int d = 0; d < 3; d++) {
        in.x[d] = s.x[d * s.cap_j + e];
        in.v[d] = s.v[d * s.cap_j + e];
        in.a[d] = s.a[d * s.cap_j + e];
        in.j[d] = s.jk[d * s.cap_j + e];
    }
}
template <>
__device__ __forceinline__ void pred_load<RecMix>(const State &s, int64_t e, PredIn<RecMix> &in)
{
    in.t = s.t[e];
    in.b = s.base[e];
}

template <typename Rec>
__device__ __forceinline__ void pred_store(const PredIn<Rec> &in, Rec *rec, int64_t e, double tnow);
template <>
__device__ __forceinline__ void pred_store<RecF64>(const PredIn<RecF64> &in, RecF64 *rec, int64_t e, double tnow)
{
    const double D = tnow - in.t;
    double xp[3], vp[3];
#pragma unroll
    for (int d = 0; d < 3; d++) predict_xv(D, in.x[d], in.v[d], in.a[d], in.j[d], xp[d], vp[d]);
    store_rec<RecF64>(rec, e, xp, vp, in.m);
}
template <>
__device__ __forceinline__ void pred_store<RecMix>(const PredIn<RecMix> &in, RecMix *rec, int64_t e, double tnow)
{
    rec[e] = mix_from_base(in.b, __double2float_rn(tnow - in.t), e);
}

// Predicted record of entry e at tnow, in the form's own arithmetic.
template <typename Rec>
__device__ __forceinline__ void predict_entry(const State &s, Rec *rec, int64_t e, double tnow)
{
    PredIn<Rec> in;
    pred_load<Rec>(s, e, in);
    pred_store<Rec>(in, rec, e, tnow);
}

template <typename Rec>
__global__ void k_predict(State s, Rec *rec, Lists L, DevScalars *ds, StepCtl c)
{
    after_previous();
    double tnow;
    if (!step_time(ds, c, &tnow)) {
        if (c.mode == 0 && blockIdx.x == 0 && threadIdx.x == 0) ds->done = 1;
        return;
    }
    if (c.mode == 0 && blockIdx.x == 0 && threadIdx.x == 0) {
        ds->tmin[c.slot_next] = 0x7FF0000000000000ull;  // +inf
        ds->work = 0u;
        ds->n_act_last = 0;
        ds->block_steps += 1ull;
    }

    const int64_t nj = ds->nj;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < nj; e += (int64_t)gridDim.x * blockDim.x)
        predict_entry<Rec>(s, rec, e, tnow);
    if (c.mode == 0) select_tiles(s, L, ds, c, tnow);
}

// ------------------------------------------------------ pairwise kernels
// Plummer-softened pair term (Makino & Aarseth 1992): r = x_j - x_i,
// w = v_j - v_i, s = r^2 + eps^2; a += m r s^-3/2;
// jerk += m (w s^-3/2 - 3 (r.w) r s^-5/2); pot -= m s^-1/2.

struct AccF64 {
    double ax, ay, az, jx, jy, jz, p;
    __device__ void zero() { ax = ay = az = jx = jy = jz = p = 0.0; }
};

struct IF64 {
    double x, y, z, vx, vy, vz;
};

__device__ __forceinline__ void load_i(const RecF64 *rec, int64_t i, IF64 &o)
{
    const RecF64 r = rec[i];
    o.x = r.xm.x; o.y = r.xm.y; o.z = r.xm.z;
    o.vx = r.v.x; o.vy = r.v.y; o.vz = r.v.z;
}

__device__ __forceinline__ void interact(const IF64 &I, const RecF64 &J, bool self, double eps2, AccF64 &A)
{
    const double dx = J.xm.x - I.x, dy = J.xm.y - I.y, dz = J.xm.z - I.z;
    const double wx = J.v.x - I.vx, wy = J.v.y - I.vy, wz = J.v.z - I.vz;
    double r2 = fma(dx, dx, fma(dy, dy, fma(dz, dz, eps2)));
    r2 = self ? 1.0 : r2;
    const double mj = self ? 0.0 : J.xm.w;
    const double rw = fma(dx, wx, fma(dy, wy, dz * wz));
    const double rinv = rsqrt(r2);
    const double rinv2 = rinv * rinv;
    const double mr = mj * rinv;
    const double mr3 = mr * rinv2;
    const double al = 3.0 * rw * rinv2;
    A.p += mr;
    A.ax = fma(mr3, dx, A.ax);
    A.ay = fma(mr3, dy, A.ay);
    A.az = fma(mr3, dz, A.az);
    A.jx = fma(mr3, fma(-al, dx, wx), A.jx);
    A.jy = fma(mr3, fma(-al, dy, wy), A.jy);
    A.jz = fma(mr3, fma(-al, dz, wz), A.jz);
}

// Differences as fused multiply-adds with 1: an FP64 add issues in 76 cycles
// here, a fused multiply-add in 64.
__device__ __forceinline__ void interact_int(const IF64 &I, const RecF64 &J, bool self, const Soft64 &eps, double unit,
                                             int smin, AccI64 &A)
{
    double d[3], w[3];
    d[0] = fma(J.xm.x, unit, -I.x);
    d[1] = fma(J.xm.y, unit, -I.y);
    d[2] = fma(J.xm.z, unit, -I.z);
    w[0] = fma(J.v.x, unit, -I.vx);
    w[1] = fma(J.v.y, unit, -I.vy);
    w[2] = fma(J.v.z, unit, -I.vz);
    pair_add(d, w, J.xm.w, (uint64_t)__double_as_longlong(J.v.w), self, eps, smin, A);
}

// Mixed: chunk partials in FP32, folded into (hi, lo) pairs after each
// staged chunk with Knuth's TwoSum, so that the running sum is carried to
// about 2^-48 relative while the inner loop stays plain FP32.
struct __align__(8) F2 {
    float h, l;
};

__device__ __forceinline__ void two_sum_into(F2 &acc, float b)
{
    const float s = __fadd_rn(acc.h, b);
    const float bb = __fsub_rn(s, acc.h);
    const float err = __fadd_rn(__fsub_rn(acc.h, __fsub_rn(s, bb)), __fsub_rn(b, bb));
    acc.h = s;
    acc.l = __fadd_rn(acc.l, err);
}

// (h1, l1) + (h2, l2) with one TwoSum on the heads and a renormalising
// Fast2Sum (Dekker): deterministic for a fixed operand order.
__device__ __forceinline__ F2 f2_add(F2 a, F2 b)
{
    const float s = __fadd_rn(a.h, b.h);
    const float bb = __fsub_rn(s, a.h);
    float e = __fadd_rn(__fsub_rn(a.h, __fsub_rn(s, bb)), __fsub_rn(b.h, bb));
    e = __fadd_rn(e, __fadd_rn(a.l, b.l));
    F2 r;
    r.h = __fadd_rn(s, e);
    r.l = __fsub_rn(e, __fsub_rn(r.h, s));
    return r;
}

struct AccMix {
    float2 axy, jxy, azjz;  // current chunk: (ax, ay), (jx, jy), (az, jz)
    float p;
    F2 Ax, Ay, Az, Jx, Jy, Jz, P;     // running compensated sums
    __device__ void zero()
    {
        axy = jxy = azjz = make_float2(0.f, 0.f);
        p = 0.f;
        Ax = Ay = Az = Jx = Jy = Jz = P = F2{0.f, 0.f};
    }
    __device__ void fold()
    {
        two_sum_into(Ax, axy.x); two_sum_into(Ay, axy.y); two_sum_into(Az, azjz.x);
        two_sum_into(Jx, jxy.x); two_sum_into(Jy, jxy.y); two_sum_into(Jz, azjz.y);
        two_sum_into(P, p);
        axy = jxy = azjz = make_float2(0.f, 0.f);
        p = 0.f;
    }
};

// The i particle, negated (differences are sums then), x and y together.
struct IMix {
    float2 h, l, v;
    float hz, lz, vz;
};

__device__ __forceinline__ void load_i(const RecMix *rec, int64_t i, IMix &o)
{
    const RecMix r = rec[i];
    o.h = make_float2(-r.hm.x, -r.hm.y);
    o.l = make_float2(-r.lo.x, -r.lo.y);
    o.v = make_float2(-r.v.x, -r.v.y);
    o.hz = -r.hm.z;
    o.lz = -r.lo.z;
    o.vz = -r.v.z;
}

// 1/sqrt estimate.  With kNormal (the softening, and so every r2, is a normal
// number) without the scaling of subnormal arguments: the same bits, three
// instructions less.
template <bool kNormal>
__device__ __forceinline__ float rsqrt_est(float x)
{
    if (!kNormal) return rsqrtf(x);
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Bound by instruction issue (60 a pair, 78% of the issue slots at 6 warps a
// sub-partition), so the x and y components, and the z components of the two
// sums, go two to an instruction (packed FP32: each half rounds as the single
// instruction does, so the sums keep their bits), the self test reads the index
// that comes with the record, and the estimate skips the subnormal scaling: 46
// instructions, 82 -> 64 cycles a warp and pair (the FP32 pipe's own time is
// about 45).  Two pairs at a time in packed scalars (39 instructions) measured 3%
// more with 6 warps a sub-partition and is left out.
template <bool kNormal>
__device__ __forceinline__ void interact(const IMix &I, const RecMix &J, bool self, float eps2, AccMix &A)
{
    // i-j difference of the float pairs: (hi_j - hi_i) + (lo_j - lo_i)
    const float2 dxy = __fadd2_rn(__fadd2_rn(make_float2(J.hm.x, J.hm.y), I.h),
                                  __fadd2_rn(make_float2(J.lo.x, J.lo.y), I.l));
    const float dz = __fadd_rn(__fadd_rn(J.hm.z, I.hz), __fadd_rn(J.lo.z, I.lz));
    const float2 wxy = __fadd2_rn(make_float2(J.v.x, J.v.y), I.v);
    const float wz = __fadd_rn(J.v.z, I.vz);
    float r2 = fmaf(dxy.x, dxy.x, fmaf(dxy.y, dxy.y, fmaf(dz, dz, eps2)));
    r2 = self ? 1.f : r2;
    const float mj = self ? 0.f : J.hm.w;
    const float rw = fmaf(dxy.x, wxy.x, fmaf(dxy.y, wxy.y, dz * wz));
    // 1/sqrt: hardware estimate, then one Newton-Raphson step
    // y <- y + (y/2) h, h = 1 - r2 y^2, with the residual formed exactly
    // (r2 y = p + e by an FMA) so the step lands within ~1/2 ulp.
    const float y0 = rsqrt_est<kNormal>(r2);
    const float pr = r2 * y0;
    const float er = fmaf(r2, y0, -pr);
    const float hres = fmaf(-er, y0, fmaf(-pr, y0, 1.f));
    const float rinv = fmaf(0.5f * y0, hres, y0);
    const float rinv2 = rinv * rinv;
    const float mr = mj * rinv;
    const float mr3 = mr * rinv2;
    const float al = 3.f * rw * rinv2;
    const float2 m2 = make_float2(mr3, mr3);
    const float2 ixy = __ffma2_rn(make_float2(-al, -al), dxy, wxy);
    const float iz = fmaf(-al, dz, wz);
    A.p += mr;
    A.axy = __ffma2_rn(m2, dxy, A.axy);
    A.jxy = __ffma2_rn(m2, ixy, A.jxy);
    A.azjz = __ffma2_rn(m2, make_float2(dz, iz), A.azjz);
}

// ---------------------------------------------- cross-slice reductions
__device__ __forceinline__ F2 f2_shfl(F2 a, int off)
{
    F2 b;
    b.h = __shfl_xor_sync(0xffffffffu, a.h, off);
    b.l = __shfl_xor_sync(0xffffffffu, a.l, off);
    // operand order by lane bit keeps both partners bitwise identical
    return ((threadIdx.x & off) == 0) ? f2_add(a, b) : f2_add(b, a);
}

__device__ __forceinline__ void acc_shfl_add(AccMix &A, int off)
{
    A.Ax = f2_shfl(A.Ax, off); A.Ay = f2_shfl(A.Ay, off); A.Az = f2_shfl(A.Az, off);
    A.Jx = f2_shfl(A.Jx, off); A.Jy = f2_shfl(A.Jy, off); A.Jz = f2_shfl(A.Jz, off);
    A.P = f2_shfl(A.P, off);
}

// Adds the partner's sums (lane + delta) into this lane's where `take`; every
// lane takes part in the shuffles.  The receiving lane's sums come first, so
// the order of every addition is fixed.
__device__ __forceinline__ F2 f2_shfl_down_take(F2 a, int delta, bool take)
{
    F2 o;
    o.h = __shfl_down_sync(0xffffffffu, a.h, delta);
    o.l = __shfl_down_sync(0xffffffffu, a.l, delta);
    return take ? f2_add(a, o) : a;
}

__device__ __forceinline__ void acc_shfl_down_add(AccMix &A, int delta, bool take)
{
    A.Ax = f2_shfl_down_take(A.Ax, delta, take);
    A.Ay = f2_shfl_down_take(A.Ay, delta, take);
    A.Az = f2_shfl_down_take(A.Az, delta, take);
    A.Jx = f2_shfl_down_take(A.Jx, delta, take);
    A.Jy = f2_shfl_down_take(A.Jy, delta, take);
    A.Jz = f2_shfl_down_take(A.Jz, delta, take);
    A.P = f2_shfl_down_take(A.P, delta, take);
}

struct RedF64 {
    double v[7];
};
struct RedMix {
    F2 v[7];
};

__device__ __forceinline__ void to_red(const AccF64 &A, RedF64 &r)
{
    r.v[0] = A.ax; r.v[1] = A.ay; r.v[2] = A.az; r.v[3] = A.jx; r.v[4] = A.jy; r.v[5] = A.jz; r.v[6] = A.p;
}
__device__ __forceinline__ void to_red(const AccI64 &A, RedF64 &r)
{
#pragma unroll
    for (int k = 0; k < 3; k++) {
        r.v[k] = sum_get(A.a.u[k], A.a.o[k], A.a.e);
        r.v[3 + k] = sum_get(A.j.u[k], A.j.o[k], A.j.e);
    }
    r.v[6] = sum_get(A.p.u[0], A.p.o[0], A.p.e);
}
__device__ __forceinline__ void to_red(const AccMix &A, RedMix &r)
{
    r.v[0] = A.Ax; r.v[1] = A.Ay; r.v[2] = A.Az; r.v[3] = A.Jx; r.v[4] = A.Jy; r.v[5] = A.Jz; r.v[6] = A.P;
}
// partial sums written by other CTAs are read through L2 (bypassing L1)
// One component of a reduction record (double, or an FP32 pair).
__device__ __forceinline__ double shfl_down_e(double v, int d) { return __shfl_down_sync(0xffffffffu, v, d); }
__device__ __forceinline__ F2 shfl_down_e(const F2 &v, int d)
{
    F2 r;
    r.h = __shfl_down_sync(0xffffffffu, v.h, d);
    r.l = __shfl_down_sync(0xffffffffu, v.l, d);
    return r;
}
__device__ __forceinline__ void comp_add(double &a, double b) { a += b; }
__device__ __forceinline__ void comp_add(F2 &a, const F2 &b) { a = f2_add(a, b); }
__device__ __forceinline__ double comp_get(double a) { return a; }
__device__ __forceinline__ double comp_get(const F2 &a) { return (double)a.h + (double)a.l; }
__device__ __forceinline__ double ld_comp_cg(const double *p) { return __ldcg(p); }
__device__ __forceinline__ F2 ld_comp_cg(const F2 *p)
{
    const float2 u = __ldcg(reinterpret_cast<const float2 *>(p));
    return F2{u.x, u.y};
}

template <typename Rec>
struct Traits;
template <>
struct Traits<RecF64> {
    using I = IF64;
    using Acc = AccI64;
    using Red = RedF64;
    using Eps = double;
};
template <>
struct Traits<RecMix> {
    using I = IMix;
    using Acc = AccMix;
    using Red = RedMix;
    using Eps = float;
};

__device__ __forceinline__ void fold_chunk(AccMix &A) { A.fold(); }

// ------------------------------------------------------------ list force
// One 128-thread group (4 warps) per work item = (tile, part of its group's
// list).  With n_a active particles in the tile each warp holds floor(32 /
// n_a) j slices of n_a lanes (lane = i slot + n_a * slice; leftover lanes
// idle), and the slices stride through each staged chunk of the part.  (Plain
// form: the slices lie across the whole group, floor(128 / n_a) of them.)
// Slices are summed in a fixed order (shuffles, then warps).  A list split
// into several parts leaves per-part sums in the partials buffer; the group
// that finishes a tile's last part (acquire-release arrival counter: no
// waiting) adds the parts in part order.  So each particle's result depends
// only on its list, its tile's active count and the part length (which follows
// the configuration and, in the plain form's large evaluations and steps, the
// number of active particles), never on scheduling.
// Asynchronous global -> shared copies (16 B each) for chunk staging,
// cached in L1: the 16-byte pieces of one record, and the records of
// neighbouring list entries (consecutive particles of a leaf, sibling
// cells), share sectors, which L1 then serves instead of L2.  Measured on
// real tree lists (N = 65536, staging alone) at 1.0e11 records/s against
// 5.9e10 through L2 only.  The records are rewritten every block step, but
// always before a grid barrier or a kernel boundary that orders them before
// these (weak) reads, as for any plain load.
__device__ __forceinline__ void cp_async16(void *smem, const void *gmem)
{
    const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(sa), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

template <typename Rec>
__device__ __forceinline__ void cp_async_rec(Rec *dst, const Rec *src)
{
    static_assert(sizeof(Rec) % 16 == 0, "records are whole 16-byte pieces");
#pragma unroll
    for (int q = 0; q < (int)(sizeof(Rec) / 16); q++)
        cp_async16(reinterpret_cast<char *>(dst) + 16 * q, reinterpret_cast<const char *>(src) + 16 * q);
}

// Staged list chunks per 128-thread group: one is summed while kStages - 1
// are in flight.  (Three stages measured no faster in the tree loop and up to
// 18% slower for short list parts: the deeper prologue adds latency to every
// part, and parts are only a few chunks long.)
constexpr int kStages = 2;

template <typename Rec, int TJ>
struct ForceSmem {
    Rec rec[kStages][TJ];  // ring of staged list chunks
    int32_t idx[kStages][std::is_same<Rec, RecF64>::value ? TJ : 1];  // plain form (mixed: in the records)
    typename Traits<Rec>::Red red[kThreads / 32][kMaxTileI];
    int item;
    int last;
    double tn[kThreads / 32];  // per-warp minimum of t + dt after the corrector
    int lv[kMaxTileI];         // new step level of each corrected particle, by active index
    typename Traits<Rec>::I iv[std::is_same<Rec, RecF64>::value ? kMaxTileI : 1];  // plain form: the item's active particles
    int pidx[kMaxTileI];       // its active particles
    double fin[kMaxTileI][7];  // the completed tile's new acc, jerk, pot by active index (for its corrector)
};

// GPU-scope acquire / release operations (PTX memory model): an
// acquire-release arrival on a counter sees every earlier arrival's writes and
// passes its own on, without full fences.
__device__ __forceinline__ unsigned int atom_add_acq_rel_gpu(unsigned int *p, unsigned int v)
{
    unsigned int old;
    asm volatile("atom.add.acq_rel.gpu.global.u32 %0, [%1], %2;" : "=r"(old) : "l"(p), "r"(v) : "memory");
    return old;
}
__device__ __forceinline__ unsigned int ld_acquire_gpu(const unsigned int *p)
{
    unsigned int v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void red_release_max_gpu(unsigned int *p, unsigned int v)
{
    asm volatile("red.release.gpu.global.max.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// Barrier over the 128 threads working on one item: the whole CTA
// (bar_id 0) or one of several 128-thread worker groups of a larger CTA
// (named barrier bar_id = 1 + group).
__device__ __forceinline__ void group_sync(int bar_id)
{
    if (bar_id == 0) __syncthreads();
    else asm volatile("bar.sync %0, %1;" ::"r"(bar_id), "r"(kThreads) : "memory");
}

// The same, returning whether `pred` holds in any thread of the group.
__device__ __forceinline__ bool group_any(int bar_id, bool pred)
{
    if (bar_id == 0) return __syncthreads_or(pred) != 0;
    int r;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\tsetp.ne.s32 p, %1, 0;\n\tbarrier.cta.red.or.pred q, %2, %3, p;\n\t"
        "selp.s32 %0, 1, 0, q;\n\t}"
        : "=r"(r)
        : "r"((int)pred), "r"(bar_id), "r"(kThreads)
        : "memory");
    return r != 0;
}

// A thread's sums over its entries of a list part in FP64 arithmetic (jslice,
// jslice + S, ... of each chunk of tj entries), straight from the records: the
// parts that the integer pair term does not take.
static __device__ __noinline__ void part_sums_f64(const RecF64 *__restrict__ rec, const int32_t *idx, int64_t len, int tj,
                                                  int jslice, int S, int64_t pi, const IF64 &I, double eps2, RedF64 &out)
{
    AccF64 A;
    A.zero();
    for (int64_t c = 0; c < len; c += tj)
        for (int64_t e = c + jslice; e < min(len, c + (int64_t)tj); e += S) {
            const int32_t j = idx[e];
            interact(I, rec[j], (int64_t)j == pi, eps2, A);
        }
    to_red(A, out);
}

// The same with the integers' scalars and FP64 components (20 FP64 operations a pair
// instead of 34): the parts that the integers take but for a component that is too
// small for them.
static __device__ __noinline__ void part_sums_thin(const RecF64 *__restrict__ rec, const int32_t *idx, int64_t len, int tj,
                                                   int jslice, int S, int64_t pi, const IF64 &I, double eps2, RedF64 &out)
{
    AccF64 A;
    A.zero();
    const Soft64 soft = soft_of(eps2);
    for (int64_t c = 0; c < len; c += tj)
        for (int64_t e = c + jslice; e < min(len, c + (int64_t)tj); e += S) {
            const int32_t j = idx[e];
            const RecF64 J = rec[j];
            if ((int64_t)j == pi) continue;
            const double d[3] = {J.xm.x - I.x, J.xm.y - I.y, J.xm.z - I.z};
            const double wx = J.v.x - I.vx, wy = J.v.y - I.vy, wz = J.v.z - I.vz;
            double mr, u, z3;
            pair_scalars_f64(d, J.xm.w, (uint64_t)__double_as_longlong(J.v.w), soft, mr, u, z3);
            const double al = fma(d[0], wx, fma(d[1], wy, d[2] * wz)) * z3;
            A.p += mr;
            A.ax = fma(u, d[0], A.ax);
            A.ay = fma(u, d[1], A.ay);
            A.az = fma(u, d[2], A.az);
            A.jx = fma(u, fma(-al, d[0], wx), A.jx);
            A.jy = fma(u, fma(-al, d[1], wy), A.jy);
            A.jz = fma(u, fma(-al, d[2], wz), A.jz);
        }
    to_red(A, out);
}

// A slice of a few terms often is thin where its particle is not: maxima over the
// lanes of a warp that work on the same particle (thread = particle + I x slice;
// in lanes 0 to I - 1), then over the warps.
__device__ __forceinline__ void warp_span(Span64 &s, int I)
{
    for (int step = I; step < 32; step <<= 1)
#pragma unroll
        for (int k = 0; k < 3; k++) s.k[k] = addmax_u16x2(__shfl_down_sync(0xffffffffu, s.k[k], step), 0u, s.k[k]);
}

// Whether one of the item's particles is thin, from the warps' spans.  buf: a span
// per warp and particle.
__device__ __forceinline__ bool thin_particles(Span64 s, Span64 *buf, int islot, int I, int tid, int bar_id)
{
    if ((tid & 31) < I) buf[(tid & ~31) + islot] = s;
    group_sync(bar_id);
    if (tid < I)
        for (int w = 32; w < kThreads; w += 32)
#pragma unroll
            for (int k = 0; k < 3; k++) s.k[k] = addmax_u16x2(buf[w + tid].k[k], 0u, s.k[k]);
    return group_any(bar_id, tid < I && thin(s));
}

// a / b for 0 <= a < 2^14, 0 < b <= 2^8: one reciprocal and a product instead of
// an integer division's chain, of which a part's path has five ((a + 1/2) / b
// is at least 1 / (2 b) from every integer, and the quotient's error, two units of
// FP32, at most (a + 1/2) / b 2^-22: less as long as a < 2^20).
__device__ __forceinline__ int small_div(int a, int b) { return (int)__fdividef((float)a + 0.5f, (float)b); }

// item = (tile, part | sim << 16, active mask, parts of the tile); tid is
// the thread's index in its 128-thread group.  Returns true (in every thread
// of the group) for the item that wrote the tile's final forces.
template <typename Rec, int TJ, bool kMapI>
__device__ __forceinline__ bool force_item(const State &s, const Rec *__restrict__ rec, const Lists &L,
                                           typename Traits<Rec>::Eps eps2, double unit, const WorkItem &it,
                                           ForceSmem<Rec, TJ> &sm, unsigned long long &n_int, const int tid,
                                           const int bar_id)
{
    using T = Traits<Rec>;
    using Red = typename T::Red;
    const int lane = tid & 31, warp = tid >> 5;
    Red *partials = reinterpret_cast<Red *>(L.partials);
    const int p0 = it.p_begin;
    const uint32_t mask = it.mask;
    const int n_a = __popc(mask);
    const int pj = it.part_len;
    const int part = it.part_sim & 0xFFFF, slot0 = it.slot;

    // Lane mapping.  Mixed form: every warp holds K = floor(32 / n_a) j slices
    // of n_a lanes (lane = i slot + n_a * slice); the 32 - K n_a leftover lanes
    // idle.  So no lane is spent on a missing particle (rounding n_a up to a
    // power of two left up to half the lanes idle).  Plain form: the slices lie
    // across the group's 128 threads (its slice sums go through shared memory,
    // so a slice may straddle two warps): 7 slices of 18 particles where the
    // warps alone hold 4.  Tree groups of n_crit 64 hold 18 particles on
    // average: 56% of the lanes at work before, 98% now, and an evaluation of
    // N = 65536 went from 3.95 to 3.53 ms.
    constexpr bool kPlain = std::is_same<Rec, RecF64>::value;
    const int I = n_a;
    const int K = small_div(kPlain ? kThreads : 32, I);  // slices of the group (plain), of each warp (mixed)
    const int kslice = small_div(kPlain ? tid : lane, I), islot = (kPlain ? tid : lane) - kslice * I;
    const bool idle = kslice >= K;
    const int jslice = kPlain ? kslice : warp * K + kslice;
    const int S = kPlain ? K : (kThreads / 32) * K;
    const bool has_i = !idle;
    int64_t pi = -1;
    {
        uint32_t mm = mask;
        for (int q = 0; q < islot && mm; q++) mm &= mm - 1;
        if (has_i) pi = p0 + (__ffs(mm) - 1);
    }
    int64_t pload = has_i ? pi : p0 + (__ffs(mask) - 1);  // spare slots repeat a live one; dropped
    if constexpr (kMapI) {
        // slots are positions in a caller's active list; i is its j index
        pload = L.i_map[pload];
        if (has_i) pi = pload;
    }
    typename T::I Iv;
    load_i(rec, pload, Iv);
    // (plain form: read again for every pair, which keeps 12 registers free:
    // a tree interval of N = 65536 takes 52.8 ms against 53.9 ms)
    if (kPlain && tid < I) sm.iv[tid] = Iv;
    typename T::Acc A;
    A.zero();

    const int64_t gb = it.gb, ge = it.ge;
    const int n_parts = it.n_parts;
    const int64_t lb = gb + (int64_t)part * pj;
    const int64_t le = min(ge, lb + (int64_t)pj);
    const int64_t len = le - lb;
    if (tid == 0 && part == 0) n_int += (unsigned long long)n_a * (unsigned long long)(ge - gb - 1);
    // Chunks of TJ list entries are staged in a ring of kStages shared
    // buffers: while one is summed, cp.async fills the next kStages - 1; the
    // list indices of the chunk after those are already loading into
    // registers.  Every step commits one copy group (empty past the end), so
    // waiting for all but the newest kStages - 1 groups means chunk c landed.
    constexpr int EPT = TJ / kThreads;  // staged entries per thread and chunk
    const int n_chunks = (int)((len + TJ - 1) / TJ);
    int32_t nxt[EPT];
    auto load_idx = [&](int c) {
#pragma unroll
        for (int q = 0; q < EPT; q++) {
            const int64_t e = (int64_t)c * TJ + q * kThreads + tid;
            nxt[q] = (c < n_chunks && e < len) ? L.idx[lb + e] : -1;
        }
    };
    auto issue = [&](int c) {  // chunk c's records into buffer c % kStages, indices from nxt
        if (c < n_chunks) {
            const int b = c % kStages;
#pragma unroll
            for (int q = 0; q < EPT; q++) {
                const int e = q * kThreads + tid;
                if constexpr (kPlain) sm.idx[b][e] = nxt[q];
                if (nxt[q] >= 0) cp_async_rec(&sm.rec[b][e], &rec[nxt[q]]);
            }
        }
        cp_async_commit();
    };
    if (n_chunks > 0) {
#pragma unroll
        for (int k = 0; k < kStages - 1; k++) {
            load_idx(k);
            issue(k);
        }
        load_idx(kStages - 1);
    }
    // plain form: softening in integers, room in the sums for a thread's terms
    Soft64 soft{};
    int smin = 0;
    if constexpr (kPlain) {
        soft = soft_of(eps2);
        smin = max(2, 32 - __clz((int)((uint32_t)len / (uint32_t)S + 1u + (uint32_t)n_chunks)));
        A.bad = !soft.ok;
    }
    for (int c = 0; c < n_chunks; c++) {
        const int b = c % kStages;
        const int nc = (len - (int64_t)c * TJ < (int64_t)TJ) ? (int)(len - (int64_t)c * TJ) : TJ;
        issue(c + kStages - 1);  // into the buffer summed in step c - 1 (freed by its closing barrier)
        load_idx(c + kStages);
        cp_async_wait<kStages - 1>();
        group_sync(bar_id);
        if constexpr (kPlain) {
            for (int e = idle ? nc : jslice; e < nc; e += S) {
                asm volatile("" ::: "memory");  // (no hoisting of iv's loads out of the loop)
                interact_int(sm.iv[islot], sm.rec[b][e], (int64_t)sm.idx[b][e] == pi, soft, unit, smin, A);
            }
        } else {
            // FP32 partials are folded into the compensated sums every
            // kFold terms per thread (short plain-FP32 runs keep the
            // partial-sum rounding below the per-term rounding).
            auto chunk = [&](auto normal) {
                for (int e = idle ? nc : jslice; e < nc;) {
                    const int e_end = min(nc, e + kFold * S);
                    for (; e < e_end; e += S) {
                        const RecMix &J = sm.rec[b][e];
                        interact<decltype(normal)::value>(Iv, J, __float_as_int(J.v.w) == (int)pi, eps2, A);
                    }
                    fold_chunk(A);
                }
            };
            if (eps2 >= 1.17549435e-38f) chunk(std::true_type{});
            else chunk(std::false_type{});
        }
        group_sync(bar_id);  // buffer b is refilled by the next step's issue
    }
    // Plain form: sum over the group's K slices for each (i slot,
    // component): the partials go to shared memory, then P contiguous lanes of
    // one warp (P a power of two, P * 7 n_a <= 128) each add a contiguous run
    // of slices in order and a shuffle tree adds the P runs.  A fixed order,
    // with about K / P + log2 P adds per thread, where a butterfly over the
    // lanes costs 7 adds per level for every lane (a warp instruction costs the
    // FP64 pipe the same with one lane active).  With P = 1 a thread may own
    // two outputs (7 n_a <= 224).  Mixed form (FP32 pair adds are cheap, the
    // extra barriers are not): a butterfly over the lanes when n_a is a power
    // of two, else a tree towards slice 0, then a sum over the four warps.
    constexpr bool kTreeTail = kPlain;
    if constexpr (!kTreeTail) {
        if ((I & (I - 1)) == 0) {
            for (int off = I; off < 32; off <<= 1) acc_shfl_add(A, off);
        } else {
            for (int step = 1; step < K; step <<= 1)
                acc_shfl_down_add(A, step * I, !idle && (kslice & (2 * step - 1)) == 0 && kslice + step < K);
        }
    }
    if (kTreeTail ? !idle : lane < I) {
        Red rr;
        to_red(A, rr);
        (&sm.red[0][0])[kPlain ? tid : warp * kMaxTileI + lane] = rr;
    }
    if constexpr (kPlain) {
        // a term that the integers do not take (a number beyond their range,
        // a mass that is not positive), or a particle one of whose components
        // is too small for them: the whole part again in FP64
        warp_span(A.span, I);
        if (group_any(bar_id, A.bad || (lane < I && thin(A.span)))) {
            const bool bad = group_any(bar_id, A.bad);
            if (bad || thin_particles(A.span, reinterpret_cast<Span64 *>(&sm.rec[0][0]), islot, I, tid, bar_id)) {
                RedF64 &out = (&sm.red[0][0])[tid];
                if (!idle && bad) part_sums_f64(rec, L.idx + lb, len, TJ, jslice, S, pi, sm.iv[islot], eps2, out);
                if (!idle && !bad) part_sums_thin(rec, L.idx + lb, len, TJ, jslice, S, pi, sm.iv[islot], eps2, out);
                group_sync(bar_id);
            }
        }
    } else {
        group_sync(bar_id);
    }
    using E = typename std::remove_reference<decltype(sm.red[0][0].v[0])>::type;
    const int n_out = 7 * n_a;
    const int n_sl = kTreeTail ? K : kThreads / 32;  // terms per output
    int lgP = 0;  // (mixed form: one thread per output, warps 0..3 in order)
    if (kTreeTail)
        while (lgP < 5 && (2 << lgP) * n_out <= kThreads && (2 << lgP) <= n_sl) lgP++;
    const int P = 1 << lgP, per = (n_sl + P - 1) >> lgP;
    E r[2] = {E{}, E{}};
    bool has[2] = {false, false};
#pragma unroll
    for (int u = 0; u < 2; u++) {
        const int t = tid + u * kThreads;
        const int o = t >> lgP, q = t & (P - 1);
        if ((u == 0 || P == 1) && o < n_out) {
            const int slot = o / 7, comp = o - 7 * slot;
            const int x1 = min(n_sl, (q + 1) * per);
            for (int x = q * per; x < x1; x++) {
                const E v = (&sm.red[0][0])[kTreeTail ? x * I + slot : x * kMaxTileI + slot].v[comp];
                if (has[u]) comp_add(r[u], v);
                else {
                    r[u] = v;
                    has[u] = true;
                }
            }
        }
        if (u == 0)
            for (int off = P >> 1; off > 0; off >>= 1) {  // P is the same in every lane
                const E ov = shfl_down_e(r[0], off);
                const bool oh = __shfl_down_sync(0xffffffffu, (int)has[0], off) != 0;
                if (q < off && oh) {
                    if (has[0]) comp_add(r[0], ov);
                    else {
                        r[0] = ov;
                        has[0] = true;
                    }
                }
            }
    }
    // the sums, one per output, back into slot order: thread t then holds
    // output t (and t + 128) for the part merge below (already so when P = 1)
    if (P > 1) {
        group_sync(bar_id);
        E *outv = &sm.red[0][0].v[0];
        const int o = tid >> lgP;
        if (o < n_out && (tid & (P - 1)) == 0) outv[o] = r[0];
        group_sync(bar_id);
        if (tid < n_out) r[0] = outv[tid];
    }
    bool write_out = n_parts == 1;
    if (n_parts > 1) {
        // the group's partials are ordered before its arrival by the group
        // barrier and the arrival's release; the last arrival's acquire (and
        // the barrier after it) orders the other parts' partials before the sum
        Red *mine = partials + ((int64_t)slot0 + part) * kMaxTileI;
#pragma unroll
        for (int u = 0; u < 2; u++) {
            const int t = tid + u * kThreads, slot = t / 7, comp = t - 7 * (t / 7);
            if (t < n_out) mine[slot].v[comp] = r[u];
        }
        group_sync(bar_id);
        if (tid == 0) {
            const unsigned int old = atom_add_acq_rel_gpu(reinterpret_cast<unsigned int *>(&L.tile_cnt[it.tile]), 1u);
            sm.last = ((int)old == n_parts - 1);
        }
        group_sync(bar_id);
        write_out = sm.last;
        if (write_out) {
            const Red *base = partials + (int64_t)slot0 * kMaxTileI;
            // Parts are added in blocks of kMergeBlock consecutive parts (more
            // if the block sums would not fit the staging buffers, idle now):
            // (output, block) pairs over all the group's threads each add
            // their block's parts in part order, every load issued first;
            // then each output adds its block sums in block order.  The order
            // depends only on the number of parts, so results stay
            // deterministic; with at most kMergeBlock parts it is the plain
            // sequence p0 + p1 + p2 + ...  A long sequential chain of
            // dependent adds would otherwise dominate a small block step split
            // into many short parts.
            E *buf = reinterpret_cast<E *>(&sm.rec[0][0]);
            constexpr int kBuf = (int)(sizeof(sm.rec) / sizeof(E));
            constexpr int kMergeBlock = 8;
            static_assert(kBuf <= (1 << 14), "small_div");
            static_assert(kMergeBlock == 8, "lgb starts at 3");
            int lgb = 3;
            while (n_out * ((n_parts + (1 << lgb) - 1) >> lgb) > kBuf) lgb++;
            const int blk = 1 << lgb, n_blk = (n_parts + blk - 1) >> lgb;
            for (int x = tid; x < n_out * n_blk; x += kThreads) {
                const int b = small_div(x, n_out), o = x - b * n_out;  // x < kBuf
                const int q0 = b * blk, q1 = min(n_parts, q0 + blk);
                const Red *src = base + o / 7;
                const int comp = o - 7 * (o / 7);
                E vals[kMergeBlock];
#pragma unroll
                for (int k = 0; k < kMergeBlock; k++)
                    if (q0 + k < q1) vals[k] = ld_comp_cg(&src[(int64_t)(q0 + k) * kMaxTileI].v[comp]);
                E acc = vals[0];
#pragma unroll
                for (int k = 1; k < kMergeBlock; k++)
                    if (q0 + k < q1) comp_add(acc, vals[k]);
                for (int q = q0 + kMergeBlock; q < q1; q++)  // blocks longer than kMergeBlock
                    comp_add(acc, ld_comp_cg(&src[(int64_t)q * kMaxTileI].v[comp]));
                buf[x] = acc;
            }
            group_sync(bar_id);
#pragma unroll
            for (int u = 0; u < 2; u++) {
                const int t = tid + u * kThreads;
                if (t < n_out) {
                    r[u] = buf[t];
                    for (int b = 1; b < n_blk; b++) comp_add(r[u], buf[b * n_out + t]);
                }
            }
            if (tid == 0) L.tile_cnt[it.tile] = 0;
        }
    }
    if (write_out) {
#pragma unroll
        for (int u = 0; u < 2; u++) {
            const int t = tid + u * kThreads, slot = t / 7, comp = t - 7 * (t / 7);
            if (t < n_out) {
                uint32_t mm = mask;
                for (int q = 0; q < slot; q++) mm &= mm - 1;
                const int64_t p = p0 + (__ffs(mm) - 1);
                const double v = comp_get(r[u]);
                sm.fin[slot][comp] = v;
                if (comp == 0) sm.pidx[slot] = (int)p;
                if (comp < 3) s.acc1[comp * s.cap_n + p] = v;
                else if (comp < 6) s.jerk1[(comp - 3) * s.cap_n + p] = v;
                else s.pot1[p] = -v;
            }
        }
    }
    // callers put a barrier before the shared buffers are reused
    return write_out;
}

template <typename Rec, int TJ, bool kMapI = false>
__global__ void __launch_bounds__(kThreads, std::is_same<Rec, RecF64>::value ? 4 : 6) k_force(State s, const Rec *__restrict__ rec, Lists L, DevScalars *ds,
                                                    StepCtl c, Params prm)
{
    after_previous();
    double tnow;
    if (!step_time(ds, c, &tnow)) return;
    __shared__ ForceSmem<Rec, TJ> sm;
    const int n_items = (int)ds->n_items;
    const typename Traits<Rec>::Eps eps2 = (typename Traits<Rec>::Eps)prm.eps2;
    unsigned long long n_int = 0;
    for (;;) {
        if (threadIdx.x == 0) sm.item = (int)atomicAdd(&ds->work, 1u);
        __syncthreads();
        const int item = sm.item;
        if (item >= n_items) break;
        force_item<Rec, TJ, kMapI>(s, rec, L, eps2, prm.unit, L.items[item], sm, n_int, threadIdx.x, 0);
        // the next iteration's first barrier protects sm reuse
    }
    if (threadIdx.x == 0 && n_int) atomicAdd(&ds->interactions, n_int);
}

// -------------------------------------------------------------- corrector
__device__ __forceinline__ double norm3(double a, double b, double c) { return sqrt(a * a + b * b + c * c); }

// Largest power of two <= |x| for finite x, as frexp / ldexp give it (so 1/2
// for a zero, whose frexp exponent is 0), on the bits.
__device__ __forceinline__ long long pow2_floor_abs_bits(long long W)
{
    const long long b = W & 0x7FFFFFFFFFFFFFFFll;
    if (b == 0) return 0x3FE0000000000000ll;                          // 1/2
    if ((b >> 52) == 0) return 1ll << (63 - __clzll((unsigned long long)b));  // subnormal: its top bit
    return b & (long long)0xFFF0000000000000ull;
}

// fmod(t, 2^k) == 0 on t's bits: t finite and a multiple of 2^k (fmod of an
// infinity or a NaN is a NaN, so those are not).
__device__ __forceinline__ bool multiple_of_pow2(double t, int k)
{
    const long long b = __double_as_longlong(t) & 0x7FFFFFFFFFFFFFFFll;  // |t|
    if (b == 0) return true;
    const int ef = (int)(b >> 52);
    if (ef == 0x7ff) return false;
    const long long m = ef ? ((b & 0xFFFFFFFFFFFFFll) | (1ll << 52)) : b;  // |t| = m 2^(max(ef, 1) - 1075)
    return (ef ? ef : 1) - 1075 + (__ffsll(m) - 1) >= k;
}

// Block quantisation (McMillan 1986): the largest power of two <= want, at
// most double the old step, doubled only where t_new is a multiple of the
// new step, clamped to [dt_min, dt_max]; a NaN keeps the old step and an
// infinity asks to double.  (The largest power of two below |want| follows
// frexp, so a zero asks for 1/2.)  When dt_old is a normal power of two (as
// in the block-step loops) and dt_min, dt_max are positive normal values,
// every candidate is a positive power of two, IEEE order is the integer order
// of the bits and the multiple test is exact on t_new's bits: the path below
// then uses no FP64 instruction (the FP64 pipe is narrow); otherwise the same
// rule runs in FP64.
__device__ __forceinline__ double block_dt(double want, double dt_old, double t_new, double dt_min, double dt_max)
{
    const long long O = __double_as_longlong(dt_old), Mn = __double_as_longlong(dt_min),
                    Mx = __double_as_longlong(dt_max);
    const long long kNormLo = 0x0010000000000000ll, kTop = 0x7FE0000000000000ll;  // normal, doubling stays finite
    if (O >= kNormLo && O < kTop && (O & 0xFFFFFFFFFFFFFll) == 0 && Mn >= kNormLo && Mn < 0x7FF0000000000000ll && Mx >= kNormLo &&
        Mx < 0x7FF0000000000000ll) {
        const long long W = __double_as_longlong(want);
        const long long O2 = O + (1ll << 52);  // 2 dt_old
        long long Q;
        if ((W & 0x7FF0000000000000ll) == 0x7FF0000000000000ll) Q = (W & 0xFFFFFFFFFFFFFll) ? O : O2;  // NaN, inf
        else Q = pow2_floor_abs_bits(W);
        if (Q > O2) Q = O2;
        if (Q > O && !multiple_of_pow2(t_new, (int)((Q >> 52) & 0x7ff) - 1023)) Q = O;
        if (Q > Mx) Q = Mx;
        if (Q < Mn) Q = Mn;
        return __longlong_as_double(Q);
    }
    double q;
    if (isnan(want)) q = dt_old;
    else if (isinf(want)) q = 2.0 * dt_old;
    else {
        int e;
        frexp(want, &e);
        q = ldexp(1.0, e - 1);
    }
    if (q > 2.0 * dt_old) q = 2.0 * dt_old;
    if (q > dt_old && fmod(t_new, q) != 0.0) q = dt_old;
    if (q > dt_max) q = dt_max;
    if (q < dt_min) q = dt_min;
    return q;
}

__device__ __forceinline__ void atomic_min_time(unsigned long long *slot, double t)
{
    atomicMin(slot, (unsigned long long)__double_as_longlong(t));
}

// Hermite corrector (Makino & Aarseth 1992) for the active particles:
// a2 = (-6 (a0 - a1) - D (4 j0 + 2 j1)) / D^2, a3 = (12 (a0 - a1) + 6 D (j0 + j1)) / D^3,
// x1 = x_p + a2 D^4/24 + a3 D^5/120, v1 = v_p + a2 D^3/6 + a3 D^4/24;
// new step from Aarseth's criterion at the end of the step.
//
// The FP64 pipe is narrow on this GPU (a warp instruction issues in 64 to 76
// cycles per SM sub-partition, however few lanes it has), and a small block
// step's corrector is one warp: its time is the number of its FP64
// instructions.  D is the particle's power-of-two step, so 1/D^2 and 1/D^3 are
// exact powers of two; the timestep criterion works on FP32 values taken from
// the bits (no FP64 norms), and the mixed form's base records are converted on
// the bits: 22 FP64 instructions fewer.  The plain form takes predictor and
// corrector in one Horner form in units of the acceleration, with p = D j0,
// q = D j1, A = a1 - a0:
//   h = D^2 a2 / 2 = 3 A - (2 p + q),  g = D^3 a3 / 6 = p + q - 2 A,
//   x1 = x + D (v + D/2 (a0 + p/3 + h/6 + g/10)),  v1 = v + D (a0 + p/2 + h/3 + g/4),
// 19 FP64 operations a component instead of 27.  (The mixed form keeps the
// longer form: its forces amplify a change of rounding in the corrected
// positions to FP32 size, and now and then to another block step.)  The force phase
// of a small step went from 10.6 to 9.9 us (mixed) and from 12.0 to 11.1 us (plain).
// The per-component arithmetic is shared by the one-thread-per-particle and the
// three-lanes-per-particle correctors, so both give the same bits.

// Powers of D (a power of two) needed by the corrector, exact.
struct StepPowers {
    double D, iD2, iD3, D3, D4;
};

__device__ __forceinline__ StepPowers step_powers(double D)
{
    StepPowers P;
    P.D = D;
    const long long b = __double_as_longlong(D);
    if ((b & ((1ll << 52) - 1)) == 0 && b > 0) {
        const int e = (int)((b >> 52) & 0x7ff) - 1023;  // D = 2^e
        auto p2 = [](int k) { return __longlong_as_double((long long)(1023 + k) << 52); };
        P.iD2 = p2(-2 * e);
        P.iD3 = p2(-3 * e);
        P.D3 = p2(3 * e);
        P.D4 = p2(4 * e);
    } else {  // not reached from the block-step loops (D is a level step)
        const double iD = 1.0 / D;
        P.iD2 = iD * iD;
        P.iD3 = P.iD2 * iD;
        P.D3 = D * D * D;
        P.D4 = D * D * D * D;
    }
    return P;
}

// One Cartesian component: state (x, v, a0, j0) at t, new force (a1, j1) at
// t + D.  Corrected x and v, and for the criterion j1, a^(2) at t + D and
// a^(3), in units that differ by powers of D and constants (crit_units).
struct CorrComp {
    double x, v, q, s, g;
};

template <bool kPlain>
__device__ __forceinline__ CorrComp correct_component(double x, double v, double a0, double j0, double a1, double j1,
                                                      double D)
{
    CorrComp c;
    if constexpr (kPlain) {
        const double p = D * j0, A = a1 - a0;
        c.q = D * j1;
        const double w = p + c.q;
        const double h = fma(3.0, A, -(p + w));
        c.g = fma(-2.0, A, w);  // D^3 a3 / 6
        const double E = fma(0.1, c.g, fma(1.0 / 6.0, h, fma(1.0 / 3.0, p, a0)));
        const double F = fma(1.0 / 3.0, h, fma(0.25, c.g, fma(0.5, p, a0)));
        c.x = fma(D, fma(0.5 * D, E, v), x);
        c.v = fma(D, F, v);
        c.s = fma(3.0, c.g, h);  // D^2 a^(2) / 2
    } else {
        const StepPowers P = step_powers(D);
        const double h = 0.5 * D, th = D * (1.0 / 3.0);
        const double xp = x + D * (v + h * (a0 + th * j0));
        const double vp = v + D * (a0 + h * j0);
        const double a2 = (-6.0 * (a0 - a1) - D * (4.0 * j0 + 2.0 * j1)) * P.iD2;
        const double a3 = (12.0 * (a0 - a1) + 6.0 * D * (j0 + j1)) * P.iD3;
        c.x = xp + P.D4 * (a2 * (1.0 / 24.0) + a3 * D * (1.0 / 120.0));
        c.v = vp + P.D3 * (a2 * (1.0 / 6.0) + a3 * D * (1.0 / 24.0));
        c.q = j1;
        c.s = a2 + a3 * D;
        c.g = a3;
    }
    return c;
}

// |u|^2 from the components' squares, summed x, y, z with single roundings.
__device__ __forceinline__ double norm2_of(double sx, double sy, double sz) { return __dadd_rn(__dadd_rn(sx, sy), sz); }
__device__ __forceinline__ double sq(double u) { return __dmul_rn(u, u); }

// Aarseth's criterion dt^2 = eta (|a||a2| + |j|^2) / (|j||a3| + |a2|^2) from
// A = |a|^2, J = |j|^2, S = |a2|^2, T = |a3|^2.  Only the largest power of
// two below dt is used (block_dt), so it is screened in FP32, which keeps the
// narrow FP64 pipe free.
//
// The criterion is invariant under a change of time unit (J, S, T scale as
// c^-2, c^-4, c^-6 and dt as c) and under a common factor on A, J, S, T.  So
// the four norms are first normalised by exact powers of two taken from the
// exponents of A and J (A' in [1, 2), J' in [1, 8)), which brings the
// shortest steps' huge higher derivatives into FP32 range, and the power of
// two found for the normalised step is shifted back.  The screen works on
// w2 = dt'^2 itself: the power of two below dt' = sqrt(w2) is 2^floor(e / 2)
// for w2's exponent e, and its boundaries are w2's even powers of two.
// Error bound of the FP32 w2 against the exact value of the same normalised
// inputs: truncation to FP32 2^-23 per input (and eta), the square roots as
// y rsqrtf(y) (rsqrtf within 2 ulp), the quotient by __fdividef (within 2
// ulp), the sums of positive terms and the products: at most 24 * 2^-24 in
// all.  When w2 is at least 128 ulps (>= 2^-17 relative) from the even power
// of two on its side (the lower one for an even exponent, the upper one for
// an odd exponent), the exact value and the FP64 expression (within ~1e-15 of
// it) lie between the same two even powers of two, and the exact power of two
// below the FP64 value is returned.  Otherwise (near a boundary, zero or
// non-normal inputs, normalised values outside [2^-60, 2^61), eta outside
// [2^-30, 2^30], or products and steps near the FP64 range's ends, where the
// FP64 expression itself would lose range) the FP64 expression decides.
__device__ __forceinline__ int exp2_of(double x) { return (int)((__double_as_longlong(x) >> 52) & 0x7ff) - 1023; }

// x * 2^m in FP32 for a positive normal double x, mantissa truncated; the
// caller keeps the exponent in FP32's normal range.
__device__ __forceinline__ float f32_scaled(double x, int m)
{
    const long long b = __double_as_longlong(x);
    const int e = (int)((b >> 52) & 0x7ff) - 1023 + m;
    return __int_as_float(((e + 127) << 23) | (int)((b >> 29) & 0x7fffff));
}

__device__ __forceinline__ bool normal_pos(double x)
{
    const long long b = __double_as_longlong(x);
    return b >= 0x0010000000000000ll && b < 0x7ff0000000000000ll;
}

// The screen on FP32 values A, J, S, T (each within 2^-21 of its exact value,
// in [2^-62, 2^62]; the bound above then is 34 * 2^-24): true, and the exponent of the
// power of two below sqrt(eta (sqrt(A S) + J) / (sqrt(J T) + S)), where that is
// certain.
__device__ __forceinline__ bool aarseth_screen(float A, float J, float S, float T, double eta, int &exponent)
{
    const float p1 = A * S, p2 = J * T;
    const float num = p1 * rsqrtf(p1) + J, den = p2 * rsqrtf(p2) + S;
    const float w2 = f32_scaled(eta, 0) * __fdividef(num, den);
    const int wb = __float_as_int(w2);
    const int frac = wb & 0x7fffff, ex = (wb >> 23) & 0xff;
    const int e = ex - 127, odd = e & 1;
    exponent = e >> 1;
    return ex > 0 && ex < 255 && (odd ? frac <= 0x7fffff - 128 : frac >= 128);
}

__device__ __forceinline__ double aarseth_want(double A, double J, double S, double T, double eta)
{
    if (normal_pos(A) && normal_pos(J) && normal_pos(S) && normal_pos(T) && eta >= 0x1p-30 && eta <= 0x1p30) {
        const int eA = exp2_of(A), eJ = exp2_of(J), eS = exp2_of(S), eT = exp2_of(T);
        const int k = (eJ - eA) >> 1;  // 2^2k ~ J / A: the time unit
        const int mA = -eA, mJ = -eA - 2 * k, mS = -eA - 4 * k, mT = -eA - 6 * k;
        const int xS = eS + mS, xT = eT + mT;
        // the FP64 expression of the original inputs stays finite and normal
        const bool fp64_ok = eA + eS > -1000 && eA + eS < 1000 && eJ + eT > -1000 && eJ + eT < 1000;
        if (fp64_ok && xS >= -60 && xS <= 60 && xT >= -60 && xT <= 60) {
            int e2;
            if (aarseth_screen(f32_scaled(A, mA), f32_scaled(J, mJ), f32_scaled(S, mS), f32_scaled(T, mT), eta, e2)) {
                e2 -= k;  // dt = sqrt(w2) / 2^k: exponent of the power of two below dt
                if (e2 > -400 && e2 < 400) return __longlong_as_double((long long)(e2 + 1023) << 52);
            }
        }
    }
    return sqrt(eta * (sqrt(A * S) + J) / (sqrt(J * T) + S));
}

// The corrector's criterion from its components, in units of the acceleration:
// dt = D sqrt(eta (|a| |s| + |q|^2) / (|q| |t| + |s|^2)) with s = D^2 a^(2),
// t = D^3 a^(3), q = D j1 (the same value as above: the unit of time is D).  The
// components' squares come from truncated FP32 values relative to the largest
// component of a (biased exponent ea); the mixed form's j1, a^(2) and a^(3) carry
// their powers of D in the exponent offset.
__device__ __forceinline__ int biased_exp(double x) { return (int)((f64_hi(x) >> 20) & 0x7ffu); }

// (|x| 2^(1023 - ea))^2, |x| truncated to FP32; 0 below 2^-62, infinite above 2^60.
__device__ __forceinline__ float rel_square(double x, int ea)
{
    const uint32_t hi = f64_hi(x);
    const int e = (int)((hi >> 20) & 0x7ffu), r = e - ea;
    const uint32_t b = __funnelshift_l(f64_lo(x), hi & 0x7fffffffu, 3) - ((uint32_t)(ea - 127) << 23);
    const float f = r < -62 || e == 0 ? 0.f : r > 60 ? __int_as_float(0x7f800000) : __uint_as_float(b);
    return __fmul_rn(f, f);
}

// The four squares of one component.
struct CritSquares {
    float a, j, s, t;
};
template <bool kPlain>
__device__ __forceinline__ CritSquares crit_squares(double a1, const CorrComp &c, int ea, double D)
{
    const int k = kPlain ? 0 : biased_exp(D) - 1023;
    return CritSquares{rel_square(a1, ea), rel_square(c.q, ea - k), rel_square(c.s, ea - 2 * k),
                       rel_square(c.g, ea - 3 * k)};
}

// True, and the power of two below the criterion's value, where the screen is
// certain (for a power-of-two D) from the components' summed squares.
template <bool kPlain>
__device__ __forceinline__ bool corrector_screen(float A, float J, float S, float T, double D, double eta, int ea,
                                                 double &want)
{
    if (kPlain) {  // s and t come without their factors 2 and 6
        S = __fmul_rn(4.f, S);
        T = __fmul_rn(36.f, T);
    }
    const float lo = fminf(fminf(A, J), fminf(S, T)), hi = fmaxf(fmaxf(A, J), fmaxf(S, T));
    const long long b = __double_as_longlong(D);
    int e;
    const bool ok = lo >= 0x1p-60f && hi <= 0x1p60f && ea > 0 && ea < 0x7ff && (b & 0xFFFFFFFFFFFFFll) == 0 && b > 0 &&
                    eta >= 0x1p-30 && eta <= 0x1p30 && aarseth_screen(A, J, S, T, eta, e);
    if (!ok) return false;
    const int f = (int)(b >> 52) + e;
    want = __longlong_as_double((long long)f << 52);
    return f > 0 && f < 0x7ff;
}

// The same from FP64 squares.
template <bool kPlain>
__device__ __forceinline__ double corrector_want(double A, double J, double S, double T, double D, double eta)
{
    if (!kPlain) return aarseth_want(A, J, S, T, eta);
    S *= 4.0;
    T *= 36.0;
    return D * sqrt(eta * (sqrt(A * S) + J) / (sqrt(J * T) + S));
}

template <bool kPlain>
__device__ __forceinline__ void correct_particle(const State &s, int64_t p, double tnow, const Params &prm)
{
    const double D = tnow - s.t[p];
    double a1[3];
    CorrComp c[3];
    int ea = 0;
#pragma unroll
    for (int d = 0; d < 3; d++) {
        const double a0 = s.a[d * s.cap_j + p], j0 = s.jk[d * s.cap_j + p];
        a1[d] = s.acc1[d * s.cap_n + p];
        const double j1 = s.jerk1[d * s.cap_n + p];
        c[d] = correct_component<kPlain>(s.x[d * s.cap_j + p], s.v[d * s.cap_j + p], a0, j0, a1[d], j1, D);
        s.x[d * s.cap_j + p] = c[d].x;
        s.v[d * s.cap_j + p] = c[d].v;
        s.a[d * s.cap_j + p] = a1[d];
        s.jk[d * s.cap_j + p] = j1;
        ea = max(ea, biased_exp(a1[d]));
    }
    CritSquares u[3];
#pragma unroll
    for (int d = 0; d < 3; d++) u[d] = crit_squares<kPlain>(a1[d], c[d], ea, D);
    auto sum3 = [](float x, float y, float z) { return __fadd_rn(__fadd_rn(x, y), z); };
    double want;
    if (!corrector_screen<kPlain>(sum3(u[0].a, u[1].a, u[2].a), sum3(u[0].j, u[1].j, u[2].j),
                                  sum3(u[0].s, u[1].s, u[2].s), sum3(u[0].t, u[1].t, u[2].t), D, prm.eta, ea, want))
        want = corrector_want<kPlain>(norm2_of(sq(a1[0]), sq(a1[1]), sq(a1[2])),
                                      norm2_of(sq(c[0].q), sq(c[1].q), sq(c[2].q)),
                                      norm2_of(sq(c[0].s), sq(c[1].s), sq(c[2].s)),
                                      norm2_of(sq(c[0].g), sq(c[1].g), sq(c[2].g)), D, prm.eta);
    const double dtn = block_dt(want, s.dt[p], tnow, prm.dt_min, prm.dt_max);
    s.t[p] = tnow;
    s.dt[p] = dtn;
    if (s.base) refresh_base(s, p);
}

static __global__ void k_correct(State s, DevScalars *ds, StepCtl c, Params prm)
{
    double tnow;
    if (!step_time(ds, c, &tnow)) return;
    const int64_t n = ds->n;
    double my_min = __longlong_as_double(0x7FF0000000000000LL);
    int my_cnt = 0;
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < n; p += (int64_t)gridDim.x * blockDim.x) {
        const bool act = is_active(s, c, p, tnow);
        if (act) {
            if (c.mode == 1 && s.t[p] + s.dt[p] != tnow) {
                atomicExch(&ds->err, -1);  // HH_EINVAL: marked particle not due at t
                continue;
            }
            if (s.base) correct_particle<false>(s, p, tnow, prm);
            else correct_particle<true>(s, p, tnow, prm);
            my_cnt++;
        }
        const double tn = s.t[p] + s.dt[p];
        my_min = tn < my_min ? tn : my_min;
    }
    if (c.mode != 0) return;
    // block min, then one atomic per CTA
    for (int off = 16; off > 0; off >>= 1) {
        my_min = fmin(my_min, __shfl_xor_sync(0xffffffffu, my_min, off));
        my_cnt += __shfl_xor_sync(0xffffffffu, my_cnt, off);
    }
    __shared__ double s_min[32];
    __shared__ int s_cnt[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0) {
        s_min[warp] = my_min;
        s_cnt[warp] = my_cnt;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double mn = s_min[0];
        int cn = s_cnt[0];
        for (int w = 1; w < (int)(blockDim.x >> 5); w++) {
            mn = fmin(mn, s_min[w]);
            cn += s_cnt[w];
        }
        atomic_min_time(&ds->tmin[c.slot_next], mn);
        if (blockIdx.x == 0) {  // the force kernel of this step has finished
            ds->n_items = 0u;
            ds->slot_ctr = 0u;
        }
        if (cn) {
            atomicAdd(&ds->n_act_last, cn);
            atomicAdd(&ds->particle_steps, (unsigned long long)cn);
        }
    }
}

// min over particles of t_i + dt_i into tmin[slot] (slot preset to +inf).
static __global__ void k_min_time(State s, DevScalars *ds, int slot)
{
    const int64_t n = ds->n;
    double my_min = __longlong_as_double(0x7FF0000000000000LL);
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < n; p += (int64_t)gridDim.x * blockDim.x) {
        const double tn = s.t[p] + s.dt[p];
        my_min = tn < my_min ? tn : my_min;
    }
    for (int off = 16; off > 0; off >>= 1) my_min = fmin(my_min, __shfl_xor_sync(0xffffffffu, my_min, off));
    if ((threadIdx.x & 31) == 0) atomic_min_time(&ds->tmin[slot], my_min);
}

// Initial step from eta_s |a| / |jk|, quantised (reading: the paper is silent).
static __global__ void k_init_dt(State s, DevScalars *ds, Params prm)
{
    const int64_t n = ds->n;
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < n; p += (int64_t)gridDim.x * blockDim.x) {
        const double na = norm3(s.a[p], s.a[s.cap_j + p], s.a[2 * s.cap_j + p]);
        const double nj = norm3(s.jk[p], s.jk[s.cap_j + p], s.jk[2 * s.cap_j + p]);
        double q;
        if (nj == 0.0) q = prm.dt_max;
        else {
            const double want = prm.eta_s * na / nj;
            q = (want > 0.0 && want < 1.0e300) ? pow2_floor(want) : prm.dt_max;
        }
        if (q > prm.dt_max) q = prm.dt_max;
        if (q < prm.dt_min) q = prm.dt_min;
        s.dt[p] = q;
    }
}

// a, jk of every particle <- last force results (initial forces).
static __global__ void k_adopt_forces(State s, DevScalars *ds)
{
    const int64_t n = ds->n;
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < n; p += (int64_t)gridDim.x * blockDim.x) {
#pragma unroll
        for (int d = 0; d < 3; d++) {
            s.a[d * s.cap_j + p] = s.acc1[d * s.cap_n + p];
            s.jk[d * s.cap_j + p] = s.jerk1[d * s.cap_n + p];
        }
        if (s.base) refresh_base(s, p);
    }
}

// A load through the second set of state buffers: checks x, v (finite: bit 0 of
// *bad) and m (finite and > 0: bit 1) of n particles there.
static __global__ void k_load_check(State s, int64_t n, int32_t *bad)
{
    int32_t wrong = 0;
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < n; q += (int64_t)gridDim.x * blockDim.x) {
        for (int d = 0; d < 3; d++) {
            const uint32_t x = f64_hi(s.x[d * s.cap_j + q]), v = f64_hi(s.v[d * s.cap_j + q]);
            if ((x & 0x7ff00000u) == 0x7ff00000u || (v & 0x7ff00000u) == 0x7ff00000u) wrong |= 1;
        }
        const long long m = __double_as_longlong(s.m[q]);  // (positive and finite, as an integer)
        if (m <= 0 || m >= 0x7ff0000000000000ll) wrong |= 2;
    }
    if (wrong) atomicOr(bad, wrong);
}

// What a load of particle q at time t leaves besides x, v and m.
__device__ __forceinline__ void load_rest(const State &s, int64_t q, double t)
{
    for (int d = 0; d < 3; d++) s.a[d * s.cap_j + q] = s.jk[d * s.cap_j + q] = 0.0;
    s.t[q] = t;
    if (s.base) refresh_base(s, q);
}

// Then, if all was right, the particles from there into the state, and the verdict.
static __global__ void k_load_checked(State from, State s, int64_t n, double t, const int32_t *bad, volatile int32_t *verdict)
{
    const int32_t wrong = *bad;
    if (blockIdx.x == 0 && threadIdx.x == 0) *verdict = wrong;
    if (wrong) return;
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < n; q += (int64_t)gridDim.x * blockDim.x) {
        for (int d = 0; d < 3; d++) {
            s.x[d * s.cap_j + q] = from.x[d * from.cap_j + q];
            s.v[d * s.cap_j + q] = from.v[d * from.cap_j + q];
        }
        s.m[q] = from.m[q];
        load_rest(s, q, t);
    }
}

static __global__ void k_load_rest(State s, int64_t n, double t)
{
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < n; q += (int64_t)gridDim.x * blockDim.x)
        load_rest(s, q, t);
}

static __global__ void k_refresh_base(State s, int64_t first, int64_t n)
{
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < n; q += (int64_t)gridDim.x * blockDim.x)
        refresh_base(s, first + q);
}

// Start of an explicit evaluation: marks the listed particles and empties the
// work queue.  An index outside [0, n_part) sets ds->err; *verdict (host
// memory) is then set, as it is for an error that was pending.
static __global__ void k_mark_begin(int32_t *mark, const int32_t *idx, int32_t n, int64_t n_part, DevScalars *ds,
                                    volatile int32_t *verdict)
{
    after_previous();
    const int q0 = blockIdx.x * blockDim.x + threadIdx.x;
    if (q0 == 0) {
        if (*(volatile int32_t *)&ds->err) *verdict = 1;
        ds->work = 0u;
        ds->n_items = 0u;
        ds->slot_ctr = 0u;
    }
    for (int q = q0; q < n; q += gridDim.x * blockDim.x) {
        const int32_t p = idx[q];
        if (p < 0 || p >= n_part) {
            atomicExch(&ds->err, -1);
            *verdict = 1;
        } else {
            mark[p] = 1;
        }
    }
}

// End of it: out[3][n_act] (SoA) <- acc1 etc. at idx (with out set), marks
// cleared; *verdict (host memory, may be NULL) <- ds->err.
static __global__ void k_mark_end(State s, const int32_t *idx, int32_t n_act, int64_t n_part, bool out, double *acc,
                                  double *jerk, double *pot, const DevScalars *ds, volatile int32_t *verdict)
{
    wait_previous();  // (the caller's own kernels may come next)
    const int32_t err = *(volatile const int32_t *)&ds->err;
    const int q0 = blockIdx.x * blockDim.x + threadIdx.x;
    if (q0 == 0 && verdict) *verdict = err;
    for (int q = q0; q < n_act; q += gridDim.x * blockDim.x) {
        const int64_t p = idx[q];
        if (p < 0 || p >= n_part) continue;
        if (out && !err) {
#pragma unroll
            for (int d = 0; d < 3; d++) {
                if (acc) acc[(int64_t)d * n_act + q] = s.acc1[d * s.cap_n + p];
                if (jerk) jerk[(int64_t)d * n_act + q] = s.jerk1[d * s.cap_n + p];
            }
            if (pot) pot[q] = s.pot1[p];
        }
        s.mark[p] = 0;
    }
}

// Device-side input validation for *_dev uploads: finite values, m > 0.
static __global__ void k_check_j(const State s, int64_t first, int64_t n, DevScalars *ds)
{
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < n; q += (int64_t)gridDim.x * blockDim.x) {
        const int64_t e = first + q;
        bool ok = s.m[e] > 0.0 && isfinite(s.m[e]) && isfinite(s.t[e]);
        for (int d = 0; d < 3; d++)
            ok = ok && isfinite(s.x[d * s.cap_j + e]) && isfinite(s.v[d * s.cap_j + e]) &&
                 isfinite(s.a[d * s.cap_j + e]) && isfinite(s.jk[d * s.cap_j + e]);
        if (!ok) atomicExch(&ds->err, -1);
    }
}

}  // namespace hh
