// Krylov solvers of the reduced camera system S dx_p = -b~ (Section 3.2), for one problem or for
// a batch of independent problems that share every launch.
//
// Algorithm 1 (block-Jacobi PCG) and Algorithm 2 (MCG) run as a fixed sequence of kernels per
// iteration.  All data-dependent control (the stop test, the tau-test and the width of the next
// direction block, the history size) lives in one device struct Ctl per problem, written only by
// the per-problem "decide" steps (run by one CTA of the kernel after an update, and by the small
// solve) and read by the others.  A whole solve is one CUDA graph: a conditional WHILE node
// repeats a body of `chunk` iterations while k_loop_cond finds a problem that is not done (the
// float64 iterative refinement of mixed precision is an outer WHILE node around it), so the host
// launches the graph once and reads the results once; nothing inside a solve waits on the host.
// A problem whose Ctl::done is set is skipped by every later launch while the others go on.
// Problems of a few cameras run their whole sweep in one launch (k_one_cta, k_pcg_cluster), beside that
// loop where a batch has larger ones too.
//
// Batches: problem b owns the cameras [c0, c0 + nc) of the handle (S is block-diagonal over the
// problems, since no landmark is seen by two of them).  Per-problem kernels take the problem from
// blockIdx.y; the block-sparse products run over one work list of all problems' rows, each item
// tagged with its problem.  Every per-problem result is summed in an order fixed by the problem
// alone (its own cameras, rows and work items), so a problem solved inside a batch gives the
// same bits as the same problem solved alone.  One problem is the batch of one.
//
// MCG data: the search blocks P_j and their images Q_j are kept as columns of two column-major
// arrays per problem (column c at hoff + c * n, n = 9 nc); block j starts at column blk_off[j]
// and is blk_w[j] wide (1 for a global step, N_eff for a local one).  The pseudo-inverse of
// Delta_j is kept for the full reorthogonalisation
//     beta_{i,j} = Delta_j^+ Q_j^T Z_{i+1},  P_{i+1} = Z_{i+1} - sum_j P_j beta_{i,j},
//     Q_{i+1}   = S Z_{i+1} - sum_j Q_j beta_{i,j}            (Eq. 18 with j = 0..i)
// where S Z_{i+1} applies each block S_jk only to the column of the subset of pose k
// (the product trick of Section 3.2).
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <functional>
#include <numeric>
#include <queue>
#include <utility>
#include <vector>

#include "ba_internal.cuh"
#include "df64.cuh"

namespace ba {

namespace {

constexpr int kGramMax = kMaxDirs * kMaxDirs + kMaxDirs;   // Delta (w x w) and gamma (w)
constexpr int kChunkCams = 112;                             // cameras per Phi partial
constexpr double kStagnation = 1e-4;                        // float32 sweep stop on t_i (see Ctl::stag)
// Cameras and threads per CTA of the update kernels (126 rows).  Their time is a chain of latencies
// (the camera sums, D^{-1} r, the CTA sum), so the CTAs are small: 72 of them for 1000 cameras; with 252
// rows each, half as many SMs carried twice the arithmetic.
constexpr int kUpdCams = 14;
constexpr int kUpdThreads = 128;
constexpr int kMaxProblemCams = 28 * 65535;   // accepted in one problem (no grid is near its limit there)

// Where one problem of the batch lives (fixed for a solve).
struct Layout {           // no padding (compared as bytes)
    int c0, nc;          // first camera, number of cameras
    int64_t hoff;        // first element of its direction history (cap columns of 9 nc rows)
    int64_t phoff;       // first Phi partial
    int64_t boff;        // first beta row (16 values each)
    int n_eff, sz, K, cap;
};

struct Ctl {
    Layout lay;
    int it;            // completed steps
    int done;
    int status;
    int cols;          // history columns in use
    int hist_cols;     // columns the current reorthogonalisation runs over
    int new_off;       // first column of the block being formed
    int w_new;         // its width
    int local;         // 1 if the block being formed holds the local directions
    int local_steps;
    int n_eff;
    int sz;            // poses per subset
    int K;             // Phi partials per subset
    int max_iters;
    int cap;
    int w_cur;         // width of the current block (set by decide for the next gram)
    int off_cur;
    double rr0, rr, rz, ga, tol2, tau;
    double rr0_inv;    // 1 / rr0: the residual history stores rr / rr0 without a division per step
    int alone;         // k_one_cta or k_pcg_cluster solves the problem; done is set for everyone else
    int live;          // the problem was not done at this iteration's update (read by the kernel whose
                       // first CTA runs the decide step, which may set done meanwhile)
    double alpha_v[kMaxDirs];
    double true_rr, bb;                 // true residual and |rhs|^2
    int scaled_exp;    // mixed precision: the largest exponent of Lam (true residual)
    double stag;       // float32 sweeps: stop when t_i (energy decrease / r^T D^-1 r) falls below this
    int direct_q;      // 1: Q_{i+1} = S P_{i+1} (Algorithm 2); 0: the Q update of Eq. 18
    int pinv_steps;    // steps whose Delta_i took the eigen-decomposition pseudo-inverse
    int hist_off;      // residual history: this sweep's first row (earlier sweeps' steps)
    double hist_scale; // and the factor that puts its values in units of the outer |b~|^2
};

// Per-solve arguments read by the kernels (one copy in device memory, written before each launch of
// the solve graph, so one captured graph serves every tolerance, tau and iteration budget).
struct Params {
    double tol, tau, inner_tol;
    int max_iters, max_refine, mcg, pad;
};

// Loop counters of a solve (zeroed before each launch): body passes of the Krylov loop (all sweeps),
// passes of the refinement loop, passes of the current sweep, and whether the safety bound ended a
// loop with a problem still running.
struct Loops {
    int inner, outer, cur, capped;
};

// Float64 iterative refinement of one problem (mixed precision).
struct Outer {
    double bb;         // |b~|^2
    double tr;         // |-b~ - S x|^2 of the current x
    double tr_prev;    // the same before the last sweep (scales that sweep's residual history)
    double tol_in;     // relative tolerance of the next inner sweep
    double unit;       // power of two near the largest value of Lam (-b~ - S x), the residual of the sweeps'
                       // scaled system: the sweep solves for that residual divided by it
    int se;            // its exponent
    int status;
    int active;        // still refining
    int swept;         // takes part in the sweep being run
    int sweeps, iters, locals, pinvs;
    int max_in;        // iteration budget of the next sweep
    int cols;          // history columns of its last sweep
};

__device__ __forceinline__ int64_t gtid() { return int64_t(blockIdx.x) * blockDim.x + threadIdx.x; }
__device__ __forceinline__ int64_t gstride() { return int64_t(gridDim.x) * blockDim.x; }

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) v += __shfl_xor_sync(0xffffffffu, v, s);
    return v;
}
__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) v += __shfl_xor_sync(0xffffffffu, v, s);
    return v;
}

// Sum of products a_i b_i of float32 (or float64) values.  float64: plain float64 accumulation.
// float32: each product is split exactly into p + e (p = fl(a b), e = fma(a, b, -p)) and added to
// a float pair (hi, lo) with an error-free two-sum, so the sum keeps about 48 bits without
// float64 arithmetic, which runs at a small fraction of the float32 rate on this GPU.
template <typename T>
struct ExactSum;
template <>
struct ExactSum<double> {
    double s = 0.0;
    __device__ __forceinline__ void add(double a, double b) { s += a * b; }
    __device__ __forceinline__ double value() const { return s; }
};
template <>
struct ExactSum<float> {
    float hi = 0.f, lo = 0.f;
    __device__ __forceinline__ void add(float a, float b) {
        const float p = __fmul_rn(a, b);
        const float pe = __fmaf_rn(a, b, -p);
        const float t = __fadd_rn(hi, p);
        const float bv = __fsub_rn(t, hi);
        const float te = __fadd_rn(__fsub_rn(hi, __fsub_rn(t, bv)), __fsub_rn(p, bv));
        hi = t;
        lo = __fadd_rn(lo, __fadd_rn(te, pe));
    }
    __device__ __forceinline__ double value() const { return double(hi) + double(lo); }
    // add another pair (h, l): error-free two-sum of the high parts, low parts added
    __device__ __forceinline__ void add_pair(float h, float l) {
        const float t = __fadd_rn(hi, h);
        const float bv = __fsub_rn(t, hi);
        const float te = __fadd_rn(__fsub_rn(hi, __fsub_rn(t, bv)), __fsub_rn(h, bv));
        hi = t;
        lo = __fadd_rn(lo, __fadd_rn(te, l));
    }
};

// A Gram partial sum as stored between the Gram and the small-solve kernels: float64, or (for the
// float32 sweeps) the float pair (hi, lo) in the same 8 bytes, so that adding the partials needs no
// float64 arithmetic either.
__device__ __forceinline__ void store_partial(double* slot, const ExactSum<double>& s) { *slot = s.value(); }
__device__ __forceinline__ void store_partial(double* slot, const ExactSum<float>& s) {
    *reinterpret_cast<float2*>(slot) = make_float2(s.hi, s.lo);
}
__device__ __forceinline__ void load_partial(ExactSum<double>& s, const double* slot) { s.s += *slot; }
__device__ __forceinline__ void combine(ExactSum<double>& a, const ExactSum<double>& b) { a.s += b.s; }
__device__ __forceinline__ void combine(ExactSum<float>& a, const ExactSum<float>& b) { a.add_pair(b.hi, b.lo); }
// a += the same sum held by lane (lane ^ o) (every lane of the warp calls this)
__device__ __forceinline__ void combine_shfl(ExactSum<double>& a, int o) { a.s += __shfl_xor_sync(0xffffffffu, a.s, o); }
__device__ __forceinline__ void combine_shfl(ExactSum<float>& a, int o) {
    const float h = __shfl_xor_sync(0xffffffffu, a.hi, o), l = __shfl_xor_sync(0xffffffffu, a.lo, o);
    a.add_pair(h, l);
}
__device__ __forceinline__ void load_partial(ExactSum<float>& s, const double* slot) {
    const float2 v = *reinterpret_cast<const float2*>(slot);
    s.add_pair(v.x, v.y);
}

// add the slot whose 8 bytes are in v (loaded earlier)
__device__ __forceinline__ void add_slot(ExactSum<double>& s, double v) { s.s += v; }
__device__ __forceinline__ void add_slot(ExactSum<float>& s, double v) {
    s.add_pair(__int_as_float(__double2loint(v)), __int_as_float(__double2hiint(v)));
}
template <typename T>
__device__ __forceinline__ ExactSum<T> warp_total(ExactSum<T> s) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) combine_shfl(s, o);
    return s;
}

// A sum over lanes, warps and CTAs that stays within a float64 sum's error.  A float pair loses 2^-48 of the
// partial sum at every addition, against 2^-53 in float64; a third term keeps what the low parts' additions
// round off (two-sums again, on the float32 pipe), so the additions lose about 2^-72 and the total is rounded
// once, by value().  float64: the sum itself.
__device__ __forceinline__ float two_sum(float a, float b, float& e) {   // fl(a + b), e = its exact error
    const float t = __fadd_rn(a, b), bv = __fsub_rn(t, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(t, bv)), __fsub_rn(b, bv));
    return t;
}
// a float32 as float64, from its bits: a conversion instruction runs on the float64 pipe (about 150 cycles), this
// on the integer pipe.  Subnormals (below 1e-38 of sums that start near one) become zero.
__device__ __forceinline__ double widen(float f) {
    const int b = __float_as_int(f), e = b & 0x7f800000;
    // exponent 255 (infinities and NaN) becomes 2047
    const long long m = (static_cast<long long>(b & 0x7fffffff) << 29) + (e == 0x7f800000 ? 1792ll << 52 : 896ll << 52);
    return __longlong_as_double((e == 0 ? 0ll : m) | (static_cast<long long>(b & int(0x80000000)) << 32));
}
template <typename T>
struct WideSum;
template <>
struct WideSum<double> {
    using Slot = double;   // as stored between kernels
    double s = 0.0;
    __device__ __forceinline__ WideSum() {}
    __device__ __forceinline__ WideSum(const ExactSum<double>& a) : s(a.s) {}
    __device__ __forceinline__ void set(double v) { s = v; }
    __device__ __forceinline__ void add(double v) { s += v; }
    __device__ __forceinline__ void add(const WideSum& b) { s += b.s; }
    __device__ __forceinline__ WideSum shfl_xor(int o) const {
        WideSum b;
        b.s = __shfl_xor_sync(0xffffffffu, s, o);
        return b;
    }
    __device__ __forceinline__ Slot slot() const { return s; }
    __device__ __forceinline__ double value() const { return s; }
};
template <>
struct WideSum<float> {
    using Slot = float4;
    float hi = 0.f, lo = 0.f, c = 0.f;
    __device__ __forceinline__ WideSum() {}
    __device__ __forceinline__ WideSum(const ExactSum<float>& a) : hi(a.hi), lo(a.lo) {}
    __device__ __forceinline__ void add3(float h, float l, float k) {
        float te, ue, ve;
        hi = two_sum(hi, h, te);
        lo = two_sum(lo, l, ue);
        lo = two_sum(lo, te, ve);
        c = __fadd_rn(__fadd_rn(c, k), __fadd_rn(ue, ve));
    }
    __device__ __forceinline__ void mul_add(float a, float b) {
        const float p = __fmul_rn(a, b);
        add3(p, __fmaf_rn(a, b, -p), 0.f);
    }
    __device__ __forceinline__ void set(const Slot& v) { hi = v.x, lo = v.y, c = v.z; }
    __device__ __forceinline__ void add(const Slot& v) { add3(v.x, v.y, v.z); }
    __device__ __forceinline__ void add(const WideSum& b) { add3(b.hi, b.lo, b.c); }
    __device__ __forceinline__ WideSum shfl_xor(int o) const {
        WideSum b;
        b.hi = __shfl_xor_sync(0xffffffffu, hi, o);
        b.lo = __shfl_xor_sync(0xffffffffu, lo, o);
        b.c = __shfl_xor_sync(0xffffffffu, c, o);
        return b;
    }
    __device__ __forceinline__ Slot slot() const { return make_float4(hi, lo, c, 0.f); }
    __device__ __forceinline__ double value() const { return widen(hi) + (widen(lo) + widen(c)); }
};
template <typename T>
using WideSlot = typename WideSum<T>::Slot;
// the sum in a slot of store_partial
template <typename T>
__device__ __forceinline__ WideSum<T> pair_of(double slot) {
    WideSum<T> s;
    if constexpr (sizeof(T) == 4) {
        s.hi = __int_as_float(__double2loint(slot));
        s.lo = __int_as_float(__double2hiint(slot));
    } else {
        s.s = slot;
    }
    return s;
}
template <typename T>
__device__ __forceinline__ WideSum<T> warp_total(WideSum<T> s) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s.add(s.shfl_xor(o));
    return s;
}

// Value k of the kThreads / 32 warp sums in red (row stride nv), added as a fixed tree
// ((w0 + w1) + (w2 + w3)) + ((w4 + w5) + (w6 + w7)): three dependent float64 additions.
__device__ __forceinline__ double sum_warps(const double* red, int nv, int k) {
    static_assert(kThreads == 256, "tree over eight warps");
    const double a = red[0 * nv + k] + red[1 * nv + k], b = red[2 * nv + k] + red[3 * nv + k];
    const double c = red[4 * nv + k] + red[5 * nv + k], d = red[6 * nv + k] + red[7 * nv + k];
    return (a + b) + (c + d);
}

// Sum `nv` values per thread over the CTA; threads 0..NV-1 write them to out[0..NV) (global or
// shared memory), visible to the whole CTA on return.
template <int NV>
__device__ __forceinline__ void cta_sum_write(double (&v)[NV], double* out) {
    __shared__ double red[kThreads / 32][NV];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < NV; ++k) {
        double s = warp_sum(v[k]);
        if (lane == 0) red[wid][k] = s;
    }
    __syncthreads();
    if (threadIdx.x < NV) out[threadIdx.x] = sum_warps(&red[0][0], NV, threadIdx.x);
    __syncthreads();
}

// Sum of the slots [0 .. np) in a fixed order (one warp; every lane returns it).
template <typename T>
__device__ __forceinline__ WideSum<T> warp_sum_slots(const WideSlot<T>* slots, int np) {
    WideSum<T> s;
    for (int p = threadIdx.x & 31; p < np; p += 32) s.add(slots[p]);
    return warp_total(s);
}

// Sum partial[p * stride + k] over p < np in a fixed order (called by one warp; every lane returns it).
__device__ __forceinline__ double sum_partials(const double* partial, int np, int stride, int k) {
    const int lane = threadIdx.x & 31;
    double s = 0.0;
    for (int p = lane; p < np; p += 32) s += partial[int64_t(p) * stride + k];
    return warp_sum(s);
}

// ---------------------------------------------------------------------------------------
// block-sparse products

// Work items of the block-sparse products.  Item = a chunk [q0, q1) of the blocks of block-row
// `row` that feed output column `seg` (the subset of the column cameras in MCG's local step, 0
// otherwise) of problem `prob`; it is chunk k of the ng chunks of its output group (row, seg),
// whose partial-sum slots are slot - k .. slot - k + ng - 1.  Each chunk writes its 9 partial
// sums, and the warp that finishes last (atomic count, no waiting) adds the partials in chunk
// order, so the result does not depend on scheduling or on the order of the list.  Counters reset
// themselves.
struct SpItem {
    int row, seg, q0, q1, grp, k, ng, prob, slot;
};

struct ItemList {
    const SpItem* items = nullptr;
    int64_t n = 0;
    int* cnt = nullptr;       // one per group, zero between launches
    void* part = nullptr;     // n x 9 partial sums (element type of the product), by slot
    int nprob = 0;            // problems the list covers
    int polls = kDefaultWaitPolls;   // polls of a tile barrier before a wait gives up (0: at once)
    int ngrp = 0;             // groups (counters)
    // Balanced order: warp g of a launch with nw warps takes items wptr[g] .. wptr[g + 1] - 1 (the
    // list is ordered so that the warps' tiles are about equal); a launch with another warp count
    // takes every (its warps)-th item instead.
    const int64_t* wptr = nullptr;
    int64_t nw = 0;
};

// The items of this warp: its range of the balanced order, or every W-th item.
struct WarpItems {
    int64_t i0, end, step;
};
__device__ __forceinline__ WarpItems warp_items(const ItemList& L, int NW, int wid) {
    const int64_t W = int64_t(gridDim.x) * NW, g = int64_t(blockIdx.x) * NW + wid;
    if (L.wptr != nullptr && W == L.nw) return {L.wptr[g], L.wptr[g + 1], 1};
    return {g, L.n, W};
}

// Which problems a product serves: every live one, those forming a global (local) block, or those
// whose new block is one column wide (wider).
enum : int { kSelLive = 0, kSelGlobal = 1, kSelLocal = 2, kSelW1 = 3, kSelWide = 4 };

__device__ __forceinline__ bool selected(const Ctl* ctl, int prob, int sel) {
    const Ctl& c = ctl[prob];
    if (c.done) return false;
    switch (sel) {
        case kSelGlobal: return c.local == 0;
        case kSelLocal: return c.local != 0;
        case kSelW1: return c.w_new == 1;
        case kSelWide: return c.w_new > 1;
        default: return true;
    }
}

// true when no problem of the list is selected (checked for small batches only; every warp of the
// CTA reaches the same answer, so the whole CTA may return)
__device__ __forceinline__ bool nothing_selected(const Ctl* ctl, const ItemList& L, int sel) {
    if (L.nprob > 64) return false;
    bool any = false;
    for (int b = threadIdx.x & 31; b < L.nprob; b += 32) any = any || selected(ctl, b, sel);
    return !__any_sync(0xffffffffu, any);
}

// Sum the CTA's NV values (kUpdThreads threads) into partial[blockIdx.x * NV ..], as accurately as in float64
// (a thread's value is one product, exact as a pair).
// Warp k adds value k: 3 additions and one shuffle tree per value instead of a tree in every warp.
// The next kernel adds the CTAs' partials (total_of): with the last CTA to arrive doing it here, its
// fences, its counter and a second round of loads held an update for 3 us.
template <typename T, int NV>
__device__ __forceinline__ void cta_publish(const ExactSum<T> (&v)[NV], WideSlot<T>* partial) {
    static_assert(NV <= kUpdThreads / 32, "one warp per value");
    __shared__ double st[NV][kUpdThreads];   // slots of store_partial
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < NV; ++k) store_partial(&st[k][threadIdx.x], v[k]);
    __syncthreads();
    if (wid < NV) {
        static_assert(kUpdThreads == 128, "four values a lane");
        WideSum<T> s = pair_of<T>(st[wid][lane]);
        s.add(pair_of<T>(st[wid][lane + 32]));
        if constexpr (sizeof(T) == 4) {   // two chains: a wide addition is a dozen dependent operations
            WideSum<T> s2 = pair_of<T>(st[wid][lane + 64]);
            s2.add(pair_of<T>(st[wid][lane + 96]));
            s.add(s2);
        } else {
            s.add(pair_of<T>(st[wid][lane + 64]));
            s.add(pair_of<T>(st[wid][lane + 96]));
        }
        s = warp_total(s);
        if (lane == 0) partial[int64_t(blockIdx.x) * NV + wid] = s.slot();
    }
}

// Total of value k over np CTA partials (one warp; every lane returns it): lane l adds partials
// l, l + 32, ..., eight loads in flight, then the fixed shuffle tree.
template <typename T, int NV>
__device__ __forceinline__ WideSum<T> total_of(const WideSlot<T>* partial, int np, int k) {
    WideSum<T> s;
    const int lane = threadIdx.x & 31;
    for (int b0 = 0; b0 < np; b0 += 8 * 32) {
        WideSlot<T> v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u)
            v[u] = b0 + 32 * u + lane < np ? partial[int64_t(b0 + 32 * u + lane) * NV + k] : WideSlot<T>{};
#pragma unroll
        for (int u = 0; u < 8; ++u)
            if (b0 + 32 * u < np) {   // the same in every lane; past np the slots are zero
                if (b0 == 0 && u == 0) s.set(v[u]);
                else s.add(v[u]);
            }
    }
    return warp_total(s);
}

// Row of a camera's D^{-1} block, and its product with the camera's residual.  The float32 sweeps keep
// the blocks in double-float (k_block_jacobi) and form the product with error-free transformations,
// rounded once to float32, like the float64 product that it replaces: nine dependent float64
// multiply-adds and nine conversions per row held the update at 12 us on 1000 cameras.
template <typename T>
struct DinvRow;
template <>
struct DinvRow<double> {
    double d[9];
    __device__ __forceinline__ void load(const double* row, bool act) {
#pragma unroll
        for (int b = 0; b < 9; ++b) d[b] = act ? row[b] : 0.0;
    }
    __device__ __forceinline__ double dot(const double* r) const {
        double s[3] = {0.0, 0.0, 0.0};   // a float64 operation takes about 150 cycles: short chains
#pragma unroll
        for (int b = 0; b < 9; ++b) s[b % 3] += d[b] * r[b];
        return (s[0] + s[1]) + s[2];
    }
};
template <>
struct DinvRow<float> {
    float2 d[9];
    __device__ __forceinline__ void load(const double* row, bool act) {
#pragma unroll
        for (int b = 0; b < 9; ++b) d[b] = act ? reinterpret_cast<const float2*>(row)[b] : make_float2(0.f, 0.f);
    }
    __device__ __forceinline__ float dot(const float* r) const {
        ExactSum<float> s;
#pragma unroll
        for (int b = 0; b < 9; ++b) {
            s.add(d[b].x, r[b]);
            s.lo = __fmaf_rn(d[b].y, r[b], s.lo);
        }
        return __fadd_rn(s.hi, s.lo);
    }
};

// 16-byte asynchronous copies global -> shared (both addresses 16-byte aligned)
template <typename T>
__device__ __forceinline__ void cp_async16(T* dst, const T* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(static_cast<uint32_t>(__cvta_generic_to_shared(dst))),
                 "l"(src)
                 : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_prev() { asm volatile("cp.async.wait_group 1;" ::: "memory"); }

// ---- bulk copies (cp.async.bulk + mbarrier) --------------------------------------------

// Bounded mbarrier waits: after `polls` unsuccessful polls a wait gives up (polls = 0: at once); the
// kernel then records BA_ERR_TIMEOUT and drains its own copies in flight with the default bound.

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void mbar_init(uint64_t* bar) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void fence_mbar_init() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
// one elected thread: bytes from global src to shared dst, completion counted on bar
__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     smem_u32(dst)),
                 "l"(src), "r"(bytes), "r"(smem_u32(bar))
                 : "memory");
}
// The same copy marked evict-first in L2 (`policy` from l2_evict_first): a stream read once per
// launch then gives way to data that a later kernel reads again.
__device__ __forceinline__ uint64_t l2_evict_first() {
    uint64_t pol;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
    return pol;
}
__device__ __forceinline__ void bulk_load_ef(void* dst, const void* src, uint32_t bytes, uint64_t* bar, uint64_t pol) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;" ::"r"(
            smem_u32(dst)),
        "l"(src), "r"(bytes), "r"(smem_u32(bar)), "l"(pol)
        : "memory");
}
// First statement of the kernels of a solve iteration, which are launched chained (launch_chained):
// such a kernel may be scheduled while the previous kernel on the stream drains (its CTAs retire,
// the implicit trigger), and waits here for that kernel to complete and its writes to be visible.
// Without the chained attribute it returns at once.  (An explicit early trigger, letting the next
// kernel's CTAs take SM resources while this one runs, made the 1936-camera PCG solve slower:
// 4.2 -> 4.8 ms.)
__device__ __forceinline__ void wait_prior_grid() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, int polls) {
    for (int i = 0; i < polls; ++i) {
        uint32_t ok;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(ok)
            : "r"(smem_u32(bar)), "r"(parity)
            : "memory");
        if (ok) return true;
    }
    return false;
}

// Warps per CTA and copy stages of the tile-streaming one-column product, one CTA per SM.  Three
// shapes per precision (ba_options.spmv_config, chosen by ba_autotune); shape 0 is the default:
// float32 16 warps x 1 stage (measured faster than 8 x 2 for the full-pattern product: more warps
// cover the gathers of p), float64 8 x 1: two warps per scheduler keep the float64 pipe busy while one
// waits for its copy (1936 cameras: 0.566 ms, 0.94 of the pipe's rate, against 0.824 ms for 4 x 2 and
// 1.59 ms for 2 x 4; 601 cameras 85 us against 129 us).  Shape 1 has always been 8 x 1 in float64; 4 x 2, the
// default before, is slower from 300 cameras on and no faster below.  The symmetric product does twice the
// arithmetic per tile, so a second stage per warp keeps the next copy in flight during it (shapes 1
// and 2).  Every shape keeps its stages within 207 KB.
template <typename T, int CFG>
struct SpmvShape;
template <> struct SpmvShape<float, 0> { static constexpr int kWarps = 16, kStages = 1; };
template <> struct SpmvShape<float, 1> { static constexpr int kWarps = 8, kStages = 2; };
template <> struct SpmvShape<float, 2> { static constexpr int kWarps = 10, kStages = 2; };
template <> struct SpmvShape<double, 0> { static constexpr int kWarps = 8, kStages = 1; };
template <> struct SpmvShape<double, 1> { static constexpr int kWarps = 8, kStages = 1; };
template <> struct SpmvShape<double, 2> { static constexpr int kWarps = 2, kStages = 4; };
constexpr int kSpmvShapes = 3;
// Shared memory of k_spmv: the warps' tile stages, the stages' barriers, then the warps' row sums.
constexpr int kRowSums = 9 * 33;   // nine sums of 32 lanes, one bank apart
template <typename T, int CFG>
constexpr size_t spmv_smem() {
    return sizeof(T) * SpmvShape<T, CFG>::kWarps * SpmvShape<T, CFG>::kStages * kTileElems +
           sizeof(uint64_t) * SpmvShape<T, CFG>::kWarps * SpmvShape<T, CFG>::kStages +
           sizeof(T) * SpmvShape<T, CFG>::kWarps * kRowSums;
}

// Sum of acc[a] over the warp's lanes in lane a (a < 9; the other lanes return zero).  The sums meet in
// shared memory: three lanes add 11, 11 and 10 of a row's 32 values (two interleaved chains), then
// the three.  Nine shuffle trees cost 45 warp-wide additions, in float64 more than half of the 81
// multiply-adds of a tile; this costs 12.
template <typename T>
__device__ __forceinline__ T row_sums(const T (&acc)[9], T* red) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int a = 0; a < 9; ++a) red[33 * a + lane] = acc[a];
    __syncwarp();
    T v0 = T(0), v1 = T(0);
    if (lane < 27) {
        const T* p = red + 33 * (lane / 3) + 11 * (lane % 3);
#pragma unroll
        for (int u = 0; u < 10; u += 2) {
            v0 += p[u];
            v1 += p[u + 1];
        }
        if (lane % 3 < 2) v0 += p[10];
    }
    __syncwarp();
    const T v = v0 + v1;
    const int from = lane < 9 ? 3 * lane : 0;
    const T s0 = __shfl_sync(0xffffffffu, v, from), s1 = __shfl_sync(0xffffffffu, v, from + 1),
            s2 = __shfl_sync(0xffffffffu, v, from + 2);
    return lane < 9 ? (s0 + s1) + s2 : T(0);
}

// The transposed terms of the symmetric product, one slot per stored upper block: values 0..7 of slot
// e at tb[8 e ..] (one 32-byte sector in float32, written whole by two 16-byte stores, so that L2
// never fills a partly written sector from DRAM) and value 8 at tb[8 n_slots + e].
constexpr int kTbHead = 8;


// One camera's sums q^T p and p^T r (a warp; lanes 0..8 hold the rows, the others zeros) into the two
// slots at camdot.
template <typename T>
__device__ __forceinline__ void camera_dots(int lane, T q, T p, T r, double* camdot) {
    ExactSum<T> dq, dr;
    dq.add(q, p);
    dr.add(p, r);
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) {   // lanes 16..31 hold zeros
        combine_shfl(dq, o);
        combine_shfl(dr, o);
    }
    if (lane == 0) {
        store_partial(camdot, dq);
        store_partial(camdot + 1, dr);
    }
}

// A warp that gives up at item i leaves it and its later ones undone: their problems (of a batch, possibly
// others than the one whose copy was waited for) end with the status at their next decide step.
// (Not inlined, with the list position found again: k_spmm has no register to spare for this path.)
__device__ __noinline__ void report_timeout(Ctl* ctl, const SpItem* items, int sel, int64_t item, int64_t end,
                                            int64_t step) {
    if (threadIdx.x & 31) return;
    for (int64_t i = item; i < end; i += step) {
        const int prob = items[i].prob;
        if (selected(ctl, prob, sel)) atomicExch(&ctl[prob].status, BA_ERR_TIMEOUT);
    }
}

// Tile cursor of a warp: the tiles of its selected items (WarpItems) in order, skipping empty
// items.  The consumer loop selects items with the same predicate, which no kernel changes while
// it runs.
struct TileCursor {
    int64_t item, end, step;
    int t, te;
    int64_t base;
};
__device__ __forceinline__ void cursor_seek(TileCursor& c, const ItemList& L, const int64_t* tile_ptr,
                                            const Ctl* ctl, int sel, int64_t item) {
    for (; item < c.end; item += c.step) {
        const SpItem it = L.items[item];
        if (it.q1 > it.q0 && selected(ctl, it.prob, sel)) {
            c.item = item;
            c.t = it.q0 >> 5;
            c.te = (it.q1 + 31) >> 5;
            c.base = tile_ptr[it.row];
            return;
        }
    }
    c.item = c.end;
    c.t = c.te = 0;
    c.base = 0;
}
__device__ __forceinline__ void cursor_start(TileCursor& c, const ItemList& L, const int64_t* tile_ptr,
                                             const Ctl* ctl, int sel, const WarpItems& wi) {
    c.end = wi.end;
    c.step = wi.step;
    cursor_seek(c, L, tile_ptr, ctl, sel, wi.i0);
}

// y(row, seg) = sum over the item's blocks of S_row,col(q) z_col(q).  Each warp streams the
// tiles of its items through kStages shared-memory buffers with bulk copies (issued by lane 0,
// NS tiles ahead) and multiplies them with the gathered z blocks.
// ZH: z is a column of the problem's direction history (column new_off in MODE 2, column 0
//     otherwise); else z is a vector over all cameras.
// MODE 0: y goes to column new_off + seg of the problem's Q.
// MODE 1 (Algorithm 1): q = y (Q column 0) and, per camera, the sums of q^T p and p^T r
//         (Delta and gamma of Algorithm 1, before the sum over cameras).
// MODE 2 (Algorithm 2, width 1): y goes to column new_off of Q.
// SYM: S is the upper triangle (row j: S_jj, then S_jk for k > j).  Each lane's block also gives the
// transposed term S_jk^T z_j of row k, written to slot cslot[32 tile_ptr[j] + q] of tb/tb8 (the terms
// of column k are consecutive there, in row order), which k_spmv_col adds to row k; in MODE 1 the
// per-camera sums then move to k_spmv_col as well.
template <typename T, int MODE, bool ZH, bool SYM, int CFG>
__global__ void __launch_bounds__(SpmvShape<T, CFG>::kWarps * 32, 1) k_spmv(
    const int64_t* __restrict__ row_ptr, const int64_t* __restrict__ tile_ptr, const int32_t* __restrict__ col,
    const T* __restrict__ S, const T* __restrict__ z, ItemList L, int sel, T* __restrict__ out,
    const T* __restrict__ rvec, double* __restrict__ camdot, Ctl* ctl, T* __restrict__ tb, T* __restrict__ tb8,
    const int32_t* __restrict__ cslot) {
    wait_prior_grid();   // chained launch: the previous kernel's results are visible from here
    constexpr int NW = SpmvShape<T, CFG>::kWarps, NS = SpmvShape<T, CFG>::kStages;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    if (nothing_selected(ctl, L, sel)) return;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    T* tiles = reinterpret_cast<T*>(smem_raw) + size_t(wid) * NS * kTileElems;
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem_raw + sizeof(T) * NW * NS * kTileElems) + wid * NS;
    T* red = reinterpret_cast<T*>(smem_raw + (sizeof(T) * kTileElems + sizeof(uint64_t)) * NW * NS) + wid * kRowSums;
    T* part = static_cast<T*>(L.part);
    constexpr uint32_t tile_bytes = sizeof(T) * kTileElems;

    if (lane == 0) {
        for (int st = 0; st < NS; ++st) mbar_init(&bars[st]);
        fence_mbar_init();
    }
    __syncwarp();
    const WarpItems wi = warp_items(L, NW, wid);
    TileCursor f;
    cursor_start(f, L, tile_ptr, ctl, sel, wi);
    // the symmetric product reads its tiles once and its transposed terms tb again in k_spmv_col:
    // the tiles go first when L2 must evict
    const uint64_t pol = SYM ? l2_evict_first() : 0;
    auto load_tile = [&](int st) {
        T* dst = tiles + st * kTileElems;
        const T* src = S + (f.base + f.t) * kTileElems;
        if (SYM) bulk_load_ef(dst, src, tile_bytes, &bars[st], pol);
        else bulk_load(dst, src, tile_bytes, &bars[st]);
    };
    uint32_t parity = 0, inflight = 0;
    for (int st = 0; st < NS; ++st) {
        if (f.item < f.end) {
            if (lane == 0) load_tile(st);
            inflight |= 1u << st;
            if (++f.t == f.te) cursor_seek(f, L, tile_ptr, ctl, sel, f.item + f.step);
        }
    }
    int stage = 0;
    bool bad = false;
    int bad_item = 0;
    for (int64_t i = wi.i0; i < wi.end && !bad; i += wi.step) {
        const SpItem it = L.items[i];
        if (!selected(ctl, it.prob, sel)) continue;
        const Ctl& c = ctl[it.prob];
        const int64_t n = int64_t(c.lay.nc) * 9;
        const int64_t hb = c.lay.hoff - 9 * int64_t(c.lay.c0);   // history column 0 at global row i: hb + i
        const int64_t zoff = ZH ? hb + int64_t(MODE == 2 ? c.new_off : 0) * n : 0;
        const int64_t ooff = hb + int64_t(MODE == 1 ? 0 : (MODE == 2 ? c.new_off : c.new_off + it.seg)) * n;
        const int64_t rj = row_ptr[it.row];
        const int64_t tb0 = SYM ? tile_ptr[it.row] * kTile : 0;   // tiled index of the row's first block
        T acc[9];
#pragma unroll
        for (int a = 0; a < 9; ++a) acc[a] = T(0);
        T zr[9];   // SYM: z of the row camera, the factor of every transposed term of the item
#pragma unroll
        for (int b = 0; b < 9; ++b) zr[b] = SYM ? z[zoff + 9 * int64_t(it.row) + b] : T(0);
        if (it.q1 > it.q0) {
            const int t0 = it.q0 >> 5, t1 = (it.q1 + 31) >> 5;
            // the 9 entries of z this lane needs for tile t (and SYM: the slot of its transposed
            // term, -1 for none), fetched one tile ahead
            T zn[9];
            int csn = -1;
            {
                const int q = t0 * 32 + lane;
                const bool in = q >= it.q0 && q < it.q1;
                const T* zk = z + zoff + int64_t(in ? col[rj + q] : it.row) * 9;
#pragma unroll
                for (int b = 0; b < 9; ++b) zn[b] = in ? zk[b] : T(0);
                if (SYM && in) csn = cslot[tb0 + q];
            }
            for (int t = t0; t < t1; ++t) {
                T zv[9];
#pragma unroll
                for (int b = 0; b < 9; ++b) zv[b] = zn[b];
                const int csv = csn;
                if (t + 1 < t1) {
                    const int qn = (t + 1) * 32 + lane;
                    const bool in = qn < it.q1;
                    const T* zk = z + zoff + int64_t(in ? col[rj + qn] : it.row) * 9;
#pragma unroll
                    for (int b = 0; b < 9; ++b) zn[b] = in ? zk[b] : T(0);
                    csn = SYM && in ? cslot[tb0 + qn] : -1;
                }
                // every lane observes the phase (visibility of the copied bytes); the warp agrees
                const bool ok = mbar_wait(&bars[stage], (parity >> stage) & 1u, L.polls);
                if (!__all_sync(0xffffffffu, ok)) {
                    bad = true;
                    bad_item = int(i);
                    break;
                }
                parity ^= 1u << stage;
                inflight &= ~(1u << stage);
                const T* tile = tiles + stage * kTileElems;
                const int q = t * 32 + lane;
                const bool inq = q >= it.q0 && q < it.q1;
                if (SYM) {
                    T v[9];
#pragma unroll
                    for (int b = 0; b < 9; ++b) v[b] = T(0);
                    if (inq) {
                        const T* blk = tile + lane * 81;
#pragma unroll
                        for (int a = 0; a < 9; ++a)
#pragma unroll
                            for (int b = 0; b < 9; ++b) {
                                const T sab = blk[9 * a + b];
                                acc[a] += sab * zv[b];
                                v[b] += sab * zr[a];
                            }
                    }
                    // q = 0 is S_jj, whose row term covers it (its slot is -1)
                    if (csv >= 0) {
                        T* dst = tb + int64_t(csv) * kTbHead;
                        if constexpr (sizeof(T) == 4) {
                            reinterpret_cast<float4*>(dst)[0] = make_float4(v[0], v[1], v[2], v[3]);
                            reinterpret_cast<float4*>(dst)[1] = make_float4(v[4], v[5], v[6], v[7]);
                        } else {
#pragma unroll
                            for (int b = 0; b < 8; ++b) dst[b] = v[b];
                        }
                        tb8[csv] = v[8];
                    }
                } else if (inq) {
                    const T* blk = tile + lane * 81;
#pragma unroll
                    for (int a = 0; a < 9; ++a)
#pragma unroll
                        for (int b = 0; b < 9; ++b) acc[a] += blk[9 * a + b] * zv[b];
                }
                __syncwarp();
                if (f.item < f.end) {
                    fence_proxy_async();
                    if (lane == 0) load_tile(stage);
                    inflight |= 1u << stage;
                    if (++f.t == f.te) cursor_seek(f, L, tile_ptr, ctl, sel, f.item + f.step);
                }
                stage = stage + 1 == NS ? 0 : stage + 1;
            }
            if (bad) break;
        }
        T val = row_sums(acc, red);
        bool fin = true;
        if (it.ng > 1) {
            if (lane < 9) part[int64_t(it.slot) * 9 + lane] = val;
            __threadfence();
            int last = 0;
            if (lane == 0) last = (atomicAdd(L.cnt + it.grp, 1) == it.ng - 1);
            last = __shfl_sync(0xffffffffu, last, 0);
            fin = last != 0;
            if (fin) {
                __threadfence();
                T sum = T(0);
                const int64_t first = int64_t(it.slot) - it.k;
                if (lane < 9)
                    for (int cc = 0; cc < it.ng; ++cc) sum += __ldcg(part + (first + cc) * 9 + lane);
                val = sum;
                if (lane == 0) L.cnt[it.grp] = 0;
            }
        }
        if (fin) {
            const int64_t rowi = 9 * int64_t(it.row) + lane;
            if (lane < 9) out[ooff + rowi] = val;
            if (MODE == 1 && !SYM)
                camera_dots(lane, lane < 9 ? val : T(0), lane < 9 ? z[zoff + rowi] : T(0),
                            lane < 9 ? rvec[rowi] : T(0), camdot + 2 * int64_t(it.row));
        }
    }
    if (bad) {
        // a copy did not land in time: report, then wait (bounded) for this warp's copies in flight;
        // the problem's next decide step ends it with the status
        const WarpItems left = warp_items(L, NW, wid);
        report_timeout(ctl, L.items, sel, bad_item, left.end, left.step);
        for (int st = 0; st < NS; ++st)
            if (inflight & (1u << st)) mbar_wait(&bars[st], (parity >> st) & 1u, kDefaultWaitPolls);
    }
}

// Second pass of the symmetric product: y_k += sum over the stored blocks (j, k), j < k, of their
// transposed terms S_jk^T z_j (a fixed order: lane-strided sums in each warp's share of the column's
// slots, then the warps' sums in warp order), then in MODE 1 the per-camera sums q^T p and p^T r.
// One CTA of kColWarps warps per camera (its slots qptr[k] .. qptr[k + 1] - 1 of tb are consecutive,
// up to n_c - 1 of them); grid: CTAs x problems.  CTAs take the cameras from the last one down:
// camera k's column holds the blocks (j, k), j < k, so on a dense pattern the long columns start
// in the first wave and the short ones fill the tail.
constexpr int kColWarps = 4;   // 12 CTAs per SM: 1824 cameras in flight
template <typename T, int MODE, bool ZH>
__global__ void __launch_bounds__(kColWarps * 32, 12) k_spmv_col(const int64_t* __restrict__ qptr,
                                                             const T* __restrict__ tb, const T* __restrict__ tb8,
                                                             const T* __restrict__ z, int sel, T* __restrict__ out,
                                                             const T* __restrict__ rvec, double* __restrict__ camdot,
                                                             const Ctl* __restrict__ ctl) {
    wait_prior_grid();   // chained launch: the previous kernel's results are visible from here
    const int p = blockIdx.y;
    if (!selected(ctl, p, sel)) return;
    const Ctl& c = ctl[p];
    __shared__ T red[kColWarps][9];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int64_t n = int64_t(c.lay.nc) * 9;
    const int64_t hb = c.lay.hoff - 9 * int64_t(c.lay.c0);
    const int64_t zoff = ZH ? hb + int64_t(MODE == 2 ? c.new_off : 0) * n : 0;
    const int64_t ooff = hb + int64_t(MODE == 1 ? 0 : c.new_off) * n;
    for (int64_t jr = blockIdx.x; jr < c.lay.nc; jr += gridDim.x) {
        const int64_t j = c.lay.c0 + (c.lay.nc - 1 - jr);
        T acc[9];
#pragma unroll
        for (int b = 0; b < 9; ++b) acc[b] = T(0);
        // warp w takes slots w * 32 + lane + k * kColWarps * 32, four per lane in flight (slots past
        // the end add exact zeros)
        constexpr int step = kColWarps * 32;
        const int64_t e1 = qptr[j + 1];
        for (int64_t e = qptr[j] + wid * 32 + lane; e < e1; e += 4 * step) {
            T v[4][9];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int64_t eu = e + u * step;
                const T* t = tb + eu * kTbHead;
                if (eu < e1) {
                    if constexpr (sizeof(T) == 4) {
                        const float4 a = reinterpret_cast<const float4*>(t)[0];
                        const float4 c = reinterpret_cast<const float4*>(t)[1];
                        v[u][0] = a.x, v[u][1] = a.y, v[u][2] = a.z, v[u][3] = a.w;
                        v[u][4] = c.x, v[u][5] = c.y, v[u][6] = c.z, v[u][7] = c.w;
                    } else {
#pragma unroll
                        for (int b = 0; b < 8; ++b) v[u][b] = t[b];
                    }
                    v[u][8] = tb8[eu];
                } else {
#pragma unroll
                    for (int b = 0; b < 9; ++b) v[u][b] = T(0);
                }
            }
#pragma unroll
            for (int b = 0; b < 9; ++b) acc[b] += (v[0][b] + v[1][b]) + (v[2][b] + v[3][b]);
        }
#pragma unroll
        for (int b = 0; b < 9; ++b) acc[b] = warp_sum(acc[b]);
        if (lane == 0)
#pragma unroll
            for (int b = 0; b < 9; ++b) red[wid][b] = acc[b];
        __syncthreads();
        if (wid == 0) {
            T val = T(0);
            if (lane < 9) {
                val = red[0][lane];
#pragma unroll
                for (int w = 1; w < kColWarps; ++w) val += red[w][lane];
            }
            const int64_t rowi = 9 * j + lane;
            if (lane < 9) {
                val = out[ooff + rowi] + val;
                out[ooff + rowi] = val;
            }
            if (MODE == 1)
                camera_dots(lane, lane < 9 ? val : T(0), lane < 9 ? z[zoff + rowi] : T(0),
                            lane < 9 ? rvec[rowi] : T(0), camdot + 2 * j);
        }
        __syncthreads();
    }
}

// Q[:, new_off + c] = S P[:, new_off + c] for the w > 1 columns of a new local block (Algorithm 2,
// used by the float32 sweeps, where the Eq. 18 update cancels).  Tiles stream through
// shared memory as in k_spmv; CL lanes share a block (CL = 4, or 2 when no block is wider than 8
// columns): lane = CL qi + g takes tile-local blocks qi, qi + 32 / CL, ... and columns
// 4g .. 4g + 3, so each 9x9 block multiplies up to 4 CL columns per read from shared memory.  No unit is at
// its limit (1000 dense cameras: L1 and shared memory 65 %, DRAM 43 %, issue 36 %); a warp waits most for its P
// gathers, then for its 81 words of S and 36 of P per 324 multiply-adds.  Lanes left without columns wait like
// the others: N = 8 on 1000 dense cameras took 94 us per local step with four lanes a block and takes 75 us
// with two (one lane for N = 4: 76 us).  PT is the row-major copy (9 n_c x 16, all problems) of the new blocks.
// The multi-column product waits on L2 gathers of PT more than on its tiles, so it runs twice
// the warps of k_spmv with one tile stage each (the other warps' copies and arithmetic cover a
// warp's wait for its next tile); at most 128 registers a thread.
struct SpmmCfg {
    static constexpr int kWarps = 16, kStages = 1;
};
template <typename T>
constexpr size_t spmm_tiles_smem() {
    return sizeof(T) * SpmmCfg::kWarps * SpmmCfg::kStages * kTileElems +
           sizeof(uint64_t) * SpmmCfg::kWarps * SpmmCfg::kStages;
}
template <typename T>
constexpr size_t spmm_smem() {
    return spmm_tiles_smem<T>() + sizeof(T) * SpmmCfg::kWarps * kMaxDirs * 9;
}

// rows b = 0..8 of a 16-column PT block, 4 columns from p: (p[16 b], p[16 b + 1]) and
// (p[16 b + 2], p[16 b + 3]) as float pairs (one 16-byte load per row)
__device__ __forceinline__ void load_prow(const float* p, float2 (&v)[9][2]) {
#pragma unroll
    for (int b = 0; b < 9; ++b) {
        const float4 t = *reinterpret_cast<const float4*>(p + b * kMaxDirs);
        v[b][0] = make_float2(t.x, t.y);
        v[b][1] = make_float2(t.z, t.w);
    }
}

template <typename T, int CL>
__global__ void __launch_bounds__(SpmmCfg::kWarps * 32, 1) k_spmm(
    const int64_t* __restrict__ row_ptr, const int64_t* __restrict__ tile_ptr, const int32_t* __restrict__ col,
    const T* __restrict__ S, const T* __restrict__ PT, ItemList L, T* __restrict__ part, T* __restrict__ Q,
    Ctl* ctl) {
    wait_prior_grid();   // chained launch: the previous kernel's results are visible from here
    static_assert(sizeof(T) == 4, "the multi-column product serves the float32 sweeps");
    constexpr int NW = SpmmCfg::kWarps, NS = SpmmCfg::kStages;
    constexpr int sel = kSelWide;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    if (nothing_selected(ctl, L, sel)) return;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    constexpr int NBK = 32 / CL;   // blocks per round
    const int qi = lane / CL, g = lane % CL;
    T* tiles = reinterpret_cast<T*>(smem_raw) + size_t(wid) * NS * kTileElems;
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem_raw + sizeof(T) * NW * NS * kTileElems) + wid * NS;
    T* red = reinterpret_cast<T*>(smem_raw + spmm_tiles_smem<T>()) + wid * (kMaxDirs * 9);
    constexpr uint32_t tile_bytes = sizeof(T) * kTileElems;
    if (lane == 0) {
        for (int st = 0; st < NS; ++st) mbar_init(&bars[st]);
        fence_mbar_init();
    }
    __syncwarp();
    const WarpItems wi = warp_items(L, NW, wid);
    TileCursor f;
    cursor_start(f, L, tile_ptr, ctl, sel, wi);
    uint32_t parity = 0, inflight = 0;
    for (int st = 0; st < NS; ++st) {
        if (f.item < f.end) {
            if (lane == 0) bulk_load(tiles + st * kTileElems, S + (f.base + f.t) * kTileElems, tile_bytes, &bars[st]);
            inflight |= 1u << st;
            if (++f.t == f.te) cursor_seek(f, L, tile_ptr, ctl, sel, f.item + f.step);
        }
    }
    int stage = 0;
    bool bad = false;
    int bad_item = 0;
    for (int64_t i = wi.i0; i < wi.end && !bad; i += wi.step) {
        const SpItem it = L.items[i];
        if (!selected(ctl, it.prob, sel)) continue;
        const Ctl& c = ctl[it.prob];
        const int w = c.w_new;
        const int nout = 9 * w;
        const int64_t n = int64_t(c.lay.nc) * 9;
        const int64_t ooff = c.lay.hoff - 9 * int64_t(c.lay.c0) + int64_t(c.new_off) * n;
        const int64_t rj = row_ptr[it.row];
        // columns (4g, 4g + 1) and (4g + 2, 4g + 3) of the 9 rows, as float pairs for the packed
        // float32 multiply-add (each pair operation rounds like two scalar fused multiply-adds)
        float2 acc[9][2];
#pragma unroll
        for (int a = 0; a < 9; ++a) acc[a][0] = acc[a][1] = make_float2(0.f, 0.f);
        if (it.q1 > it.q0) {
            const int t0 = it.q0 >> 5, t1 = (it.q1 + 31) >> 5;
            const bool active = 4 * g < w;
            // column cameras of this lane's blocks r NBK + qi (r < CL) of tile t, -1 outside the
            // item; fetched one tile ahead.  The P rows of a block are gathered right before its
            // arithmetic: the other warps of the SM cover the wait
            int kc[CL], kn[CL];
#pragma unroll
            for (int r = 0; r < CL; ++r) {
                const int q = t0 * 32 + r * NBK + qi;
                kc[r] = (active && q >= it.q0 && q < it.q1) ? col[rj + q] : -1;
            }
            float2 pv[9][2];
            for (int t = t0; t < t1; ++t) {
#pragma unroll
                for (int r = 0; r < CL; ++r) {
                    const int q = (t + 1) * 32 + r * NBK + qi;
                    kn[r] = (active && t + 1 < t1 && q < it.q1) ? col[rj + q] : -1;
                }
                const bool ok = mbar_wait(&bars[stage], (parity >> stage) & 1u, L.polls);
                if (!__all_sync(0xffffffffu, ok)) {
                    bad = true;
                    bad_item = int(i);
                    break;
                }
                parity ^= 1u << stage;
                inflight &= ~(1u << stage);
                const T* tile = tiles + stage * kTileElems;
                if (active) {
#pragma unroll
                    for (int r = 0; r < CL; ++r) {
                        if (kc[r] < 0) continue;
                        // rows 9k .. 9k + 8, columns 4g .. 4g + 3 of PT for this block
                        load_prow(PT + (int64_t(kc[r]) * 9) * kMaxDirs + 4 * g, pv);
                        const T* blk = tile + (r * NBK + qi) * 81;
#pragma unroll
                        for (int a = 0; a < 9; ++a)
#pragma unroll
                            for (int b = 0; b < 9; ++b) {
                                const float sab = blk[9 * a + b];
                                const float2 s2 = make_float2(sab, sab);
                                acc[a][0] = __ffma2_rn(s2, pv[b][0], acc[a][0]);
                                acc[a][1] = __ffma2_rn(s2, pv[b][1], acc[a][1]);
                            }
                    }
                }
#pragma unroll
                for (int r = 0; r < CL; ++r) kc[r] = kn[r];
                __syncwarp();
                if (f.item < f.end) {
                    fence_proxy_async();
                    if (lane == 0)
                        bulk_load(tiles + stage * kTileElems, S + (f.base + f.t) * kTileElems, tile_bytes, &bars[stage]);
                    inflight |= 1u << stage;
                    if (++f.t == f.te) cursor_seek(f, L, tile_ptr, ctl, sel, f.item + f.step);
                }
                stage = stage + 1 == NS ? 0 : stage + 1;
            }
            if (bad) break;
        }
        // sum over the NBK lanes of each column group, then lanes 0 .. CL - 1 hold their columns
        T accs[9][4];
#pragma unroll
        for (int a = 0; a < 9; ++a) {
            accs[a][0] = acc[a][0].x;
            accs[a][1] = acc[a][0].y;
            accs[a][2] = acc[a][1].x;
            accs[a][3] = acc[a][1].y;
        }
#pragma unroll
        for (int a = 0; a < 9; ++a)
#pragma unroll
            for (int cc = 0; cc < 4; ++cc) {
                T v = accs[a][cc];
#pragma unroll
                for (int o = CL; o < 32; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
                accs[a][cc] = v;
            }
        __syncwarp();
        if (qi == 0) {
#pragma unroll
            for (int cc = 0; cc < 4; ++cc) {
                const int ci = 4 * g + cc;
                if (ci < w)
#pragma unroll
                    for (int a = 0; a < 9; ++a) red[ci * 9 + a] = accs[a][cc];
            }
        }
        __syncwarp();
        bool fin = true;
        if (it.ng > 1) {
            for (int o = lane; o < nout; o += 32) part[int64_t(it.slot) * (kMaxDirs * 9) + o] = red[o];
            __threadfence();
            int last = 0;
            if (lane == 0) last = (atomicAdd(L.cnt + it.grp, 1) == it.ng - 1);
            last = __shfl_sync(0xffffffffu, last, 0);
            fin = last != 0;
            if (fin) {
                __threadfence();
                const int64_t first = int64_t(it.slot) - it.k;
                for (int o = lane; o < nout; o += 32) {
                    T sum = T(0);
                    for (int cc = 0; cc < it.ng; ++cc) sum += __ldcg(part + (first + cc) * (kMaxDirs * 9) + o);
                    red[o] = sum;
                }
                __syncwarp();
                if (lane == 0) L.cnt[it.grp] = 0;
            }
        }
        if (fin) {
            for (int o = lane; o < nout; o += 32) {
                const int ci = o / 9, a = o % 9;
                Q[ooff + int64_t(ci) * n + 9 * int64_t(it.row) + a] = red[o];
            }
        }
        __syncwarp();
    }
    if (bad) {
        const WarpItems left = warp_items(L, NW, wid);
        report_timeout(ctl, L.items, sel, bad_item, left.end, left.step);
        for (int st = 0; st < NS; ++st)
            if (inflight & (1u << st)) mbar_wait(&bars[st], (parity >> st) & 1u, kDefaultWaitPolls);
    }
}

// ---------------------------------------------------------------------------------------
// initialisation shared by both algorithms: x = 0, r = sign * rhs, z = D^{-1} r, P_0 = z
// (grid: update CTAs x problems; thread = row, as in the update kernels; partial: one slot per CTA).
// outer (mixed precision, may be null): r is divided by the sweep's unit, a power of two near its largest value,
// so that a sweep starts with that in [1, 4) whatever the residual's size and the units of the cameras and
// landmarks (the error terms of its float32 sums, and Delta^+ in double-float, would otherwise leave the
// float32 range on late sweeps, or on the first one of a scene with coordinates of 1e-9).

template <typename T>
__global__ void __launch_bounds__(kUpdThreads) k_init_vec(const Layout* __restrict__ lay, const double* __restrict__ rhs,
                                                          double sign, const double* __restrict__ scale,
                                                          const double* __restrict__ Dinv, const Outer* __restrict__ outer,
                                                          T* __restrict__ x, T* __restrict__ r, T* __restrict__ z,
                                                          T* __restrict__ P, WideSlot<T>* __restrict__ partial) {
    const Layout L = lay[blockIdx.y];
    __shared__ T sr[kUpdCams * 9];
    const int t = threadIdx.x, cl = t / 9, a = t - 9 * (t / 9);
    const int64_t jl = int64_t(blockIdx.x) * kUpdCams + cl;
    const bool act = t < kUpdCams * 9 && jl < L.nc;
    const int64_t i = 9 * (L.c0 + jl) + a;
    if (outer) sign /= outer[blockIdx.y].unit;
    DinvRow<T> D;
    D.load(Dinv + 9 * i, act);
    T rv = T(0);
    if (act) {
        rv = T(sign * (scale ? scale[i] : 1.0) * rhs[i]);
        r[i] = rv;
        x[i] = T(0);
    }
    if (t < kUpdCams * 9) sr[t] = rv;
    ExactSum<T> v[1];
    v[0].add(rv, rv);
    __syncthreads();
    if (act) {
        const T zs = D.dot(sr + 9 * cl);
        z[i] = zs;
        P[L.hoff + 9 * jl + a] = zs;
    }
    cta_publish<T, 1>(v, partial + int64_t(blockIdx.y) * gridDim.x);
}

// Which problems k_one_cta (mixed precision) and k_pcg_cluster (float64 PCG) solve; their comments say why.
constexpr int kOneCams = 20, kOneDirs = 10, kCluCams = 24;
__host__ __device__ __forceinline__ bool solved_alone(const Layout& L, bool fp32, bool mcg) {
    return fp32 ? L.nc <= kOneCams && (!mcg || L.n_eff <= kOneDirs) : L.nc <= kCluCams && !mcg;
}

// One warp per problem.  outer (mixed precision, may be null) supplies the sweep's tolerance and
// iteration budget and leaves the problems that are not refined any more done from the start.  small: mark the
// problems that are solved alone; they are done for the kernels of the iterations.
template <typename T>
__global__ void k_init_ctl(Ctl* ctl, const Layout* __restrict__ lay, const WideSlot<T>* __restrict__ partial, int np,
                           const Params* __restrict__ prm, double stag, int direct_q,
                           const Outer* __restrict__ outer, int* blk_off, int* blk_w, int mi1, int small) {
    const int p = blockIdx.x;
    const double rr0 = warp_sum_slots<T>(partial + int64_t(p) * np, np).value();
    if (threadIdx.x == 0) {
        Ctl c;
        memset(&c, 0, sizeof(c));
        c.lay = lay[p];
        double tl = prm->tol;
        const double tau = prm->tau;
        int mi = prm->max_iters;
        bool act = true;
        c.hist_off = 0;
        c.hist_scale = 1.0;
        if (outer) {
            const Outer& o = outer[p];
            act = o.swept != 0;
            tl = o.tol_in;
            mi = o.max_in;
            c.hist_off = o.iters;
            c.hist_scale = o.bb > 0.0 ? o.tr / o.bb : 0.0;
        }
        c.rr0 = rr0;
        c.rr0_inv = rr0 > 0.0 ? 1.0 / rr0 : 0.0;
        c.rr = rr0;
        c.tol2 = tl * tl;
        c.tau = tau;
        c.max_iters = mi;
        c.n_eff = c.lay.n_eff;
        c.sz = c.lay.sz;
        c.K = c.lay.K;
        c.cap = c.lay.cap;
        c.cols = 1;
        c.w_new = 1;
        c.new_off = 0;
        c.local = 0;
        c.w_cur = 1;
        c.off_cur = 0;
        c.stag = stag;
        c.direct_q = direct_q;
        c.status = BA_OK;
        if (!act) { c.done = 1; }
        else if (!(rr0 == rr0) || isinf(rr0)) { c.done = 1; c.status = BA_ERR_BREAKDOWN; }
        else if (rr0 == 0.0 || mi <= 0) { c.done = 1; c.status = rr0 == 0.0 ? BA_OK : BA_ERR_NOT_CONVERGED; }
        if (small && !c.done && solved_alone(c.lay, sizeof(T) == 4, prm->mcg != 0)) c.alone = c.done = 1;
        ctl[p] = c;
        blk_off[int64_t(p) * mi1] = 0;
        blk_w[int64_t(p) * mi1] = 1;
    }
}

// Condition of the Krylov WHILE loop: continue while a problem is not done.  first = 1 (before the
// loop) starts the sweep's pass count; otherwise one body pass has ended.  `bound` passes (every
// problem stops by its iteration budget well before) end the loop in any case.  use_handle = 0 when
// the loop runs from the host (the kernel then only counts).
__global__ void k_loop_cond(cudaGraphConditionalHandle h, int use_handle, const Ctl* __restrict__ ctl, int nb,
                            Loops* lp, int first, int chunk, const Params* __restrict__ prm) {
    wait_prior_grid();   // chained launch: the previous kernel's results are visible from here
    __shared__ int any;
    if (threadIdx.x == 0) any = 0;
    __syncthreads();
    int mine = 0;
    for (int b = threadIdx.x; b < nb; b += blockDim.x) mine |= ctl[b].done == 0;
    if (mine) atomicOr(&any, 1);
    __syncthreads();
    if (threadIdx.x == 0) {
        int go = any;
        if (first) {
            lp->cur = 0;
        } else {
            lp->cur += 1;
            lp->inner += 1;
        }
        const int bound = (prm->max_iters + chunk - 1) / chunk + 2;
        if (lp->cur >= bound) {
            if (go) lp->capped = 1;
            go = 0;
        }
        if (use_handle) cudaGraphSetConditional(h, go ? 1u : 0u);
    }
}

// Nearest float32 of a float64 p > 0 in float32's normal range, and the float64 equal to such a float32,
// from their bit patterns: the conversion instructions run on the float64 pipe (about 150 cycles each),
// this on the integer pipe.
__device__ __forceinline__ float bits_to_f32(double p) {
    return __int_as_float(int(((__double_as_longlong(p) + (1ll << 28)) >> 29) - (896ll << 23)));
}
__device__ __forceinline__ double bits_to_f64(float r) {
    return __longlong_as_double((static_cast<long long>(__float_as_int(r)) + (896ll << 23)) << 29);
}

// 1 / p in float64 without the long division chain (an exact float64 division is a dependent
// sequence of about ten operations on this GPU's narrow float64 pipe): a float32 estimate
// (relative error below 2^-23) refined by Newton steps r <- r + r (1 - p r), each of which
// squares the error: one step leaves it below 2^-46 (about 1e-14), two reach float64 rounding.
// Values that are not positive or outside 2^-100 .. 2^100 divide.
template <int kSteps = 1>
__device__ __forceinline__ double fast_rcp(double p) {
    const int e = __double2hiint(p);   // sign, exponent and high fraction bits
    if (!(e >= ((1023 - 100) << 20) && e < ((1023 + 100) << 20))) return 1.0 / p;
    double r = bits_to_f64(__frcp_rn(bits_to_f32(p)));
#pragma unroll
    for (int k = 0; k < kSteps; ++k) r = fma(r, fma(-p, r, 1.0), r);
    return r;
}

// ---------------------------------------------------------------------------------------
// Algorithm 1 (grid: CTAs x problems)

// The sums over cameras [0, nc) of the per-camera sums (Delta, gamma), returned to every thread of
// the CTA: thread t takes cameras t + 128 k, eight loads in flight, then shuffle trees and the warps in
// order.  (Four dependent rounds of loads, one value per warp, took 2.6 us for 1000 cameras.)
template <typename T>
__device__ __forceinline__ void sum_camdot(const double* cd, int nc, ExactSum<T>& Delta, ExactSum<T>& gamma) {
    __shared__ __align__(16) double sh[2 * (kUpdThreads / 32)];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    ExactSum<T> d, g, d1, g1;
    for (int j = threadIdx.x; j < nc; j += 8 * kUpdThreads) {
        double2 v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u)
            v[u] = j + u * kUpdThreads < nc ? *reinterpret_cast<const double2*>(cd + 2 * int64_t(j + u * kUpdThreads))
                                            : make_double2(0.0, 0.0);
#pragma unroll
        for (int u = 0; u < 8; u += 2) {
            if (j + u * kUpdThreads < nc) {
                add_slot(d, v[u].x);
                add_slot(g, v[u].y);
            }
            if (j + (u + 1) * kUpdThreads < nc) {
                add_slot(d1, v[u + 1].x);
                add_slot(g1, v[u + 1].y);
            }
        }
    }
    combine(d, d1);
    combine(g, g1);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        combine_shfl(d, o);
        combine_shfl(g, o);
    }
    if (lane == 0) {
        store_partial(&sh[2 * wid], d);
        store_partial(&sh[2 * wid + 1], g);
    }
    __syncthreads();
#pragma unroll
    for (int w = 0; w < kUpdThreads / 32; ++w) {
        load_partial(Delta, &sh[2 * w]);
        load_partial(gamma, &sh[2 * w + 1]);
    }
}

// alpha = gamma / Delta; x += alpha p; r -= alpha q; z = D^{-1} r; per CTA the sums of |r|^2, q^T z and
// r^T z (dpart), from which k_pcg_dir takes the stop test and beta; dtot: Delta and gamma.
// Delta and gamma are the sums over the problem's cameras (camera order) of the per-camera sums
// of the product; every CTA forms them the same way.
// Thread = one row (9 per camera, kUpdCams cameras per CTA); the rows of a camera meet in
// shared memory for z = D^{-1} r.  CTA b of a problem takes its cameras [b kUpdCams, ...), so the
// partition depends on the problem alone (the grid has a CTA for every chunk of the largest).
// Bound by latency: on 1000 cameras 12 us of a 22 us iteration when the sums ran in float64 (whose
// pipe does 1.7 lanes per clock and SM, so each warp-wide addition of a shuffle tree costs as much as
// a full one); 8.6 us with the float32 sweeps' sums on the float32 pipe; 3.4 us with the camera sums' loads in
// flight together and the decide step in k_pcg_dir.
// Every CTA reads all camera sums, 16 n ceil(n / 14) bytes an iteration: 4 MB of L2 reads at 1936 cameras and
// 1 GB at 30,000, where an iteration on a banded S takes 193 us (311 us with 28 cameras a CTA and float64 sums).
template <typename T>
__global__ void __launch_bounds__(kUpdThreads) k_pcg_update(const double* __restrict__ Dinv, const T* __restrict__ P,
                                                            const T* __restrict__ Q, T* __restrict__ x,
                                                            T* __restrict__ r, T* __restrict__ z,
                                                            const double* __restrict__ camdot,
                                                            WideSlot<T>* __restrict__ dpart,
                                                            double* __restrict__ dtot, Ctl* ctl) {
    wait_prior_grid();   // chained launch: the previous kernel's results are visible from here
    const int p = blockIdx.y;
    const Ctl& c = ctl[p];
    if (blockIdx.x == 0 && threadIdx.x == 0) ctl[p].live = !c.done;
    if (c.done) return;
    const int64_t c0 = c.lay.c0;
    const int nc = c.lay.nc;
    if (int64_t(blockIdx.x) * kUpdCams >= nc) return;   // no camera (a smaller problem of the batch)
    __shared__ T sr[kUpdCams * 9];
    const int t = threadIdx.x, cl = t / 9, a = t - 9 * (t / 9);
    const int64_t jl = int64_t(blockIdx.x) * kUpdCams + cl;
    const bool act = t < kUpdCams * 9 && jl < nc;
    const int64_t hb = c.lay.hoff - 9 * c0;
    const int64_t i = 9 * (c0 + jl) + a;
    // this row's operands, requested before the CTA waits for the camera sums
    DinvRow<T> D;
    D.load(Dinv + 9 * i, act);
    const T pv = act ? P[hb + i] : T(0), qv = act ? Q[hb + i] : T(0);
    const T xv = act ? x[i] : T(0), r0 = act ? r[i] : T(0);
    ExactSum<T> Delta, gamma;
    sum_camdot<T>(camdot + 2 * c0, nc, Delta, gamma);
    // alpha = gamma / Delta; the float32 sweeps divide the rounded operands in float32 (a float64
    // division is a long dependent chain on this GPU's narrow float64 pipe)
    T alpha;
    if constexpr (sizeof(T) == 4) alpha = __fdiv_rn(__fadd_rn(gamma.hi, gamma.lo), __fadd_rn(Delta.hi, Delta.lo));
    else alpha = gamma.s * fast_rcp<2>(Delta.s);
    ExactSum<T> v[3];
    T rv = T(0);
    if (act) {
        x[i] = xv + alpha * pv;
        rv = r0 - alpha * qv;
        r[i] = rv;
        v[0].add(rv, rv);
    }
    if (t < kUpdCams * 9) sr[t] = rv;
    __syncthreads();
    if (act) {
        const T zs = D.dot(sr + 9 * cl);
        z[i] = zs;
        v[1].add(qv, zs);
        v[2].add(rv, zs);
    }
    cta_publish<T, 3>(v, dpart + int64_t(p) * gridDim.x * 3);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        store_partial(dtot + 2 * int64_t(p), Delta);
        store_partial(dtot + 2 * int64_t(p) + 1, gamma);
    }
}

// stop test for problem p (one thread); hist is iteration-major (it x nb), null: not written
__device__ void pcg_decide(Ctl* c, double D, double g, const double* tot, double* hist, int p, int nb) {
    if (c->status == BA_ERR_TIMEOUT) { c->done = 1; return; }
    const double rr = tot[0];
    const int it = c->it + 1;
    c->it = it;
    c->rr = rr;
    if (hist) hist[int64_t(c->hist_off + it - 1) * nb + p] = rr * c->rr0_inv * c->hist_scale;   // squared relative residual
    if (!(D > 0.0) || !(rr == rr) || isinf(rr)) {
        c->done = 1;
        c->status = BA_ERR_BREAKDOWN;
    } else if (rr < c->tol2 * c->rr0) {
        c->done = 1;
        c->status = BA_OK;
    } else if (it >= c->max_iters) {
        c->done = 1;
        c->status = BA_ERR_NOT_CONVERGED;
    } else if (c->stag > 0.0 && g * g < c->stag * tot[2] * D) {   // (g^2 / D) / r^T z < stag
        c->done = 1;          // no measurable progress left at this precision: end the sweep
        c->status = BA_OK;
    }
}

// beta = Phi / Delta and p = z - beta p (rows of the problem).  Every CTA adds the update's partials (gu
// slots of three per problem) and forms beta; the first CTA of a problem also runs the stop test, in
// another warp than beta (a problem that ends there gets one more direction, which nothing reads).
template <typename T>
__global__ void __launch_bounds__(kThreads) k_pcg_dir(const T* __restrict__ z, T* __restrict__ P,
                                                      const WideSlot<T>* __restrict__ dpart, int gu,
                                                      const double* __restrict__ dtot, double* __restrict__ hist,
                                                      Ctl* ctl) {
    wait_prior_grid();   // chained launch: the previous kernel's results are visible from here
    const int p = blockIdx.y;
    const Ctl& c = ctl[p];
    if (!c.live) return;
    const int nc = c.lay.nc;
    const int64_t n = int64_t(nc) * 9, r0 = 9 * int64_t(c.lay.c0);
    if (int64_t(blockIdx.x) * blockDim.x >= n) return;
    __shared__ double tot[3];
    __shared__ T sbeta;
    T* Pp = P + c.lay.hoff;
    int64_t i = gtid();
    T zv = T(0), pv = T(0);
    if (i < n) {   // requested before the CTA waits for the sums
        zv = z[r0 + i];
        pv = Pp[i];
    }
    ExactSum<T> D, g;
    load_partial(D, dtot + 2 * int64_t(p));
    load_partial(g, dtot + 2 * int64_t(p) + 1);
    const int wid = threadIdx.x >> 5;
    if (wid == 1 || (wid < 3 && blockIdx.x == 0)) {   // every CTA needs q^T z, the stop test the others
        const WideSum<T> s = total_of<T, 3>(dpart + int64_t(p) * gu * 3, (nc + kUpdCams - 1) / kUpdCams, wid);
        if ((threadIdx.x & 31) == 0) tot[wid] = s.value();
        if (wid == 1 && (threadIdx.x & 31) == 0) sbeta = T(s.value() * fast_rcp<2>(D.value()));
    }
    __syncthreads();
    if (blockIdx.x == 0 && threadIdx.x == 32 * 7) pcg_decide(ctl + p, D.value(), g.value(), tot, hist, p, gridDim.y);
    const T beta = sbeta;
    if (i < n) Pp[i] = zv - beta * pv;
    for (i += gstride(); i < n; i += gstride()) Pp[i] = z[r0 + i] - beta * Pp[i];
}

// ---------------------------------------------------------------------------------------
// Algorithm 2

// Gram partials of Delta_i = Q_i^T P_i (w x w) and gamma_i = P_i^T r (w) for the current block.
// The n rows of a problem fall into gram_parts runs of consecutive rows with a partial each, so the
// partition depends on the problem alone.
constexpr int kGramRows = 64;
constexpr int kGramThreads = 1024;     // threads that the work of a CTA is divided over
constexpr int kGramFew = 256;          // threads of a CTA when a batch has many problems
__device__ __forceinline__ int gram_parts(int n, int gmax) { return min((n + kGramRows - 1) / kGramRows, gmax); }

// A CTA takes the runs blockIdx.x, blockIdx.x + gridDim.x, ... and stages kGramRows rows at a time, the
// next ones in registers meanwhile.  Its threads split the rows over NG groups (4 to 16, as many as w x w
// threads fit); a thread adds one entry of Delta over its group's rows in two interleaved sums, and a
// row of gamma's products per half warp; the sums meet in shared memory.  Bound by the
// float-pair additions (10 instructions a term): with one thread per entry over 128 rows the kernel took
// 9 us on 1000 cameras (15.4k of its cycles staging and adding), now 4.7 us; more CTAs than SMs made a
// batch of 16 problems pay each CTA's start in turn (14.1 us; looping CTAs 13.0 us).
// NT threads do the work of kGramThreads, kGramThreads / NT each, in the same order.  A CTA of 1024 threads
// leaves no room for another on its SM, so many problems of a few runs each went through loads and barriers
// in turn (64 problems of 60 cameras, one direction: 79.1 us per iteration, 75.1 with 256 threads).
template <typename T, int NT>
__global__ void __launch_bounds__(NT, NT < kGramThreads ? 3 : 1)
    k_mcg_gram(const T* __restrict__ P, const T* __restrict__ Q, const T* __restrict__ r,
               double* __restrict__ partial, int gmax, const Ctl* __restrict__ ctl) {
    wait_prior_grid();   // chained launch: the previous kernel's results are visible from here
    const int p = blockIdx.y;
    const Ctl& c = ctl[p];
    if (c.done) return;
    const int nr = c.lay.nc * 9;
    const int64_t n = nr;
    const int gp = gram_parts(nr, gmax);
    if (int(blockIdx.x) >= gp) return;
    constexpr int TR = kGramRows, NW = kGramThreads / 32;
    static_assert(TR * kMaxDirs == kGramThreads && 2 * NW == TR, "a value of P and of Q per thread, a row per half warp");
    __shared__ T sP[TR][kMaxDirs + 1], sQ[TR][kMaxDirs + 1], sr[TR];
    __shared__ double st[kGramThreads];      // the groups' sums, slot g w w + e
    __shared__ double sg[NW][kMaxDirs];      // the warps' sums of gamma
    constexpr int V = kGramThreads / NT;     // threads of the division that a thread stands for: t + NT v
    const int t = threadIdx.x, lane = t & 31;
    const int w = c.w_cur, off = c.off_cur, ww = w * w;
    const T* Pp = P + c.lay.hoff + int64_t(off) * n;
    const T* Qp = Q + c.lay.hoff + int64_t(off) * n;
    const T* rp = r + 9 * int64_t(c.lay.c0);
    const int per = (nr + gp - 1) / gp;
    int NG = 4;   // row groups; a group has kGramThreads / NG threads
    while (NG < 16 && kGramThreads / (2 * NG) >= ww) NG *= 2;
    const int gt = kGramThreads / NG, gr = TR / NG;
    const int lr = t % TR;                   // loads: a warp reads 32 rows of one column
    T pn[V], qn[V], rn = T(0);
    auto load = [&](int base, int end) {
        const bool in = base + lr < end;
#pragma unroll
        for (int v = 0; v < V; ++v) {
            const int lc = (t + NT * v) / TR;
            pn[v] = in && lc < w ? Pp[lc * n + base + lr] : T(0);
            qn[v] = in && lc < w ? Qp[lc * n + base + lr] : T(0);
        }
        rn = in && t < TR ? rp[base + lr] : T(0);
    };
    int part = blockIdx.x, base = part * per;
    load(base, min(base + per, nr));
    while (part < gp) {
        ExactSum<T> a0[V], a1[V], ag[V];
        bool more = true;
        while (more) {
#pragma unroll
            for (int v = 0; v < V; ++v) {
                sP[lr][(t + NT * v) / TR] = pn[v];
                sQ[lr][(t + NT * v) / TR] = qn[v];
            }
            if (t < TR) sr[lr] = rn;
            __syncthreads();
            // the next rows of this run, or the first of the CTA's next run
            base += TR;
            more = base < min((part + 1) * per, nr);
            if (!more) base = (part + int(gridDim.x)) * per;
            const int np = more ? part : part + int(gridDim.x);
            if (np < gp) load(base, min((np + 1) * per, nr));
#pragma unroll
            for (int v = 0; v < V; ++v) {
                const int g = (t + NT * v) / gt, e = t + NT * v - g * gt;
                if (e < ww) {   // rows past the last one are zeros
                    const T* x = &sQ[g * gr][e / w];
                    const T* y = &sP[g * gr][e % w];
#pragma unroll 4
                    for (int k = 0; k < gr; k += 2) {
                        a0[v].add(x[k * (kMaxDirs + 1)], y[k * (kMaxDirs + 1)]);
                        a1[v].add(x[(k + 1) * (kMaxDirs + 1)], y[(k + 1) * (kMaxDirs + 1)]);
                    }
                }
                const int row = 2 * ((t + NT * v) >> 5) + (lane >> 4);
                ag[v].add(sP[row][lane & 15], sr[row]);
            }
            __syncthreads();
        }
#pragma unroll
        for (int v = 0; v < V; ++v) {
            const int g = (t + NT * v) / gt, e = t + NT * v - g * gt;
            combine(a0[v], a1[v]);
            combine_shfl(ag[v], 16);
            if (e < ww) store_partial(&st[g * ww + e], a0[v]);
            if (lane < kMaxDirs) store_partial(&sg[(t + NT * v) >> 5][lane], ag[v]);
        }
        __syncthreads();
        double* out = partial + (int64_t(p) * gmax + part) * kGramMax;
        for (int e = t; e < ww; e += NT) {
            ExactSum<T> a;
            for (int k = 0; k < NG; ++k) load_partial(a, &st[k * ww + e]);
            store_partial(out + e, a);
        }
        if (t >= NT - kMaxDirs && t - (NT - kMaxDirs) < w) {
            const int cc = t - (NT - kMaxDirs);
            ExactSum<T> a, b;
#pragma unroll
            for (int k = 0; k < NW; k += 2) {
                load_partial(a, &sg[k][cc]);
                load_partial(b, &sg[k + 1][cc]);
            }
            combine(a, b);
            store_partial(out + ww + cc, a);
        }
        part += gridDim.x;
        // st and sg are written again only after the next run's first barrier
    }
}

// Jacobi eigen-decomposition based pseudo-inverse of the symmetric w x w matrix in sA
// (w <= 16, blockDim >= 256).  Eigenvalues at or below w 2^-52 lambda_max are dropped.
// On return sX holds A^+.  sV is scratch.
__device__ void pinv_sym_jacobi(double (*sA)[kMaxDirs + 1], double (*sV)[kMaxDirs + 1],
                                double (*sX)[kMaxDirs + 1], int w) {
    __shared__ double cs[kMaxDirs][2];
    __shared__ int pp[kMaxDirs], pq[kMaxDirs];
    __shared__ double off_norm, tot_norm;
    __shared__ double lam[kMaxDirs];
    const int t = threadIdx.x;
    const int i = t / kMaxDirs, j = t % kMaxDirs;
    if (t < kMaxDirs * kMaxDirs) sV[i][j] = (i == j) ? 1.0 : 0.0;
    __syncthreads();
    const int m = (w + 1) & ~1;   // even player count (index w is a dummy when w is odd)
    for (int sweep = 0; sweep < 30 && w > 1; ++sweep) {
        if (t < 32) {
            double o = 0.0, a = 0.0;
            for (int e = t; e < w * w; e += 32) {
                const int x = e / w, y = e % w;
                const double v = sA[x][y] * sA[x][y];
                a += v;
                if (x != y) o += v;
            }
            o = warp_sum(o);
            a = warp_sum(a);
            if (t == 0) {
                off_norm = o;
                tot_norm = a;
            }
        }
        __syncthreads();
        if (!(off_norm > 1e-30 * tot_norm)) break;
        for (int round = 0; round < m - 1; ++round) {
            // round-robin pairing: player 0 fixed, the others rotate
            if (t < m / 2) {
                int a = (t == 0) ? 0 : 1 + (round + t - 1) % (m - 1);
                int b = 1 + (round + m - 2 - t) % (m - 1);
                if (t == 0) b = 1 + (round + m - 2) % (m - 1);
                int p = a < b ? a : b, q = a < b ? b : a;
                double c = 1.0, s = 0.0;
                if (q < w && p < w) {
                    double apq = sA[p][q];
                    if (fabs(apq) > 1e-300) {
                        double app = sA[p][p], aqq = sA[q][q];
                        double theta = (aqq - app) / (2.0 * apq);
                        double tt = (theta >= 0 ? 1.0 : -1.0) / (fabs(theta) + sqrt(theta * theta + 1.0));
                        c = 1.0 / sqrt(tt * tt + 1.0);
                        s = tt * c;
                    }
                }
                pp[t] = p;
                pq[t] = q;
                cs[t][0] = c;
                cs[t][1] = s;
            }
            __syncthreads();
            // rows: A <- J^T A
            double nv = 0.0, nvv = 0.0;
            int which = -1;
            if (t < kMaxDirs * kMaxDirs && i < w && j < w) {
                for (int k = 0; k < m / 2; ++k) {
                    if (pp[k] == i || pq[k] == i) { which = k; break; }
                }
                if (which >= 0 && pq[which] < w) {
                    const int p = pp[which], q = pq[which];
                    const double c = cs[which][0], s = cs[which][1];
                    nv = (i == p) ? c * sA[p][j] - s * sA[q][j] : s * sA[p][j] + c * sA[q][j];
                } else {
                    nv = sA[i][j];
                }
            }
            __syncthreads();
            if (t < kMaxDirs * kMaxDirs && i < w && j < w) sA[i][j] = nv;
            __syncthreads();
            // columns: A <- A J, V <- V J
            which = -1;
            if (t < kMaxDirs * kMaxDirs && i < w && j < w) {
                for (int k = 0; k < m / 2; ++k) {
                    if (pp[k] == j || pq[k] == j) { which = k; break; }
                }
                if (which >= 0 && pq[which] < w) {
                    const int p = pp[which], q = pq[which];
                    const double c = cs[which][0], s = cs[which][1];
                    nv = (j == p) ? c * sA[i][p] - s * sA[i][q] : s * sA[i][p] + c * sA[i][q];
                    nvv = (j == p) ? c * sV[i][p] - s * sV[i][q] : s * sV[i][p] + c * sV[i][q];
                } else {
                    nv = sA[i][j];
                    nvv = sV[i][j];
                }
            }
            __syncthreads();
            if (t < kMaxDirs * kMaxDirs && i < w && j < w) {
                sA[i][j] = nv;
                sV[i][j] = nvv;
            }
            __syncthreads();
        }
    }
    if (t == 0) {
        double top = 0.0;
        for (int k = 0; k < w; ++k) top = fmax(top, sA[k][k]);
        const double thr = w * 2.220446049250313e-16 * top;
        for (int k = 0; k < w; ++k) lam[k] = (sA[k][k] > thr) ? 1.0 / sA[k][k] : 0.0;
    }
    __syncthreads();
    if (t < kMaxDirs * kMaxDirs && i < w && j < w) {
        double s = 0.0;
        for (int k = 0; k < w; ++k) s += sV[i][k] * lam[k] * sV[j][k];
        sX[i][j] = s;
    }
    __syncthreads();
}


// Inverse of the symmetric w x w matrix in sA by symmetric Gauss-Jordan sweeps on the diagonal (no
// pivoting), accepted (certified below) only when it equals the pseudo-inverse.  The first kInvThreads
// threads of the CTA call it; thread t owns entry (i, j), i >= j, of the lower triangle (the diagonal
// entries in warp 0), so a sweep costs 5 warps of float64 operations.  A dependent float64 operation
// takes about 150 cycles here, so the chain of a sweep is kept to three of them: with t = x_ik x_kj formed
// while the pivot's reciprocal r is (an estimate from the bit pattern and one Newton step), an entry
// is x_ij - t r.  sX (full storage) receives A^{-1}; *bad is set when a pivot is not positive.
// (16 x 16: 29k cycles with a mul, an fma and five operations for the reciprocal in the chain and two
// barriers of 1024 threads per sweep.)  sA is symmetrised on the way.
constexpr int kInvThreads = 160;
__device__ __forceinline__ void inv_barrier() { asm volatile("bar.sync 1, %0;" ::"n"(kInvThreads) : "memory"); }
__device__ __forceinline__ void inverse_sweeps(double (*sA)[kMaxDirs + 1], double (*sX)[kMaxDirs + 1], int w, int* bad) {
    __shared__ double rk;
    const int t = threadIdx.x;
    // entry of this thread: the diagonal first, then the strict lower triangle row by row
    int i = t, j = t;
    if (t >= kMaxDirs) {
        int q = t - kMaxDirs;
        i = 1;
        while (q >= i) q -= i++;
        j = q;
    }
    const bool in = t < kMaxDirs * (kMaxDirs + 1) / 2 && i < w && j < w;
    double x = 0.0;
    if (in) {   // symmetrised, also for the eigen-decomposition
        x = i == j ? sA[i][i] : 0.5 * (sA[i][j] + sA[j][i]);
        sA[i][j] = sA[j][i] = x;
        sX[i][j] = sX[j][i] = x;
    }
    for (int k = 0; k < w; ++k) {
        inv_barrier();   // sX holds the matrix after k sweeps
        const double xik = in ? sX[i][k] : 0.0, xkj = in ? sX[k][j] : 0.0;
        // the new entry is b - a r in every position: x_ij - x_ik x_kj r off the pivot's row and
        // column, x_kj r and x_ik r on them, -r on the pivot
        double a = xik * xkj, b = x;
        if (i == k || j == k) {
            a = i == j ? 1.0 : -x;
            b = 0.0;
        }
        if (t == k) {
            if (!(x > 0.0)) *bad = 1;
            rk = fast_rcp(x);
        }
        inv_barrier();
        if (in) {
            x = fma(-a, rk, b);
            sX[i][j] = sX[j][i] = x;
        }
    }
    if (in) sX[i][j] = sX[j][i] = -x;   // the sweeps leave -A^{-1}
}

constexpr int kSmallThreads = 1024;
// The small solve of a step, by a CTA of 256 threads or more (all of them call it; the CTA's writes
// to m.A, m.g and m.bad = 0 come before a barrier): alpha = Delta^+ gamma into c->alpha_v, gamma^T alpha
// into c->ga, Delta^+ into m.X and (not null) Dp.
struct SmallSolve {
    double A[kMaxDirs][kMaxDirs + 1], V[kMaxDirs][kMaxDirs + 1], X[kMaxDirs][kMaxDirs + 1];
    double g[kMaxDirs], al[kMaxDirs];
    double tr;
    int bad, ok;
};
__device__ void solve_block(Ctl* c, SmallSolve& m, int w, double* Dp) {
    const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
    if (w == 1) {
        if (Dp && t < kMaxDirs * kMaxDirs && t > 0) Dp[t] = 0.0;
        if (t == 0) {
            const double x = m.A[0][0] > 0.0 ? 1.0 / m.A[0][0] : 0.0, al = x * m.g[0], ga = m.g[0] * al;
            if (Dp) Dp[0] = x;
            m.X[0][0] = x;
            c->alpha_v[0] = al;
            c->ga = ga;
            if (!(ga == ga)) { c->done = 1; c->status = BA_ERR_BREAKDOWN; }
        }
        return;
    }
    if (t < kInvThreads) {
        inverse_sweeps(m.A, m.X, w, &m.bad);
    } else if (wid == kInvThreads / 32) {
        const double d = warp_sum(lane < w ? m.A[lane][lane] : 0.0);
        if (lane == 0) m.tr = d;
    }
    __syncthreads();
    // alpha = Delta^+ gamma (warp 0: two lanes per row) and gamma^T alpha, while warp 1 checks the
    // certificate and the others store the inverse; once more after a pseudo-inverse
    for (int pass = 0; pass < 2; ++pass) {
        if (wid == 0) {
            const int a = lane >> 1, b0 = (lane & 1) * (kMaxDirs / 2);
            double s0 = 0.0, s1 = 0.0;
#pragma unroll
            for (int b = 0; b < kMaxDirs / 2; b += 2) {
                if (a < w && b0 + b < w) s0 += m.X[a][b0 + b] * m.g[b0 + b];
                if (a < w && b0 + b + 1 < w) s1 += m.X[a][b0 + b + 1] * m.g[b0 + b + 1];
            }
            double s = s0 + s1;
            s += __shfl_xor_sync(0xffffffffu, s, 1);
            if (a < w && !(lane & 1)) {
                m.al[a] = s;
                c->alpha_v[a] = s;
            }
            double ga = a < w ? m.g[a] * s : 0.0;
#pragma unroll
            for (int o = 2; o < 32; o <<= 1) ga += __shfl_xor_sync(0xffffffffu, ga, o);
            if (lane == 0) m.al[0] = ga;
        } else if (wid == 1 && pass == 0) {
            const double trinv = warp_sum(lane < w ? m.X[lane][lane] : 0.0);
            // 1 / trace(A^{-1}) > 1e3 thr, i.e. 1e3 thr trace(A^{-1}) < 1 (false for a NaN)
            const double thr = w * 2.220446049250313e-16 * m.tr;
            if (lane == 0) m.ok = !m.bad && 1e3 * thr * trinv < 1.0;
        } else if (Dp && wid >= 2) {
            for (int e = t - 64; e < kMaxDirs * kMaxDirs; e += int(blockDim.x) - 64) {
                const int ei = e / kMaxDirs, ej = e % kMaxDirs;
                Dp[e] = (ei < w && ej < w) ? m.X[ei][ej] : 0.0;
            }
        }
        __syncthreads();
        if (pass == 1 || m.ok) break;
        pinv_sym_jacobi(m.A, m.V, m.X, w);
        if (t == 0) c->pinv_steps += 1;
        __syncthreads();
    }
    if (t == 0) {
        const double ga = m.al[0];
        c->ga = ga;
        if (!(ga == ga)) { c->done = 1; c->status = BA_ERR_BREAKDOWN; }
    }
}

// Distributed shared memory of a cluster: the same variable of CTA `rank`, and the cluster's barrier.
__device__ __forceinline__ void store_remote(double* var, int rank, double v) {
    uint32_t a;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_u32(var)), "r"(rank));
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory");
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }

// Delta_i, gamma_i -> Delta_i^+ (stored for the reorthogonalisation), alpha_i, gamma^T alpha.
// One cluster of kSmallCtas CTAs per problem; gx is the stride of the Gram partials.  The CTAs share the
// entries of the Gram sums (one SM reading the partials of 9000 rows took 7k cycles), whose totals meet in
// the first CTA's shared memory; it does the rest.  A^{-1} is certified when every sweep pivot is
// positive (A positive definite) and 1 / trace(A^{-1}) <= lambda_min exceeds 1e3 times the threshold
// w 2^-52 trace(A) >= w 2^-52 lambda_max: no eigenvalue is dropped, so A^+ = A^{-1}.  Otherwise the
// eigen-decomposition runs.  1000 cameras, w = 16: 20.5 us in one CTA with the longer inverse, now 12.4 us.
constexpr int kSmallCtas = 8;
constexpr int kSmallGroups = 32;   // groups of threads that share the partials of an entry
template <typename T>
__global__ void __cluster_dims__(kSmallCtas, 1, 1) __launch_bounds__(kSmallThreads)
    k_mcg_small(Ctl* ctl, const double* __restrict__ partial, int gx, double* __restrict__ dpinv, int mi1) {
    cluster_arrive();    // waited for before the first store to another CTA: every CTA has started by then
    wait_prior_grid();   // chained launch: the previous kernel's results are visible from here
    const int p = blockIdx.x / kSmallCtas, rank = blockIdx.x % kSmallCtas;
    Ctl* c = ctl + p;
    const int t = threadIdx.x;
    const bool done = c->done != 0;
    if (rank == 0 && t == 0) {
        c->live = !done;
        c->hist_cols = c->cols;   // the next reorthogonalisation runs over every column so far
    }
    if (done) {
        cluster_wait();
        return;
    }
    __shared__ SmallSolve sm;
    __shared__ double st[kSmallThreads];
    const int w = c->w_cur;
    const int it = c->it;
    const int ne = w * w + w;
    const int np = gram_parts(c->lay.nc * 9, gx);
    const double* part = partial + int64_t(p) * gx * kGramMax;
    // Sum of the Gram CTAs' partials of this CTA's entries.  They sit in L2, so the sum is bound by load
    // latency: G threads share an entry, group g takes the partials b = g, g + G, ... six loads in
    // flight, and the groups' sums meet in shared memory.  The order depends on (w, np) alone.
    {
        const int eb = (ne + kSmallCtas - 1) / kSmallCtas;   // entries of a CTA
        const int G = min(kSmallThreads / eb, kSmallGroups);
        const int g = t / eb, el = t - eb * g, e = rank * eb + el;
        if (g < G) {
            ExactSum<T> s;
            if (e < ne)
                for (int b0 = g; b0 < np; b0 += 6 * G) {
                    double v[6];
#pragma unroll
                    for (int u = 0; u < 6; ++u) v[u] = b0 + u * G < np ? part[int64_t(b0 + u * G) * kGramMax + e] : 0.0;
#pragma unroll
                    for (int u = 0; u < 6; ++u)
                        if (b0 + u * G < np) add_slot(s, v[u]);
                }
            store_partial(&st[t], s);
        }
        if (t == 0) sm.bad = 0;
        __syncthreads();
        cluster_wait();
        if (t < eb && e < ne) {   // here g = 0 and el = t
            ExactSum<T> a, b;
#pragma unroll 4
            for (int k = 0; k + 1 < G; k += 2) {
                load_partial(a, &st[k * eb + t]);
                load_partial(b, &st[(k + 1) * eb + t]);
            }
            if (G & 1) load_partial(a, &st[(G - 1) * eb + t]);
            combine(a, b);
            store_remote(e < w * w ? &sm.A[e / w][e % w] : &sm.g[e - w * w], 0, a.value());
        }
        cluster_arrive();
        cluster_wait();
        if (rank != 0) return;
    }
    solve_block(c, sm, w, dpinv + (int64_t(p) * mi1 + it) * kMaxDirs * kMaxDirs);
}

// The same for batches of many problems of few partials each (kSmallGroups, 213 cameras), a CTA per problem: eight
// CTAs of 1024 threads for every problem are more than the chip holds at once.  64 problems of 60 cameras, one
// direction: 75.1 us per iteration with the clusters, 66.3 us; 200 float64 problems of 16 cameras 146 and
// 101 us, 1000 of 10 cameras 554 and 327 us.  An entry's partials are added in the same groups and order.
constexpr int kSmallFew = 256;
template <typename T>
__global__ void __launch_bounds__(kSmallFew, 4)
    k_mcg_small_few(Ctl* ctl, const double* __restrict__ partial, int gx, double* __restrict__ dpinv, int mi1) {
    wait_prior_grid();   // chained launch: the previous kernel's results are visible from here
    const int p = blockIdx.x, t = threadIdx.x;
    Ctl* c = ctl + p;
    const bool done = c->done != 0;
    if (t == 0) {
        c->live = !done;
        c->hist_cols = c->cols;
    }
    if (done) return;
    __shared__ SmallSolve sm;
    const int w = c->w_cur, it = c->it, ne = w * w + w;
    const int np = gram_parts(c->lay.nc * 9, gx);
    const double* part = partial + int64_t(p) * gx * kGramMax;
    const int G = min(kSmallThreads / ((ne + kSmallCtas - 1) / kSmallCtas), kSmallGroups), ng = min(G, np);
    for (int e = t; e < ne; e += kSmallFew) {
        ExactSum<T> a[2];   // the even groups and the odd ones
        for (int k = 0; k < ng; k += 4) {
            double v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) v[u] = k + u < ng ? part[int64_t(k + u) * kGramMax + e] : 0.0;
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (k + u < ng) {
                    ExactSum<T> s;
                    add_slot(s, v[u]);
                    for (int b = k + u + G; b < np; b += G) add_slot(s, part[int64_t(b) * kGramMax + e]);
                    combine(a[u & 1], s);
                }
        }
        combine(a[0], a[1]);
        const double v = a[0].value();
        if (e < w * w) sm.A[e / w][e % w] = v;
        else sm.g[e - w * w] = v;
    }
    if (t == 0) sm.bad = 0;
    __syncthreads();
    solve_block(c, sm, w, dpinv + (int64_t(p) * mi1 + it) * kMaxDirs * kMaxDirs);
}

// x += P_i alpha; r -= Q_i alpha; z = D^{-1} r; per CTA the sums of |r|^2 and r^T z (dpart), from which
// k_mcg_phi's first CTA takes the decide step (grid: CTAs x problems; thread = one row, as in
// k_pcg_update).  The columns of the block are requested together (up to 16 of P and of Q per row).
template <typename T>
__global__ void __launch_bounds__(kUpdThreads) k_mcg_update(const double* __restrict__ Dinv, const T* __restrict__ P,
                                                            const T* __restrict__ Q, T* __restrict__ x,
                                                            T* __restrict__ r, T* __restrict__ z,
                                                            WideSlot<T>* __restrict__ dpart,
                                                            const Ctl* __restrict__ ctl) {
    wait_prior_grid();   // chained launch: the previous kernel's results are visible from here
    const int p = blockIdx.y;
    const Ctl& c = ctl[p];
    if (c.done) return;
    const int64_t c0 = c.lay.c0;
    const int nc = c.lay.nc;
    const int64_t n = int64_t(nc) * 9;
    const int w = c.w_cur, off = c.off_cur;
    const T* Pp = P + c.lay.hoff + int64_t(off) * n;
    const T* Qp = Q + c.lay.hoff + int64_t(off) * n;
    if (int64_t(blockIdx.x) * kUpdCams >= nc) return;   // no camera (a smaller problem of the batch)
    __shared__ T sal[kMaxDirs];
    __shared__ T sr[kUpdCams * 9];
    const int t = threadIdx.x, cl = t / 9, a = t - 9 * (t / 9);
    const int64_t jl = int64_t(blockIdx.x) * kUpdCams + cl;
    const bool act = t < kUpdCams * 9 && jl < nc;
    const int64_t il = 9 * jl + a, i = 9 * c0 + il;
    DinvRow<T> D;
    D.load(Dinv + 9 * i, act);
    T pv[kMaxDirs], qv[kMaxDirs];
#pragma unroll
    for (int b = 0; b < kMaxDirs; ++b) {
        const bool in = act && b < w;
        pv[b] = in ? Pp[int64_t(b) * n + il] : T(0);
        qv[b] = in ? Qp[int64_t(b) * n + il] : T(0);
    }
    const T xv = act ? x[i] : T(0), r0 = act ? r[i] : T(0);
    if (threadIdx.x < kMaxDirs) sal[threadIdx.x] = int(threadIdx.x) < w ? T(c.alpha_v[threadIdx.x]) : T(0);
    __syncthreads();
    ExactSum<T> v[2];
    T rv = T(0);
    if (act) {
        T dx[2] = {T(0), T(0)}, dr[2] = {T(0), T(0)};
#pragma unroll
        for (int b = 0; b < kMaxDirs; ++b)
            if (b < w) {
                dx[b & 1] += pv[b] * sal[b];
                dr[b & 1] += qv[b] * sal[b];
            }
        x[i] = xv + (dx[0] + dx[1]);
        rv = r0 - (dr[0] + dr[1]);
        r[i] = rv;
        v[0].add(rv, rv);
    }
    if (t < kUpdCams * 9) sr[t] = rv;
    __syncthreads();
    if (act) {
        const T zs = D.dot(sr + 9 * cl);
        z[i] = zs;
        v[1].add(rv, zs);
    }
    cta_publish<T, 2>(v, dpart + int64_t(p) * gridDim.x * 2);
}

// stop test, tau-test and the layout of the next block for problem p (one thread, after the
// update's totals are in)
__device__ void mcg_decide(Ctl* c, const double* tot, double* hist, int* blk_off, int* blk_w, int mi1, int p, int nb) {
    if (c->done) return;   // the small solve found a NaN
    if (c->status == BA_ERR_TIMEOUT) { c->done = 1; return; }
    const double rr = tot[0], rz = tot[1];
    const int it = c->it + 1;
    c->it = it;
    c->rr = rr;
    c->rz = rz;
    hist[int64_t(c->hist_off + it - 1) * nb + p] = rr * c->rr0_inv * c->hist_scale;   // squared relative residual
    if (!(rr == rr) || isinf(rr)) {
        c->done = 1;
        c->status = BA_ERR_BREAKDOWN;
        return;
    }
    if (rr < c->tol2 * c->rr0) {
        c->done = 1;
        c->status = BA_OK;
        return;
    }
    if (it >= c->max_iters) {
        c->done = 1;
        c->status = BA_ERR_NOT_CONVERGED;
        return;
    }
    if (!(rz > 0.0)) {
        c->done = 1;
        c->status = BA_ERR_BREAKDOWN;
        return;
    }
    // t_i = gamma^T alpha / r^T z (rz > 0), compared without the division
    const double ga = c->ga;
    if (c->stag > 0.0 && ga < c->stag * rz) {
        c->done = 1;      // no measurable progress left at this precision: end the sweep
        c->status = BA_OK;
        return;
    }
    const int local = (ga < c->tau * rz) ? 1 : 0;
    const int w = local ? c->n_eff : 1;
    if (c->cols + w > c->cap) {
        // history full: a float32 sweep ends here and the float64 refinement restarts it from the
        // true residual; a float64 solve cannot go on
        c->done = 1;
        c->status = c->stag > 0.0 ? BA_OK : BA_ERR_OOM;
        return;
    }
    c->local = local;
    c->local_steps += local;
    c->w_new = w;
    c->new_off = c->cols;
    c->w_cur = w;
    c->off_cur = c->cols;
    blk_off[int64_t(p) * mi1 + it] = c->cols;
    blk_w[int64_t(p) * mi1 + it] = w;
    c->cols += w;
}

// partial sums of Q[:, c]^T z over row chunks inside each subset:
// phip[(c * n_eff + s) * K + k] for c < hist_cols, as WideSum slots (grid: CTAs x problems).  Q^T z nearly
// cancels against all but the last blocks, so the lanes' sums are added as wide ones: with float pairs throughout
// beta's error against 64-bit sums reached 9e-8 of its column (6e-8 with float64 or wide sums over the lanes).
// Reads the whole history once, so it is bound by memory (L2 while the history fits): a warp takes one
// row chunk of up to kPhiCols columns at once, 8 rows of each in flight (32 loads a lane), and reads z
// once for all of them.  A column at a time with float64 shuffle trees ran at 2.1 TB/s (34 us on
// 2000 columns of 9000 rows; now 21 us).  Fewer columns at once when there are not enough chunks for
// the warps; a column's sum does not depend on it.  Chunks of at most 64 (128) rows take 2 (4) steps of rows at
// once: the registers of eight steps leave room for 24 warps an SM only (200 float64 problems of 16 cameras, 9 or
// 18 rows a chunk: 1004 -> 943 us per iteration with 16 directions, 233 -> 213 with 8).  The problem's first CTA
// runs the decide step beside them.
constexpr int kPhiCols = 4;
constexpr int phi_ctas(int steps) { return steps == 8 ? 3 : steps == 4 ? 4 : 5; }   // per SM
template <typename T, int NC, int U = 8>
__device__ __forceinline__ void phi_columns(const T* __restrict__ qc, int64_t n, const T* __restrict__ zp, int r0, int r1,
                                            WideSlot<T>* __restrict__ out, int64_t ostride) {
    const int lane = threadIdx.x & 31;
    ExactSum<T> acc[NC];
    for (int base = r0 + lane; base < r1; base += 32 * U) {
        T zv[U], qv[NC][U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int row = base + 32 * u;
            const bool in = row < r1;
            zv[u] = in ? zp[row] : T(0);
#pragma unroll
            for (int c = 0; c < NC; ++c) qv[c][u] = in ? qc[c * n + row] : T(0);
        }
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
            for (int c = 0; c < NC; ++c) acc[c].add(qv[c][u], zv[u]);
    }
#pragma unroll
    for (int c = 0; c < NC; ++c) {
        const WideSum<T> s = warp_total(WideSum<T>(acc[c]));
        if (lane == 0) out[c * ostride] = s.slot();
    }
}

template <typename T, int U>
__global__ void __launch_bounds__(kThreads, phi_ctas(U))
    k_mcg_phi(const T* __restrict__ Q, const T* __restrict__ z, WideSlot<T>* __restrict__ phip,
              const WideSlot<T>* __restrict__ dpart, int gu, double* __restrict__ hist_out,
              int* __restrict__ blk_off, int* __restrict__ blk_w, int mi1, Ctl* ctl) {
    wait_prior_grid();   // chained launch: the previous kernel's results are visible from here
    const int p = blockIdx.y;
    const Ctl& c = ctl[p];
    if (!c.live) return;
    const int nc = c.lay.nc;
    if (blockIdx.x == 0) {   // the decide step; nothing it writes is read by the other CTAs
        __shared__ double tot[2];
        const int wid = threadIdx.x >> 5;
        if (wid < 2) {
            const WideSum<T> s = total_of<T, 2>(dpart + int64_t(p) * gu * 2, (nc + kUpdCams - 1) / kUpdCams, wid);
            if ((threadIdx.x & 31) == 0) tot[wid] = s.value();
        }
        __syncthreads();
        if (threadIdx.x == 0) mcg_decide(ctl + p, tot, hist_out, blk_off, blk_w, mi1, p, gridDim.y);
        return;
    }
    const int64_t n = int64_t(nc) * 9;
    const int sz = c.sz, K = c.K, hist = c.hist_cols, chunks = c.n_eff * K;
    const int cz = (sz + K - 1) / K;
    const T* Qp = Q + c.lay.hoff;
    const T* zp = z + 9 * int64_t(c.lay.c0);
    WideSlot<T>* ph = phip + c.lay.phoff;
    const int64_t warps = int64_t(gridDim.x - 1) * (kThreads / 32);
    const int nb = 2 * int64_t(hist) * chunks >= kPhiCols * warps ? kPhiCols : 1;   // columns at once
    const int64_t items = int64_t((hist + nb - 1) / nb) * chunks;   // below 2^31: the partials' buffer holds them
    for (int64_t i64 = (gtid() - kThreads) >> 5; i64 < items; i64 += warps) {
        const unsigned it = unsigned(i64), ch = it % unsigned(chunks);
        const int c0 = int(it / unsigned(chunks)) * nb;
        const int s = int(ch) / K, k = int(ch) - s * K;
        int j0 = s * sz + k * cz, j1 = j0 + cz;
        const int send = (s + 1) * sz < nc ? (s + 1) * sz : nc;
        if (j1 > send) j1 = send;
        const T* qc = Qp + int64_t(c0) * n;
        WideSlot<T>* out = ph + int64_t(c0) * chunks + ch;
        const int m = hist - c0 < nb ? hist - c0 : nb;
        if (m == kPhiCols) phi_columns<T, kPhiCols, U>(qc, n, zp, 9 * j0, 9 * j1, out, chunks);
        else
            for (int u = 0; u < m; ++u)
                phi_columns<T, 1, U>(qc + u * n, n, zp, 9 * j0, 9 * j1, out + int64_t(u) * chunks, chunks);
    }
}

// Phi_j (wj x w) of one history block, entry e = a w + s: the partials of history column off + a over
// subset s (local block) or over every subset (global block); they are contiguous.  nt threads
// (t = 0 .. nt - 1, whole warps): G of them share an entry, each adds every G-th partial into two
// interleaved sums, and the group's sums meet in a fixed shuffle tree.
template <typename T>
__device__ __forceinline__ void phi_block(const WideSlot<T>* ph, int off, int w, int ne, int m, int n_eff, int K,
                                          bool local, int t, int nt, double* sphi) {
    int G = 1;
    while (G < 32 && 2 * G * ne <= nt) G *= 2;
    const int e = t / G, g = t % G;
    if (t - (t & 31) >= ne * G) return;   // warps without an entry (their shuffles go whole)
    WideSum<T> a0, a1;
    if (e < ne) {
        const int a = e / w, s2 = e - w * (e / w);
        const int64_t cc = off + a;
        const WideSlot<T>* sp = local ? ph + (cc * n_eff + s2) * K : ph + cc * n_eff * K;
        int k = g;
        for (; k + G < m; k += 2 * G) {
            a0.add(sp[k]);
            a1.add(sp[k + G]);
        }
        if (k < m) a0.add(sp[k]);
    }
    a0.add(a1);
    for (int o = G / 2; o > 0; o >>= 1) a0.add(a0.shfl_xor(o));
    if (e < ne && g == 0) sphi[e] = a0.value();
}

// Entry (a, s) of Delta_j^+ Phi_j in float64, four interleaved sums (a float64 operation has a long
// latency on this GPU).
__device__ __forceinline__ double beta_entry(const double* Dp, const double* sphi, int a, int s, int w, int wj) {
    double v[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
    for (int b = 0; b < kMaxDirs; b += 4)
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (b + u < wj) v[u] += Dp[a * kMaxDirs + b + u] * sphi[(b + u) * w + s];
    return (v[0] + v[1]) + (v[2] + v[3]);
}

// beta_{i,j} = Delta_j^+ Phi_{i,j} for every history block j, into beta rows in the Krylov storage type
// (the float64 product rounded once).  Blocks go round the CTAs (block jb to CTA jb mod gridDim.x),
// so consecutive ones run on different SMs; a block of 64 entries or more takes the whole CTA (a
// thread per entry), smaller ones a warp each.  With a warp per 16 x 16 block the 128 float64
// multiply-adds of a warp were a chain of 13 us (2000 columns); 4.8 us with the CTA.
template <typename T>
__global__ void __launch_bounds__(kThreads)
    k_mcg_beta(const WideSlot<T>* __restrict__ phip, const double* __restrict__ dpinv, const int* __restrict__ blk_off,
               const int* __restrict__ blk_w, T* __restrict__ beta, const Ctl* __restrict__ ctl, int mi1) {
    wait_prior_grid();   // chained launch: the previous kernel's results are visible from here
    const int p = blockIdx.y;
    const Ctl& c = ctl[p];
    if (c.done) return;
    constexpr int NW = kThreads / 32;
    constexpr int kBig = 64;                          // entries from which a block takes the CTA
    __shared__ double sphi[kMaxDirs * kMaxDirs];
    __shared__ double swarp[NW][2 * kBig];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int nblk = c.it;   // blocks 0..it-1 are the history
    const int n_eff = c.n_eff, K = c.K, w = c.w_new;
    const bool local = c.local != 0;
    const int m = local ? K : n_eff * K;   // partials per Phi entry
    // with one partial per entry (every sum is that partial) and many more blocks than CTAs, as in a batch of
    // many small problems, a warp per block up to 128 entries (200 problems of 30
    // cameras, 8 directions: 142 -> 120 us per iteration); 16 x 16 blocks are bound by the float64 pipe either way
    const int big = m == 1 && nblk > 2 * int(gridDim.x) ? 2 * kBig + 1 : kBig;
    const WideSlot<T>* ph = phip + c.lay.phoff;
    const int* bo = blk_off + int64_t(p) * mi1;
    const int* bw = blk_w + int64_t(p) * mi1;
    T* Bp = beta + c.lay.boff * kMaxDirs;
    for (int64_t j0 = blockIdx.x; j0 < nblk; j0 += int64_t(gridDim.x) * NW) {
        const int64_t jw = j0 + int64_t(gridDim.x) * wid;   // this warp's block
        if (jw < nblk && bw[jw] * w < big) {
            const int off = bo[jw], ne = bw[jw] * w;
            // a warp has no more lanes than it needs for 32 entries at a time
            for (int e0 = 0; e0 < ne; e0 += 32) {
                const int part = ne - e0 < 32 ? ne - e0 : 32;
                if (e0 == 0 && part == ne) phi_block<T>(ph, off, w, ne, m, n_eff, K, local, lane, 32, swarp[wid]);
                else if (lane < part) {
                    const int e = e0 + lane, a = e / w, s2 = e - w * (e / w);
                    const int64_t cc = int64_t(off + a) * n_eff;
                    const WideSlot<T>* sp = local ? ph + (cc + s2) * K : ph + cc * K;
                    WideSum<T> a0;
                    for (int k = 0; k < m; ++k) a0.add(sp[k]);
                    swarp[wid][e] = a0.value();
                }
            }
            __syncwarp();
            const double* Dp = dpinv + (int64_t(p) * mi1 + jw) * kMaxDirs * kMaxDirs;
            for (int e = lane; e < ne; e += 32)
                Bp[int64_t(off + e / w) * kMaxDirs + e % w] = T(beta_entry(Dp, swarp[wid], e / w, e % w, w, bw[jw]));
            __syncwarp();
        }
        for (int u = 0; u < NW; ++u) {
            const int64_t jb = j0 + int64_t(gridDim.x) * u;
            if (jb >= nblk) break;
            const int wj = bw[jb], ne = wj * w;
            if (ne < big) continue;
            const int off = bo[jb], t = threadIdx.x;
            phi_block<T>(ph, off, w, ne, m, n_eff, K, local, t, kThreads, sphi);
            __syncthreads();
            const double* Dp = dpinv + (int64_t(p) * mi1 + jb) * kMaxDirs * kMaxDirs;
            if (t < ne) Bp[int64_t(off + t / w) * kMaxDirs + t % w] = T(beta_entry(Dp, sphi, t / w, t % w, w, wj));
            __syncthreads();
        }
    }
}

// P_new = Z - P_hist beta, Q_new = (S Z) - Q_hist beta (Eq. 18; Q in float64 only: the float32 sweeps
// recompute it).  A tall-skinny product over the history, bound by reading it once: a CTA takes
// 32 consecutive rows of one problem, its kSlices warps split each tile of kTile columns (warp k takes
// columns k, k + kSlices, ...; lane = row, so every column is read as 32 consecutive values, eight
// columns in flight per lane), beta tiles are staged in shared memory, and the slices' sums meet
// in shared memory, where warp s adds column s of the new block in slice order.  With 4 warps
// per CTA and 4 columns in flight, 7 warps an SM kept 4 KB of loads in flight (131 us on 2000 columns
// of 9000 rows, 0.55 TB/s; now 35 us).  A one-column block (a global step) accumulates one column
// only.
template <typename T>
struct PqShape;
template <> struct PqShape<float> { static constexpr int kSlices = 16, kTile = 256; };
template <> struct PqShape<double> { static constexpr int kSlices = 8, kTile = 128; };
constexpr int kPqFew = 4;   // warps of a CTA when a batch has many problems

// RL rows per lane: a column's 16 betas are read from shared memory once for 32 RL rows.  With one row
// that read (16 words a lane for 16 multiply-adds) slows the kernel once every SM has work (17.7 us on average
// over a 1000-camera solve, 15.5 us with two rows); with fewer rows than that, more CTAs count for more.
// NW warps a CTA, kSlices / NW slices a warp, summed in the same order: with 16 warps two CTAs fit an SM, and a
// batch of many problems, each of several row blocks and a short history, goes through their barriers and
// loads in turn.  With four warps 64 problems of 60 cameras take 59.2 instead of 65.6 us per iteration (one
// direction); with more than 8 directions the sums of four slices cost more than that gains (48 problems of 100
// to 400 cameras, 16 directions: 411 -> 432 us), so the rule stops there.
template <typename T, int RL, int NW = PqShape<T>::kSlices>
__global__ void __launch_bounds__(NW * 32, NW < PqShape<T>::kSlices ? 4 : RL == 1 ? 2 : 1)
    k_mcg_pq(T* __restrict__ P, T* __restrict__ Q, const T* __restrict__ z, const T* __restrict__ beta,
             T* __restrict__ PT, const Ctl* __restrict__ ctl) {
    wait_prior_grid();   // chained launch: the previous kernel's results are visible from here
    const Ctl& c = ctl[blockIdx.y];
    if (c.done) return;
    constexpr bool kUpdQ = sizeof(T) == 8;
    constexpr int NS = PqShape<T>::kSlices, TC = PqShape<T>::kTile;
    constexpr int SP = NS / NW;                        // slices of a warp: k, k + NW, ...
    constexpr int U = (kUpdQ ? 4 : 8) / SP;            // columns of a slice in flight (of P, and of Q)
    static_assert(SP * NW == NS && U > 0, "whole slices");
    // two beta tiles during the loop over the history, then the slices' sums
    __shared__ __align__(16) T smem[NS * 32 * (kMaxDirs + 1)];
    static_assert(2 * TC * kMaxDirs <= NS * 32 * (kMaxDirs + 1), "beta tiles fit");
    auto red = reinterpret_cast<T(*)[32][kMaxDirs + 1]>(smem);
    const int lane = threadIdx.x & 31, k = threadIdx.x >> 5;
    const int64_t n = int64_t(c.lay.nc) * 9;
    const int64_t r0g = 9 * int64_t(c.lay.c0);
    const int w = c.w_new, off = c.new_off, hc = c.hist_cols, sz = c.sz;
    const bool local = c.local != 0;
    T* Pp = P + c.lay.hoff;
    T* Qp = Q + c.lay.hoff;
    const T* Bp = beta + c.lay.boff * kMaxDirs;
    static_assert(!kUpdQ || RL == 1, "two rows per lane in the float32 sweeps only");
    for (int64_t base = int64_t(blockIdx.x) * (32 * RL); base < n; base += int64_t(gridDim.x) * (32 * RL)) {
        const int64_t row = base + lane;   // and row + 32
        T ap[RL][SP][kMaxDirs], aq[SP][kUpdQ ? kMaxDirs : 1];
#pragma unroll
        for (int j = 0; j < SP; ++j)
#pragma unroll
            for (int s = 0; s < kMaxDirs; ++s) {
#pragma unroll
                for (int h = 0; h < RL; ++h) ap[h][j][s] = T(0);
                if constexpr (kUpdQ) aq[j][s] = T(0);
            }
        // beta tile t + 1 is copied while tile t is used (rows of 16 values; past w they may hold
        // anything, which reaches only sums that are not used)
        auto copy_b = [&](int c0n) {
            const int rows = hc - c0n < TC ? hc - c0n : TC;
            constexpr int kPer = 16 / sizeof(T);
            T* dst = smem + ((c0n / TC) & 1) * TC * kMaxDirs;
            for (int t = threadIdx.x; t * kPer < rows * kMaxDirs; t += blockDim.x)
                cp_async16(dst + t * kPer, Bp + int64_t(c0n) * kMaxDirs + t * kPer);
            cp_async_commit();
        };
        copy_b(0);
        for (int c0 = 0; c0 < hc; c0 += TC) {
            const int tc = hc - c0 < TC ? hc - c0 : TC;
            copy_b(c0 + TC);   // nothing past the last tile
            cp_async_wait_prev();
            __syncthreads();
            auto sB = reinterpret_cast<const T(*)[kMaxDirs]>(smem + ((c0 / TC) & 1) * TC * kMaxDirs);
            const T* pc = Pp + int64_t(c0) * n + row;
            const T* qc = Qp + int64_t(c0) * n + row;
            for (int cl = k; cl < tc; cl += NS * U) {
                T pv[RL][SP][U], qv[SP][U];
#pragma unroll
                for (int j = 0; j < SP; ++j)
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        const int cu = cl + NW * j + u * NS;
#pragma unroll
                        for (int h = 0; h < RL; ++h)
                            pv[h][j][u] = row + 32 * h < n && cu < tc ? pc[int64_t(cu) * n + 32 * h] : T(0);
                        if constexpr (kUpdQ) qv[j][u] = row < n && cu < tc ? qc[int64_t(cu) * n] : T(0);
                    }
                if (w == 1) {
#pragma unroll
                    for (int j = 0; j < SP; ++j)
#pragma unroll
                        for (int u = 0; u < U; ++u) {
                            const int cu = cl + NW * j + u * NS;
                            const T b0 = cu < tc ? sB[cu][0] : T(0);
#pragma unroll
                            for (int h = 0; h < RL; ++h) ap[h][j][0] += pv[h][j][u] * b0;
                            if constexpr (kUpdQ) aq[j][0] += qv[j][u] * b0;
                        }
                } else {
#pragma unroll
                    for (int j = 0; j < SP; ++j)
#pragma unroll
                        for (int u = 0; u < U; ++u) {
                            const int cu = cl + NW * j + u * NS;
                            if (cu >= tc) break;
#pragma unroll
                            for (int s = 0; s < kMaxDirs; s += 2) {
                                if constexpr (kUpdQ) {
                                    ap[0][j][s] += pv[0][j][u] * sB[cu][s];
                                    ap[0][j][s + 1] += pv[0][j][u] * sB[cu][s + 1];
                                    aq[j][s] += qv[j][u] * sB[cu][s];
                                    aq[j][s + 1] += qv[j][u] * sB[cu][s + 1];
                                } else {   // packed: each half rounds like a scalar fused multiply-add
                                    const float2 b2 = *reinterpret_cast<const float2*>(&sB[cu][s]);
#pragma unroll
                                    for (int h = 0; h < RL; ++h) {
                                        const float2 v = __ffma2_rn(make_float2(pv[h][j][u], pv[h][j][u]), b2,
                                                                    make_float2(ap[h][j][s], ap[h][j][s + 1]));
                                        ap[h][j][s] = v.x;
                                        ap[h][j][s + 1] = v.y;
                                    }
                                }
                            }
                        }
                }
            }
            __syncthreads();
        }
        // column s of the new block is added by warp s mod NW, over the slices in order
        auto slices = [&](const auto& acc, auto&& put) {
            __syncthreads();
#pragma unroll
            for (int j = 0; j < SP; ++j)
#pragma unroll
                for (int s = 0; s < kMaxDirs; ++s)
                    if (s < w) red[k + NW * j][lane][s] = acc[j][s];
            __syncthreads();
#pragma unroll
            for (int i = 0; i < (kMaxDirs + NW - 1) / NW; ++i) {
                const int s = k + NW * i;
                T sum = T(0);
                if (s < w)
#pragma unroll
                    for (int kk = 0; kk < NS; ++kk) sum += red[kk][lane][s];
                put(i, s, sum);
            }
        };
#pragma unroll
        for (int h = 0; h < RL; ++h) {
            const int64_t rh = row + 32 * h;
            const bool act = rh < n;
            const int sub = act ? int(rh / 9) / sz : 0;
            const T zr = act ? z[r0g + rh] : T(0);
            T pn[kMaxDirs / NW];
            slices(ap[h], [&](int i, int s, T sum) {
                pn[i] = s < w ? (s == (local ? sub : 0) ? zr : T(0)) - sum : T(0);
                if (act && s < w) Pp[int64_t(off + s) * n + rh] = pn[i];
            });
            if constexpr (kUpdQ) {
                slices(aq, [&](int, int s, T sum) {
                    if (act && s < w) Qp[int64_t(off + s) * n + rh] -= sum;
                });
            } else {
                // row-major copy of the new block for the multi-column product (zero past w)
                __syncthreads();
#pragma unroll
                for (int i = 0; i < kMaxDirs / NW; ++i) red[0][lane][k + NW * i] = pn[i];
                __syncthreads();
#pragma unroll
                for (int x = threadIdx.x; x < 32 * kMaxDirs; x += 32 * NW) {
                    const int rr = x / kMaxDirs, ss = x % kMaxDirs;
                    if (base + 32 * h + rr < n) PT[(r0g + base + 32 * h) * kMaxDirs + x] = red[0][rr][ss];
                }
            }
        }
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------------------
// A float32 sweep of a problem of at most kOneCams cameras in one CTA.
//
// Such a problem has no work for a chip: its iterations were 4 (PCG) or 9 (MCG) launches of 2.5 to 6 us
// each.  Here a CTA runs the whole sweep between barriers, with S, the vectors and the current block in
// shared memory.  The history stays in the problem's global arrays, which this kernel alone uses for it, in
// tiles of 64 columns stored row by row (hist_at), so that threads on neighbouring columns read
// neighbouring words.  It does what the kernels above do, step by step: exact-product sums, the float64 small
// solve and Delta^+ Phi, the same decide steps.
// 13 cameras: PCG 5.4 us per iteration (launched kernels 14.5), MCG with 8 directions to 1e-9 17.9 us (35.2).
//
// The rule: float32 sweeps of problems with nc <= kOneCams (S takes 324 nc^2 bytes: 130 KB of shared memory
// at 20 cameras), by MCG with up to kOneDirs local directions, whatever else is in the batch, so a problem's
// result does not depend on the others.  Delta_j^+ Phi_j costs w w' w float64 multiply-adds per pair of
// blocks on this SM's float64 pipe alone, and a rank-deficient block's eigen-decomposition shares it:
// to 1e-9 with 8 directions 18 to 25 us per iteration against 31 to 35 us in the kernels, with 10 directions
// (20 cameras) 33.4 against 33.6 us, with 16 directions (16 cameras) 92 against 60 us.
// Larger problems run the kernels above; a handle whose tile waits give up at once (wait_polls = -1) does
// too, since there is no tile wait here.
constexpr int kOneRows = 9 * kOneCams;
constexpr int kOneTile = 64;
constexpr int kOneThreads = 512;   // solve_block uses as many; more would leave 64 registers a thread

struct OneSmem {
    Ctl c;
    SmallSolve s;
    // the current block and its image (one_at), zero past its width up to a multiple of four
    __align__(16) float PT[kOneRows * kMaxDirs + 4 * kOneCams], QT[kOneRows * kMaxDirs + 4 * kOneCams];
    float x[kOneRows], r[kOneRows], z[kOneRows];
    __align__(16) double st[kOneThreads];
    double tot[4];
    float scal[2], al[kMaxDirs];
};

// Element (row i, column 0) of PT and QT: rows of 16, a camera's nine rows 20 banks after the last one's, so
// that the 16-byte reads of four consecutive cameras fall on different banks.
__device__ __forceinline__ int one_at(int i) { return kMaxDirs * i + 4 * (i / 9); }

// element (row i, column c) of a history of n rows
__device__ __forceinline__ int64_t hist_at(int n, int i, int c) {
    return (int64_t(c / kOneTile) * n + i) * kOneTile + c % kOneTile;
}

// QT = S PT for the first w columns (S dense in shared memory, block (j, k) at 81 (nc j + k)).  Thread =
// (three rows of a camera, quarter of the column cameras, group of NCOL = 4 columns, or the one column of
// a global step); the quarters meet in shuffles.  Bound by shared-memory reads: a row of PT serves three
// rows of S (one row per thread took 6.3k cycles for one column of 13 cameras, 12.3k for seven).
template <int NCOL>
__device__ __forceinline__ void one_product(const float* S, OneSmem& m, int nc, int w) {
    const int tr = 3 * nc, total = 4 * tr * ((w + NCOL - 1) / NCOL), lane = threadIdx.x & 31;
    for (int u = threadIdx.x; u - lane < total; u += kOneThreads) {   // whole warps, for the shuffles
        const bool in = u < total;
        const int quarter = u & 3, rg = u >> 2, g = rg / tr, trio = rg - tr * g;
        const int j = trio / 3, a0 = 3 * (trio - 3 * j);
        float acc[3][NCOL];
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
            for (int cc = 0; cc < NCOL; ++cc) acc[a][cc] = 0.f;
        for (int k = in ? quarter : nc; k < nc; k += 4) {
            const float* b = S + (nc * j + k) * 81 + 9 * a0;
            const float* pk = m.PT + one_at(9 * k) + NCOL * g;
#pragma unroll
            for (int e = 0; e < 9; ++e) {
                float pv[NCOL];
                if constexpr (NCOL == 4) {
                    const float4 v = *reinterpret_cast<const float4*>(pk + kMaxDirs * e);
                    pv[0] = v.x, pv[1] = v.y, pv[2] = v.z, pv[3] = v.w;
                } else {
                    pv[0] = pk[kMaxDirs * e];
                }
#pragma unroll
                for (int a = 0; a < 3; ++a)
#pragma unroll
                    for (int cc = 0; cc < NCOL; ++cc) acc[a][cc] = fmaf(b[9 * a + e], pv[cc], acc[a][cc]);
            }
        }
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
            for (int cc = 0; cc < NCOL; ++cc) {
                acc[a][cc] += __shfl_xor_sync(0xffffffffu, acc[a][cc], 1);
                acc[a][cc] += __shfl_xor_sync(0xffffffffu, acc[a][cc], 2);
            }
        if (in && quarter == 0) {
#pragma unroll
            for (int a = 0; a < 3; ++a)
#pragma unroll
                for (int cc = 0; cc < NCOL; ++cc)
                    m.QT[one_at(9 * j + a0 + a) + NCOL * g + cc] = NCOL * g + cc < w ? acc[a][cc] : 0.f;
        }
    }
}

// Sums of NV values over the rows (threads 0 .. kOneRows - 1 hold a product each, zeros past the problem).
// one_sums: float pairs, the same in every thread (Delta and gamma); a barrier before and after they are read.
// one_wide: the warps' wide sums into st and a barrier; one_total adds them, in the threads that need a value.
constexpr int kOneRowWarps = (kOneRows + 31) / 32;
static_assert(kOneRowWarps % 2 == 0, "pairs of warps");
template <int NV>
__device__ __forceinline__ void one_sums(ExactSum<float> (&v)[NV], double* st) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (wid < kOneRowWarps) {
#pragma unroll
        for (int k = 0; k < NV; ++k) {
            v[k] = warp_total(v[k]);
            if (lane == 0) store_partial(&st[NV * wid + k], v[k]);
        }
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < NV; ++k) {
        ExactSum<float> a, b;
#pragma unroll
        for (int q = 0; q < kOneRowWarps; q += 2) {
            load_partial(a, &st[NV * q + k]);
            load_partial(b, &st[NV * (q + 1) + k]);
        }
        combine(a, b);
        v[k] = a;
    }
    __syncthreads();
}
template <int NV>
__device__ __forceinline__ void one_wide(const ExactSum<float> (&v)[NV], float4* st) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (wid < kOneRowWarps) {
#pragma unroll
        for (int k = 0; k < NV; ++k) {
            const WideSum<float> s = warp_total(WideSum<float>(v[k]));
            if (lane == 0) st[NV * wid + k] = s.slot();
        }
    }
    __syncthreads();
}
template <int NV>
__device__ __forceinline__ double one_total(const float4* st, int k) {
    WideSum<float> a, b;
    a.set(st[k]);
    b.set(st[NV + k]);
#pragma unroll
    for (int q = 2; q < kOneRowWarps; q += 2) {
        a.add(st[NV * q + k]);
        b.add(st[NV * (q + 1) + k]);
    }
    a.add(b);
    return a.value();
}

// q^T z over the rows [i0, i1) of whole cameras (QS apart in q), by one thread: as accurate as float64.  (With
// three chains of float pairs, Delta^+ in double-float and double-float products, beta's error against 64-bit
// sums reached 1.1e-7 of its column; 6e-8, float32's rounding, with wide sums and a float64 product.)
template <int QS>
__device__ __forceinline__ double one_phi(const float* q, const float* z, int i0, int i1) {
    WideSum<float> a0, a1, a2;
    for (int i = i0; i < i1; i += 9) {   // a camera's rows
        float qv[9];
#pragma unroll
        for (int e = 0; e < 9; ++e) qv[e] = q[(i + e) * QS];
#pragma unroll
        for (int e = 0; e < 9; e += 3) {
            a0.mul_add(qv[e], z[i + e]);
            a1.mul_add(qv[e + 1], z[i + e + 1]);
            a2.mul_add(qv[e + 2], z[i + e + 2]);
        }
    }
    a0.add(a1);
    a0.add(a2);
    return a0.value();
}

__global__ void __launch_bounds__(kOneThreads, 1)
    k_one_cta(int mcg, const int64_t* __restrict__ row_ptr, const int64_t* __restrict__ tile_ptr,
              const int32_t* __restrict__ col, const float* __restrict__ Sg, const double* __restrict__ Dinv,
              float* __restrict__ xg, const float* __restrict__ rg, const float* __restrict__ zg, float* P, float* Q,
              WideSlot<float>* phip, double* dpinv, float* beta, int* __restrict__ colblk, double* __restrict__ hist,
              int* blk_off, int* blk_w, int mi1, Ctl* ctl) {
    const int p = blockIdx.x, t = threadIdx.x;
    if (!ctl[p].alone) return;
    extern __shared__ __align__(16) unsigned char smem_one[];
    OneSmem& m = *reinterpret_cast<OneSmem*>(smem_one);
    float* S = reinterpret_cast<float*>(smem_one + (sizeof(OneSmem) + 15) / 16 * 16);
    const Layout L = ctl[p].lay;
    const int nc = L.nc, n = 9 * nc, c0 = L.c0;
    if (t == 0) {
        m.c = ctl[p];
        m.c.alone = m.c.done = 0;   // running, for this CTA
    }
    for (int u = t; u < nc * nc * 81; u += kOneThreads) S[u] = 0.f;
    for (int u = t; u < kOneRows * kMaxDirs + 4 * kOneCams; u += kOneThreads) m.PT[u] = m.QT[u] = 0.f;
    __syncthreads();
    for (int j = 0; j < nc; ++j) {
        const int64_t rj = row_ptr[c0 + j], base = tile_ptr[c0 + j] * kTile;
        const int nj = int(row_ptr[c0 + j + 1] - rj);
        for (int u = t; u < 81 * nj; u += kOneThreads) {
            const int q = u / 81, e = u - 81 * q;
            S[(nc * j + (col[rj + q] - c0)) * 81 + e] = Sg[(base + q) * 81 + e];
        }
    }
    const bool act = t < n;
    const int cam = t / 9, own_at = one_at(t);   // this thread's row of PT and QT
    DinvRow<float> D;
    D.load(Dinv + 9 * (9 * int64_t(c0) + t), act);
    if (act) {
        m.x[t] = 0.f;
        m.r[t] = rg[9 * c0 + t];
        m.PT[own_at] = m.z[t] = zg[9 * c0 + t];
    }
    float* Pp = P + L.hoff;
    float* Qp = Q + L.hoff;
    __syncthreads();
    if (!mcg) {
        // Algorithm 1: the direction p is column 0 of PT, q = S p column 0 of QT
        while (true) {
            one_product<1>(S, m, nc, 1);
            __syncthreads();
            ExactSum<float> d[2];
            if (act) {
                d[0].add(m.QT[own_at], m.PT[own_at]);
                d[1].add(m.PT[own_at], m.r[t]);
            }
            one_sums<2>(d, m.st);
            const float alpha = __fdiv_rn(__fadd_rn(d[1].hi, d[1].lo), __fadd_rn(d[0].hi, d[0].lo));
            ExactSum<float> v[3];
            float rv = 0.f, qv = 0.f;
            if (act) {
                qv = m.QT[own_at];
                m.x[t] += alpha * m.PT[own_at];
                rv = m.r[t] - alpha * qv;
                m.r[t] = rv;
                v[0].add(rv, rv);
            }
            __syncthreads();
            float zs = 0.f;
            if (act) {
                zs = D.dot(m.r + 9 * cam);
                v[1].add(qv, zs);
                v[2].add(rv, zs);
            }
            float4* st = reinterpret_cast<float4*>(m.st);
            one_wide<3>(v, st);
            if (t == 0) m.scal[0] = float(one_total<3>(st, 1) * fast_rcp<2>(d[0].value()));
            if (t == 32) {   // the stop test beside it
                m.tot[0] = one_total<3>(st, 0);
                m.tot[2] = one_total<3>(st, 2);
                pcg_decide(&m.c, d[0].value(), d[1].value(), m.tot, hist, p, gridDim.x);
            }
            __syncthreads();
            if (m.c.done) break;
            if (act) m.PT[own_at] = zs - m.scal[0] * m.PT[own_at];
            __syncthreads();
        }
    } else {
        const int n_eff = L.n_eff, sz = L.sz;
        double* ph = reinterpret_cast<double*>(phip + L.phoff);   // values here, not slots
        double* dp = dpinv + int64_t(p) * mi1 * kMaxDirs * kMaxDirs;
        float* bt = beta + L.boff * kMaxDirs;
        int* cb = colblk + L.boff;
        const int* bo = blk_off + int64_t(p) * mi1;
        const int* bw = blk_w + int64_t(p) * mi1;
        one_product<1>(S, m, nc, 1);   // Q_0 = S P_0
        if (t == 0) cb[0] = 0;
        __syncthreads();
        if (act) {
            Pp[hist_at(n, t, 0)] = m.PT[own_at];
            Qp[hist_at(n, t, 0)] = m.QT[own_at];
        }
        while (true) {
            const int w = m.c.w_cur, it = m.c.it, ne = w * w + w;
            // Gram: groups of ne threads over the rows
            {
                const int G = min(kOneThreads / ne, 16), g = t / ne, e = t - ne * g;
                if (t == 0) m.s.bad = 0;
                if (g < G) {
                    const int a = e < w * w ? e / w : e - w * w, b = e - w * a;
                    ExactSum<float> s0, s1;
                    for (int i = g; i < n; i += 2 * G) {
                        const int i1 = i + G, o0 = one_at(i), o1 = one_at(i1);
                        if (e < w * w) s0.add(m.QT[o0 + a], m.PT[o0 + b]);
                        else s0.add(m.PT[o0 + a], m.r[i]);
                        if (i1 < n) {
                            if (e < w * w) s1.add(m.QT[o1 + a], m.PT[o1 + b]);
                            else s1.add(m.PT[o1 + a], m.r[i1]);
                        }
                    }
                    combine(s0, s1);
                    store_partial(&m.st[t], s0);
                }
                __syncthreads();
                if (t < ne) {
                    ExactSum<float> s0, s1;
                    for (int k = 0; k < G; k += 2) {
                        load_partial(s0, &m.st[k * ne + t]);
                        if (k + 1 < G) load_partial(s1, &m.st[(k + 1) * ne + t]);
                    }
                    combine(s0, s1);
                    const double v = s0.value();
                    if (t < w * w) m.s.A[t / w][t % w] = v;
                    else m.s.g[t - w * w] = v;
                }
                __syncthreads();
            }
            solve_block(&m.c, m.s, w, dp + int64_t(it) * kMaxDirs * kMaxDirs);
            __syncthreads();
            if (t < kMaxDirs) m.al[t] = t < w ? float(m.c.alpha_v[t]) : 0.f;
            __syncthreads();
            // update
            ExactSum<float> v[2];
            if (act) {
                float dx = 0.f, dr = 0.f;
                for (int b = 0; b < w; ++b) {
                    dx += m.PT[own_at + b] * m.al[b];
                    dr += m.QT[own_at + b] * m.al[b];
                }
                m.x[t] += dx;
                const float rv = m.r[t] - dr;
                m.r[t] = rv;
                v[0].add(rv, rv);
            }
            __syncthreads();
            float zs = 0.f;
            if (act) {
                zs = D.dot(m.r + 9 * cam);
                m.z[t] = zs;
                v[1].add(m.r[t], zs);
            }
            float4* st = reinterpret_cast<float4*>(m.st);
            one_wide<2>(v, st);
            if (t == 0) {
                m.tot[0] = one_total<2>(st, 0);
                m.tot[1] = one_total<2>(st, 1);
                m.c.hist_cols = m.c.cols;
                mcg_decide(&m.c, m.tot, hist, blk_off, blk_w, mi1, p, gridDim.x);
            }
            __syncthreads();
            if (m.c.done) break;
            const int hc = m.c.hist_cols, wn = m.c.w_new, off = m.c.new_off;
            const bool local = m.c.local != 0;
            // Phi: column c of the history against z over subset s, slot s hc + c
            for (int u = t; u < hc * n_eff; u += kOneThreads) {
                const int s = u / hc, c = u - hc * s;
                ph[u] = one_phi<kOneTile>(Qp + hist_at(n, 0, c), m.z, 9 * s * sz, min(9 * (s + 1) * sz, n));
            }
            __syncthreads();
            if (!local) {   // a global step: over every subset, into the first one's slots
                for (int c = t; c < hc; c += kOneThreads) {
                    double v[kMaxDirs];
#pragma unroll
                    for (int s = 0; s < kMaxDirs; ++s) v[s] = s < n_eff ? ph[s * hc + c] : 0.0;
                    double a0 = 0.0, a1 = 0.0;
#pragma unroll
                    for (int s = 0; s < kMaxDirs; s += 2) {
                        if (s < n_eff) a0 += v[s];
                        if (s + 1 < n_eff) a1 += v[s + 1];
                    }
                    ph[c] = a0 + a1;
                }
                __syncthreads();
            }
            // beta = Delta_j^+ Phi_j, entry (column c, new column s), in float64 rounded once
            for (int u = t; u < hc * wn; u += kOneThreads) {
                const int s = u / hc, c = u - hc * s, jb = cb[c], o = bo[jb], wj = bw[jb];
                const double* Dr = dp + (int64_t(jb) * kMaxDirs + (c - o)) * kMaxDirs;
                const double* phs = ph + s * hc + o;
                double acc0 = 0.0, acc1 = 0.0;
                for (int b0 = 0; b0 < wj; b0 += 8) {   // eight terms' loads in flight
                    double v[8], dv[8];
#pragma unroll
                    for (int e = 0; e < 8; ++e) {
                        v[e] = b0 + e < wj ? phs[b0 + e] : 0.0;
                        dv[e] = b0 + e < wj ? Dr[b0 + e] : 0.0;
                    }
#pragma unroll
                    for (int e = 0; e < 8; e += 2) {
                        if (b0 + e < wj) acc0 = fma(dv[e], v[e], acc0);
                        if (b0 + e + 1 < wj) acc1 = fma(dv[e + 1], v[e + 1], acc1);
                    }
                }
                bt[int64_t(c) * kMaxDirs + s] = float(acc0 + acc1);
            }
            __syncthreads();
            // P_new = Z - P_hist beta: thread = (three rows, four new columns, an eighth of every 32 columns)
            {
                const int tr = 3 * nc, total = 8 * tr * ((wn + 3) / 4);
                for (int u = t; u - (t & 31) < total; u += kOneThreads) {   // whole warps, for the shuffles
                    const bool in = u < total;
                    const int part = u & 7, rg2 = u >> 3, g = rg2 / tr, i0 = 3 * (rg2 - tr * g);
                    float acc[3][4];
#pragma unroll
                    for (int a = 0; a < 3; ++a)
#pragma unroll
                        for (int cc = 0; cc < 4; ++cc) acc[a][cc] = 0.f;
#pragma unroll 2
                    for (int c = in ? 4 * part : hc; c < hc; c += 32) {
                        // all seven loads in flight; P past hc is not used, beta past wn reaches sums that
                        // are not used
                        float4 pl[3], bl[4];
#pragma unroll
                        for (int a = 0; a < 3; ++a) pl[a] = *reinterpret_cast<const float4*>(Pp + hist_at(n, i0 + a, c));
#pragma unroll
                        for (int e = 0; e < 4; ++e)
                            bl[e] = *reinterpret_cast<const float4*>(bt + int64_t(min(c + e, hc - 1)) * kMaxDirs + 4 * g);
#pragma unroll
                        for (int a = 0; a < 3; ++a) {
                            const float pe[4] = {pl[a].x, c + 1 < hc ? pl[a].y : 0.f, c + 2 < hc ? pl[a].z : 0.f,
                                                 c + 3 < hc ? pl[a].w : 0.f};
#pragma unroll
                            for (int e = 0; e < 4; ++e) {
                                acc[a][0] = fmaf(pe[e], bl[e].x, acc[a][0]);
                                acc[a][1] = fmaf(pe[e], bl[e].y, acc[a][1]);
                                acc[a][2] = fmaf(pe[e], bl[e].z, acc[a][2]);
                                acc[a][3] = fmaf(pe[e], bl[e].w, acc[a][3]);
                            }
                        }
                    }
#pragma unroll
                    for (int a = 0; a < 3; ++a)
#pragma unroll
                        for (int cc = 0; cc < 4; ++cc)
#pragma unroll
                            for (int o = 1; o < 8; o <<= 1) acc[a][cc] += __shfl_xor_sync(0xffffffffu, acc[a][cc], o);
                    if (in && part < 3) {   // three lanes store a row each
                        const int i = i0 + part, own = local ? (i / 9) / sz : 0;
#pragma unroll
                        for (int cc = 0; cc < 4; ++cc) {
                            const int s = 4 * g + cc;
                            const float v = part == 0 ? acc[0][cc] : (part == 1 ? acc[1][cc] : acc[2][cc]);
                            m.PT[one_at(i) + s] = s < wn ? (s == own ? m.z[i] : 0.f) - v : 0.f;
                        }
                    }
                }
            }
            for (int u = t; u < wn; u += kOneThreads) cb[off + u] = it + 1;
            __syncthreads();
            if (wn == 1) one_product<1>(S, m, nc, 1);
            else one_product<4>(S, m, nc, wn);
            __syncthreads();
            for (int u = t; u < n * wn; u += kOneThreads) {
                const int i = u / wn, s = u - wn * i;
                const int64_t o = hist_at(n, i, off + s);
                Pp[o] = m.PT[one_at(i) + s];
                Qp[o] = m.QT[one_at(i) + s];
            }
            __syncthreads();
        }
    }
    if (act) xg[9 * c0 + t] = m.x[t];
    if (t == 0) ctl[p] = m.c;
}
constexpr size_t one_smem(int nc) { return (sizeof(OneSmem) + 15) / 16 * 16 + sizeof(float) * 81 * size_t(nc) * nc; }

// ---------------------------------------------------------------------------------------
// A float64 PCG solve of a problem of at most kCluCams cameras in one cluster of 8 CTAs.
//
// As for k_one_cta, an iteration of three launches had almost no work in it (16 cameras: 15 us).  In float64
// one SM would still need 6 us for the product of 16 cameras (its pipe does 1.7 lanes a clock), so the
// cameras go round a cluster's CTAs (camera j to CTA j mod 8), each with its rows of S in shared memory; the
// rows' vectors live in the registers of its first warp, and the CTAs exchange the sums and the direction
// through distributed shared memory, three cluster barriers per iteration (16 cameras: 6 us).  The rule is
// the camera count alone, as for k_one_cta, and so is the exception (wait_polls = -1).
constexpr int kCluThreads = 256;
constexpr int kCluOwn = kCluCams / kSmallCtas;   // cameras of a CTA, 27 rows: one warp
static_assert(9 * kCluOwn <= 32 && kCluCams % kSmallCtas == 0, "a CTA's rows in one warp");

__global__ void __cluster_dims__(kSmallCtas, 1, 1) __launch_bounds__(kCluThreads)
    k_pcg_cluster(const int64_t* __restrict__ row_ptr, const int64_t* __restrict__ tile_ptr,
                  const int32_t* __restrict__ col, const double* __restrict__ Sg, const double* __restrict__ Dinv,
                  double* __restrict__ xg, const double* __restrict__ rg, const double* __restrict__ zg,
                  double* __restrict__ hist, Ctl* ctl) {
    cluster_arrive();   // waited for before the first store to another CTA: every CTA has started by then
    const int p = blockIdx.x / kSmallCtas, rank = blockIdx.x % kSmallCtas;
    const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
    if (!ctl[p].alone) {   // the same in every CTA: the first one writes ctl after barriers
        cluster_wait();
        return;
    }
    extern __shared__ double S[];   // own camera m, column camera k: block at 81 (nc m + k)
    __shared__ Ctl sc;
    __shared__ double sp[9 * kCluCams], sq[9 * kCluOwn], dots[kSmallCtas][2], sums[kSmallCtas][3], tot[3];
    __shared__ int stop;
    const Layout L = ctl[p].lay;
    const int nc = L.nc, c0 = L.c0, own = rank < nc ? (nc - rank + kSmallCtas - 1) / kSmallCtas : 0;
    if (t == 0) {
        sc = ctl[p];
        sc.alone = sc.done = 0;   // running, for this cluster
    }
    for (int u = t; u < own * nc * 81; u += kCluThreads) S[u] = 0.0;
    for (int u = t; u < 9 * nc; u += kCluThreads) sp[u] = zg[9 * c0 + u];
    __syncthreads();
    for (int m = 0; m < own; ++m) {
        const int j = c0 + rank + kSmallCtas * m;
        const int64_t rj = row_ptr[j], base = tile_ptr[j] * kTile;
        const int nj = int(row_ptr[j + 1] - rj);
        for (int u = t; u < 81 * nj; u += kCluThreads) {
            const int q = u / 81, e = u - 81 * q;
            S[(nc * m + (col[rj + q] - c0)) * 81 + e] = Sg[(base + q) * 81 + e];
        }
    }
    // the first warp's lanes hold the CTA's rows
    const int m = lane / 9, a = lane - 9 * m, j = rank + kSmallCtas * m;
    const bool act = wid == 0 && m < own;
    const int64_t gi = 9 * int64_t(c0 + j) + a;
    DinvRow<double> D;
    D.load(Dinv + 9 * gi, act);
    double x = 0.0, r = act ? rg[gi] : 0.0, pv = act ? zg[gi] : 0.0;
    // the product's threads: row ru of the CTA, column cameras part, part + 8, ...
    const int ru = t >> 3, part = t & 7;
    const bool in = ru < 9 * own;
    const double* Srow = S + (nc * (in ? ru / 9 : 0)) * 81 + 9 * (ru % 9);
    __syncthreads();
    cluster_wait();
    while (true) {
        double s3[3] = {0.0, 0.0, 0.0};
        if (in)
            for (int k = part; k < nc; k += 8)
#pragma unroll
                for (int b = 0; b < 9; ++b) s3[b % 3] += Srow[81 * k + b] * sp[9 * k + b];
        double s = (s3[0] + s3[1]) + s3[2];
#pragma unroll
        for (int o = 1; o < 8; o <<= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (in && part == 0) sq[ru] = s;
        __syncthreads();
        double q = 0.0, rD = 0.0, Delta = 0.0, gamma = 0.0, zs = 0.0;
        if (wid == 0) {
            q = act ? sq[lane] : 0.0;
            const double d = warp_sum(q * pv), g = warp_sum(pv * r);
            if (lane < kSmallCtas) {
                store_remote(&dots[rank][0], lane, d);
                store_remote(&dots[rank][1], lane, g);
            }
        }
        cluster_arrive();
        cluster_wait();
        if (wid == 0) {
            Delta = lane < kSmallCtas ? dots[lane][0] : 0.0;
            gamma = lane < kSmallCtas ? dots[lane][1] : 0.0;
#pragma unroll
            for (int o = 4; o > 0; o >>= 1) {
                Delta += __shfl_xor_sync(0xffffffffu, Delta, o);
                gamma += __shfl_xor_sync(0xffffffffu, gamma, o);
            }
            Delta = __shfl_sync(0xffffffffu, Delta, 0);
            gamma = __shfl_sync(0xffffffffu, gamma, 0);
            rD = fast_rcp<2>(Delta);
            const double alpha = gamma * rD;
            x += alpha * pv;
            r -= alpha * q;
            double rb[9];
#pragma unroll
            for (int b = 0; b < 9; ++b) rb[b] = __shfl_sync(0xffffffffu, r, (9 * m + b) & 31);
            zs = act ? D.dot(rb) : 0.0;
            const double v0 = warp_sum(r * r), v1 = warp_sum(q * zs), v2 = warp_sum(r * zs);
            if (lane < kSmallCtas) {
                store_remote(&sums[rank][0], lane, v0);
                store_remote(&sums[rank][1], lane, v1);
                store_remote(&sums[rank][2], lane, v2);
            }
        }
        cluster_arrive();
        cluster_wait();
        if (wid == 0) {
            double v[3];
#pragma unroll
            for (int k = 0; k < 3; ++k) v[k] = lane < kSmallCtas ? sums[lane][k] : 0.0;
#pragma unroll
            for (int o = 4; o > 0; o >>= 1)
#pragma unroll
                for (int k = 0; k < 3; ++k) v[k] += __shfl_xor_sync(0xffffffffu, v[k], o);
            const double beta = __shfl_sync(0xffffffffu, v[1], 0) * rD;
            pv = zs - beta * pv;
            if (act)
#pragma unroll
                for (int dst = 0; dst < kSmallCtas; ++dst) store_remote(&sp[9 * j + a], dst, pv);
            if (lane == 0) {   // every CTA takes the same decision; the first one records it
#pragma unroll
                for (int k = 0; k < 3; ++k) tot[k] = v[k];
                pcg_decide(&sc, Delta, gamma, tot, rank == 0 ? hist : nullptr, p, int(gridDim.x) / kSmallCtas);
                stop = sc.done;
            }
            __syncwarp();
        }
        cluster_arrive();
        cluster_wait();
        if (stop) break;
    }
    if (act) xg[gi] = x;
    if (rank == 0 && t == 0) ctl[p] = sc;
}
constexpr size_t clu_smem(int nc) { return sizeof(double) * 81 * size_t(nc) * ((nc + kSmallCtas - 1) / kSmallCtas); }

// ---------------------------------------------------------------------------------------
// true residual t = -b~ - S x in float64; partial[2 j], partial[2 j + 1] = camera j's sums of
// t^2 and b~^2 (one warp per camera, all problems)

__global__ void k_true_residual(int32_t n_c, const int64_t* __restrict__ row_ptr, const int64_t* __restrict__ tile_ptr,
                                const int32_t* __restrict__ col, const double* __restrict__ S,
                                const double* __restrict__ x, const double* __restrict__ bt, double* __restrict__ res,
                                double* __restrict__ partial) {
    const int lane = threadIdx.x & 31;
    for (int64_t j = gtid() >> 5; j < n_c; j += gstride() >> 5) {
        const int64_t rj = row_ptr[j], nj = row_ptr[j + 1] - rj, tb = tile_ptr[j];
        double acc[9];
#pragma unroll
        for (int a = 0; a < 9; ++a) acc[a] = 0.0;
        for (int64_t q = lane; q < nj; q += 32) {
            const double* xk = x + int64_t(col[rj + q]) * 9;
            double xv[9];
#pragma unroll
            for (int b = 0; b < 9; ++b) xv[b] = xk[b];
            const double* sp = S + (tb * kTile + q) * 81;
#pragma unroll
            for (int a = 0; a < 9; ++a) {
#pragma unroll
                for (int b = 0; b < 9; ++b) acc[a] += sp[9 * a + b] * xv[b];
            }
        }
#pragma unroll
        for (int a = 0; a < 9; ++a) acc[a] = warp_sum(acc[a]);
        double tt = 0.0, bb = 0.0;
        if (lane < 9) {
            double sx = acc[0];
#pragma unroll
            for (int a = 1; a < 9; ++a) if (lane == a) sx = acc[a];
            const double b = bt[9 * j + lane];
            const double t = -b - sx;
            if (res) res[9 * j + lane] = t;
            tt = t * t;
            bb = b * b;
        }
        tt = warp_sum(tt);
        bb = warp_sum(bb);
        if (lane == 0) {
            partial[2 * j] = tt;
            partial[2 * j + 1] = bb;
        }
    }
}

// per problem: ctl.true_rr, ctl.bb and (ns = 3) ctl.scaled_exp from the ns per-camera partials (camera
// order); a warp each
__global__ void k_true_reduce(Ctl* ctl, const double* __restrict__ partial, int ns) {
    Ctl* c = ctl + blockIdx.x;
    const int k = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const double* pp = partial + ns * int64_t(c->lay.c0);
    if (k < 2) {
        const double v = sum_partials(pp, c->lay.nc, ns, k);
        if (lane == 0) (k == 0 ? c->true_rr : c->bb) = v;
    } else {
        int top = kNoExponent;
        for (int p = lane; p < c->lay.nc; p += 32)
            top = max(top, *reinterpret_cast<const int*>(pp + int64_t(p) * ns + k));
        top = __reduce_max_sync(0xffffffffu, top);
        if (lane == 0) c->scaled_exp = top;
    }
}

// mixed precision: x += unit Lam d, a float32 sweep's correction mapped back from the scaled system,
// and x split into double-float for the true residual that follows (its per-observation products take
// no float64 input); grid: CTAs x problems
__global__ void k_accumulate(const Layout* __restrict__ lay, const Outer* __restrict__ outer,
                             const float* __restrict__ d, const double* __restrict__ lam, double* __restrict__ x,
                             float2* __restrict__ xd) {
    const Layout L = lay[blockIdx.y];
    const double unit = outer[blockIdx.y].unit;
    for (int64_t il = gtid(); il < 9 * int64_t(L.nc); il += gstride()) {
        const int64_t i = 9 * int64_t(L.c0) + il;
        const double v = x[i] + lam[i] * (unit * double(d[i]));
        x[i] = v;
        const float h = __double2float_rn(v);
        xd[i] = make_float2(h, __double2float_rn(v - double(h)));
    }
}

// refinement start: x = 0 and rt = -b~
__global__ void k_start_refine(int64_t n, const double* __restrict__ bt, double* __restrict__ x,
                               double* __restrict__ rt) {
    for (int64_t i = gtid(); i < n; i += gstride()) {
        x[i] = 0.0;
        rt[i] = -bt[i];
    }
}

// One CTA per problem: |b~|^2 (fixed order), the largest exponent of Lam b~ and the refinement state at x = 0.
__global__ void k_outer_init(const Layout* __restrict__ lay, const double* __restrict__ bt,
                             const double* __restrict__ lam, Outer* outer) {
    const Layout L = lay[blockIdx.x];
    const int64_t n = int64_t(L.nc) * 9;
    const double* b = bt + 9 * int64_t(L.c0);
    __shared__ double s[1];
    __shared__ int top;
    if (threadIdx.x == 0) top = kNoExponent;
    double v[1] = {0.0};
    int e = kNoExponent;
    for (int64_t i = threadIdx.x; i < n; i += blockDim.x) {
        v[0] += b[i] * b[i];
        e = max(e, product_exponent(lam[9 * int64_t(L.c0) + i], b[i]));
    }
    cta_sum_write<1>(v, s);
    e = __reduce_max_sync(0xffffffffu, e);
    if ((threadIdx.x & 31) == 0) atomicMax(&top, e);
    __syncthreads();
    if (threadIdx.x == 0) {
        Outer o;
        memset(&o, 0, sizeof(o));
        o.bb = s[0];
        o.tr = s[0];
        o.tr_prev = s[0];
        o.se = top;
        o.unit = 1.0;
        o.status = s[0] == 0.0 ? BA_OK : BA_ERR_NOT_CONVERGED;
        o.active = s[0] == 0.0 ? 0 : 1;
        outer[blockIdx.x] = o;
    }
}

// Plan the next float32 sweep of every problem still refining: per sweep the inner solve reduces
// its residual by inner_tol; when what is left to reach tol is within ten times that, the sweep
// aims 3x past it so that it is the last one.  One CTA over all problems; sets the refinement
// loop's condition: another sweep when any problem takes part (count = 1: a loop pass has ended).
__global__ void k_refine_plan(Outer* outer, int nb, const Params* __restrict__ prm, cudaGraphConditionalHandle h,
                              int use_handle, Loops* lp, int count) {
    __shared__ int any;
    if (threadIdx.x == 0) any = 0;
    __syncthreads();
    const double tol = prm->tol, inner_tol = prm->inner_tol;
    int mine = 0;
    for (int b = threadIdx.x; b < nb; b += blockDim.x) {
        Outer* o = outer + b;
        o->swept = 0;
        if (!o->active) continue;
        if (o->sweeps >= prm->max_refine || o->iters >= prm->max_iters) {
            o->active = 0;
            continue;
        }
        const double need = tol * sqrt(o->bb) / sqrt(o->tr);
        double t = need > 0.1 * inner_tol ? fmax(0.3 * need, 0.1 * inner_tol) : inner_tol;
        if (t >= 1.0) t = 0.5;
        o->tol_in = t;
        o->unit = o->se > kNoExponent ? ldexp(1.0, max(-900, min(900, o->se))) : 1.0;
        o->max_in = prm->max_iters - o->iters;
        o->swept = 1;
        mine = 1;
    }
    if (mine) atomicOr(&any, 1);
    __syncthreads();
    if (threadIdx.x == 0) {
        if (count) lp->outer += 1;
        if (use_handle) cudaGraphSetConditional(h, any ? 1u : 0u);
    }
}

// After a sweep and the float64 true residual: account the sweep and decide whether to go on.
__global__ void k_refine_after(const Ctl* __restrict__ ctl, Outer* outer, const Params* __restrict__ prm) {
    Outer* o = outer + blockIdx.x;
    const Ctl& c = ctl[blockIdx.x];
    if (threadIdx.x != 0 || !o->swept) return;
    const double tol = prm->tol;
    const int mcg = prm->mcg;
    o->sweeps += 1;
    o->iters += c.it;
    o->locals += c.local_steps;
    o->pinvs += c.pinv_steps;
    o->cols = mcg ? c.cols : 1;
    o->tr_prev = o->tr;
    o->tr = c.true_rr;
    o->se = c.scaled_exp;
    if (c.status == BA_ERR_BREAKDOWN || c.status == BA_ERR_OOM || c.status == BA_ERR_TIMEOUT) {
        o->status = c.status;
        o->active = 0;
        return;
    }
    if (!(o->tr == o->tr)) {
        o->status = BA_ERR_BREAKDOWN;
        o->active = 0;
        return;
    }
    if (o->tr <= tol * tol * o->bb) {
        o->status = BA_OK;
        o->active = 0;
    }
}

}  // namespace

// ---------------------------------------------------------------------------------------
// host side

// What a captured solve graph depends on besides the per-solve Params: the algorithm, precision,
// loop body, work lists, wait bound and every buffer address (a reallocation bumps `allocs`).
struct GraphKey {
    int mcg = -1, fp32 = -1, chunk = 0, mi1 = 0, use_l = -1, epoch = -1, polls = -1, nb = -1, host = -1, cfg = -1;
    int lanes = -1;                   // column lanes of k_spmm
    int one = -1;                     // cameras of the largest problem that one CTA or cluster solves
    int all = -1;                     // one of them solves every problem
    int phi = -1;                     // rows of the largest Phi chunk
    uint64_t allocs = ~uint64_t(0);   // buffer generation (any reallocation invalidates the graph)
    const void* ptrs[4] = {};
    bool operator==(const GraphKey& o) const {
        if (mcg != o.mcg || fp32 != o.fp32 || chunk != o.chunk || mi1 != o.mi1 || use_l != o.use_l ||
            epoch != o.epoch || polls != o.polls || nb != o.nb || host != o.host || cfg != o.cfg ||
            lanes != o.lanes || one != o.one || all != o.all || phi != o.phi || allocs != o.allocs)
            return false;
        for (int i = 0; i < 4; ++i) if (ptrs[i] != o.ptrs[i]) return false;
        return true;
    }
};

// Kernel launches of a solve graph before, per pass of and after its loops.
struct GraphCounts {
    int pre = 0, sweep = 0, body = 0, post = 0;
};

struct SolveExec {
    GraphKey key;
    cudaGraphExec_t exec = nullptr;
    GraphCounts gc;
};

// device buffer that only grows
struct Buf {
    void* p = nullptr;
    size_t bytes = 0;
};

struct Solver {
    int nb = 0;               // problems
    int64_t n = 0;            // 9 n_c over all problems
    int mi1 = 0;              // per-problem stride of the per-step arrays (max_iters + 1)
    int gx = 1;               // grid width of the kernels over all rows of a problem (x += d)
    int gu = 1;               // grid width of the update kernels (kUpdCams cameras per CTA)
    int gg = 1;               // Gram partials of the largest problem
    int gq = 1;               // grid width of the per-row kernels
    int gpq = 1;              // grid width of the reorthogonalisation (32-row blocks)
    int gphi = 1, gb = 1;     // Phi and beta grid widths
    int phi_rows = 1;         // rows of the largest Phi chunk
    int one_cams = 0;         // cameras of the largest problem that k_one_cta or k_pcg_cluster solves (0: none)
    bool all_small = false;   // one of those two solves every problem
    int gcol = 1;             // grid width of the column pass of the symmetric product (a CTA per camera)
    std::vector<Layout> lay;  // of the current solve
    Buf P, Q, r, z, xw, PT, part_a, part_b, part_cam, dpinv, beta, colblk, phip, hist, blk_off, blk_w, ctl, outer, rt,
        lay_d, dpart, dtot, camdot, params, loops;
    Ctl* h_ctl = nullptr;     // pinned, nb
    Outer* h_outer = nullptr; // pinned, nb
    Params* h_params = nullptr;   // pinned staging of the per-solve arguments
    Loops* h_loops = nullptr;     // pinned
    double* h_hist = nullptr;     // pinned, nb x mi1 (iteration-major device history)
    size_t h_hist_n = 0;
    std::vector<std::vector<double>> host_hist;   // per problem, residual history of the last solve
    int64_t launches = 0;     // kernel executions issued by the current solve
    cudaStream_t cap_stream = nullptr, cap2 = nullptr, cap3 = nullptr;   // capture streams (nested loops)
    cudaStream_t cap_side = nullptr;                  // and of the branch of problems solved alone
    cudaEvent_t ev_fork = nullptr, ev_join = nullptr;
    std::vector<SolveExec*> execs;   // instantiated solve graphs
    cudaEvent_t ev0 = nullptr, ev1 = nullptr;   // around a solve
    // work lists of the block-sparse products: whole rows, rows split by pose subset, and whole rows of
    // the upper triangle (the symmetric one-column products of mixed precision)
    ItemList items_g, items_l, items_u;
    Buf tb;                    // transposed terms of the symmetric product (kTbHead + 1 values per upper block)
    int items_cb = -1;         // item chunk rule the lists were built with (0 = the default)
    int items_l_dirs = -1;
    int col_lanes = 4;         // lanes that share a block in k_spmm: four columns each cover n_dirs
    bool use_l = false;        // the current MCG solve splits rows by pose subset (n_dirs > 1)
    int epoch = 0;             // incremented whenever a work list is rebuilt (captured graphs hold them)
    int spmv_cfg = 0;          // shape of the one-column products (SpmvShape)
    void* mm_part = nullptr;   // k_spmm partials: items_g.n x 16 x 9
};

// Reallocations so far: captured graphs hold buffer addresses, so any reallocation forces a new
// capture (the graph key records this count).
static std::atomic<uint64_t> g_allocs{0};

static void grow(Buf& b, size_t bytes) {
    if (bytes == 0) bytes = 16;
    if (b.bytes >= bytes) return;
    ++g_allocs;
    if (b.p) cudaFree(b.p);
    b.p = nullptr;
    b.bytes = 0;
    cudaError_t e = cudaMalloc(&b.p, bytes);
    if (e != cudaSuccess) {
        cudaGetLastError();
        b.p = nullptr;
        throw Error(e == cudaErrorMemoryAllocation ? BA_ERR_OOM : BA_ERR_CUDA,
                    std::string("cudaMalloc(") + std::to_string(bytes) + "): " + cudaGetErrorString(e));
    }
    b.bytes = bytes;
}
template <typename T>
static T* ptr(const Buf& b) {
    return static_cast<T*>(b.p);
}

// Default blocks per work item: 16 tiles, and fewer for problems whose rows are too few to keep every warp
// busy with 16 (the longest item then sets the time).  Rows up to that length are one item; longer
// rows are split, and the row's pieces combined by the last one to finish.  The rule depends on the
// problem's own camera count alone, so its products sum in the same order alone and in any batch.
// Measured on GB300, product at 512 / 256 blocks: float32 601 cameras 33.8 / 26.0 us (the solves 16 %
// faster), 1000 cameras 43.4 / 41.9 us, 1936 cameras 118.1 / 119.1 us (MCG 2.5 % slower); float64 601
// cameras 82.0 / 71.1 us, 1000 cameras 166 / 174 us.  Float64 below that, at 256 / 128 / 64 blocks: 300
// cameras 46.8 / 33.3 / 41.3 us, 150 cameras 30.9 / 28.7 / 20.9 us (a float64 tile takes about 3 us, so a
// row in one warp is a long chain), but with shape 2, which has a quarter of the warps, 61.0 us at 128 for 300
// cameras and 53.3 us at 512, so that shape keeps 512 from 200 cameras on.  What decides is the tiles of a row
// against the warps of the launch, which a batch shares: 48 float64 problems of 100 to 400 cameras pay for the
// rule (530 / 580 / 697 us), the price of summing like a solo solve; ba_autotune sets the size for a handle.
// Float32 keeps 256 there: 128 gains 14 % of a PCG solve at 300 cameras and
// nothing at 150, and costs a batch 5 %.
static int default_item_blocks(int n_cams, bool fp32, int cfg) {
    if (fp32) return n_cams < 1200 ? 256 : 512;
    if (cfg == 2 && n_cams >= 200) return 512;
    return n_cams < 200 ? 64 : (n_cams < 450 ? 128 : (n_cams < 800 ? 256 : 512));
}

// Items of the block-sparse product, problem by problem: each (row, segment) split into chunks of
// at most cb blocks (cb = forced_cb, else default_item_blocks).
// split = false: one segment per row; otherwise segment s of a row of problem b holds the blocks
// whose column camera lies in [c0 + s sz, c0 + (s + 1) sz), for s < n_eff (empty segments get
// one empty item, which writes zeros).
static std::vector<SpItem> build_items(const std::vector<int64_t>& h_row_ptr, const std::vector<int32_t>& h_col,
                                       const std::vector<Layout>& lay, bool split, int forced_cb, bool fp32,
                                       int cfg) {
    std::vector<SpItem> out;
    int grp = 0;
    for (size_t b = 0; b < lay.size(); ++b) {
        const Layout& L = lay[b];
        const int cb = forced_cb > 0 ? forced_cb : default_item_blocks(L.nc, fp32, cfg);
        const int nseg = split ? L.n_eff : 1;
        for (int32_t j = L.c0; j < L.c0 + L.nc; ++j) {
            const int64_t rj = h_row_ptr[j], nj = h_row_ptr[j + 1] - rj;
            const int32_t* cj = h_col.data() + rj;
            for (int g = 0; g < nseg; ++g) {
                int q0 = 0, q1 = int(nj);
                if (split) {
                    q0 = int(std::lower_bound(cj, cj + nj, L.c0 + g * L.sz) - cj);
                    q1 = int(std::lower_bound(cj, cj + nj, L.c0 + (g + 1) * L.sz) - cj);
                }
                const int nch = q1 > q0 ? (q1 - q0 + cb - 1) / cb : 1;
                for (int c = 0; c < nch; ++c) {
                    SpItem it;
                    it.row = j;
                    it.seg = g;
                    it.q0 = q0 + c * cb;
                    it.q1 = std::min(q1, q0 + (c + 1) * cb);
                    if (it.q1 < it.q0) it.q1 = it.q0;
                    it.grp = grp;
                    it.k = c;
                    it.ng = nch;
                    it.prob = int(b);
                    it.slot = int(out.size());
                    out.push_back(it);
                }
                ++grp;
            }
        }
    }
    return out;
}

// Order the items for a launch of W warps, NW per CTA, by the longest-processing-time rule: in
// decreasing cost (tiles of S, in quarter tiles, plus a quarter for the item's own sums and output),
// each item goes to the bin with the least cost so far (ties: the lower bin).  Bin b is run by warp
// (b % C) * NW + b / C of the C = W / NW CTAs, so that the largest items, which go to the first bins,
// are spread over the SMs instead of filling the first CTAs.  Warp g's items follow in their
// original order at wptr[g].  Chunks and slots are unchanged, so the sums are too.  (Round-robin
// over the 1936-camera upper triangle left the longest warp 1.4x the mean; this rule, 1.05x.)
static std::vector<int64_t> balance_items(std::vector<SpItem>& v, int64_t W, int64_t NW) {
    const int64_t n = int64_t(v.size());
    std::vector<int64_t> cost(n), idx(n);
    for (int64_t i = 0; i < n; ++i) {
        const SpItem& it = v[i];
        const int64_t tiles = it.q1 > it.q0 ? ((int64_t(it.q1) + 31) >> 5) - (it.q0 >> 5) : 0;
        cost[i] = 4 * tiles + 1;
    }
    std::iota(idx.begin(), idx.end(), int64_t(0));
    std::stable_sort(idx.begin(), idx.end(), [&](int64_t a, int64_t b) { return cost[a] > cost[b]; });
    using Load = std::pair<int64_t, int64_t>;   // (cost so far, warp)
    std::priority_queue<Load, std::vector<Load>, std::greater<Load>> heap;
    for (int64_t g = 0; g < W; ++g) heap.push({0, g});
    const int64_t C = W / NW;
    std::vector<int64_t> owner(n), wptr(W + 1, 0);
    for (const int64_t i : idx) {
        const Load l = heap.top();
        heap.pop();
        const int64_t b = l.second;
        owner[i] = (b % C) * NW + b / C;
        heap.push({l.first + cost[i], b});
        ++wptr[owner[i] + 1];
    }
    for (int64_t g = 0; g < W; ++g) wptr[g + 1] += wptr[g];
    std::vector<int64_t> pos(wptr.begin(), wptr.end() - 1);
    std::vector<SpItem> out(n);
    for (int64_t i = 0; i < n; ++i) out[pos[owner[i]]++] = v[i];
    v.swap(out);
    return wptr;
}

static void free_items(ItemList& L) {
    if (L.items) cudaFree(const_cast<SpItem*>(L.items));
    if (L.cnt) cudaFree(L.cnt);
    if (L.part) cudaFree(L.part);
    if (L.wptr) cudaFree(const_cast<int64_t*>(L.wptr));
    L = ItemList();
}

// Upload a list, in the balanced order for W warps, NW per CTA (W > 0).
static void upload_items(ItemList& L, std::vector<SpItem> v, int64_t W, int64_t NW) {
    free_items(L);
    std::vector<int64_t> wptr;
    if (W > 0) wptr = balance_items(v, W, NW);
    SpItem* d = nullptr;
    BA_CUDA_TRY(cudaMalloc(&d, sizeof(SpItem) * (v.empty() ? 1 : v.size())));
    if (!v.empty()) BA_CUDA_TRY(cudaMemcpy(d, v.data(), sizeof(SpItem) * v.size(), cudaMemcpyHostToDevice));
    L.items = d;
    L.n = int64_t(v.size());
    int ngrp = 1, nprob = 0;
    for (const SpItem& it : v) {
        ngrp = std::max(ngrp, it.grp + 1);
        nprob = std::max(nprob, it.prob + 1);
    }
    L.ngrp = ngrp;
    L.nprob = nprob;
    BA_CUDA_TRY(cudaMalloc(&L.cnt, sizeof(int) * ngrp));
    BA_CUDA_TRY(cudaMemset(L.cnt, 0, sizeof(int) * ngrp));
    BA_CUDA_TRY(cudaMalloc(&L.part, sizeof(double) * 9 * (v.size() > 0 ? v.size() : 1)));
    if (W > 0) {
        int64_t* dw = nullptr;
        BA_CUDA_TRY(cudaMalloc(&dw, sizeof(int64_t) * wptr.size()));
        BA_CUDA_TRY(cudaMemcpy(dw, wptr.data(), sizeof(int64_t) * wptr.size(), cudaMemcpyHostToDevice));
        L.wptr = dw;
        L.nw = W;
    }
}

// The tile-streaming products of every mode, precision and shape used here.
template <typename T, int MODE, bool ZH, bool SYM, int CFG>
static void set_spmv_attr() {
    BA_CUDA_TRY(cudaFuncSetAttribute(k_spmv<T, MODE, ZH, SYM, CFG>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     int(spmv_smem<T, CFG>())));
}
template <int CFG>
static void set_spmv_attrs() {
    set_spmv_attr<float, 0, true, true, CFG>();
    set_spmv_attr<float, 1, true, true, CFG>();
    set_spmv_attr<float, 2, true, true, CFG>();
    set_spmv_attr<double, 0, true, false, CFG>();
    set_spmv_attr<double, 0, false, false, CFG>();
    set_spmv_attr<double, 1, true, false, CFG>();
}

static void set_smem_attrs() {
    static bool done = false;
    if (done) return;
    set_spmv_attrs<0>();
    set_spmv_attrs<1>();
    set_spmv_attrs<2>();
    for (auto mm : {k_spmm<float, 2>, k_spmm<float, 4>})
        BA_CUDA_TRY(cudaFuncSetAttribute(mm, cudaFuncAttributeMaxDynamicSharedMemorySize, int(spmm_smem<float>())));
    BA_CUDA_TRY(cudaFuncSetAttribute(k_one_cta, cudaFuncAttributeMaxDynamicSharedMemorySize, int(one_smem(kOneCams))));
    BA_CUDA_TRY(cudaFuncSetAttribute(k_pcg_cluster, cudaFuncAttributeMaxDynamicSharedMemorySize, int(clu_smem(kCluCams))));
    done = true;
}

template <typename T>
static int spmv_warps(int cfg) {
    return cfg == 1 ? SpmvShape<T, 1>::kWarps : (cfg == 2 ? SpmvShape<T, 2>::kWarps : SpmvShape<T, 0>::kWarps);
}

// (Re)build the work lists when the chunk rule, the subset layout or the warps of the kernel that
// streams a list changed.  Full pattern: k_spmm (float32) or k_spmv (float64); upper triangle and
// subset segments: k_spmv.
static void ensure_items(Solver* w, const Structure& s, int n_dirs, int forced_cb, bool fp32, int cfg) {
    const int cb = forced_cb > 0 ? forced_cb : 0;
    const int64_t sms = num_sms();
    const int64_t ng = fp32 ? SpmmCfg::kWarps : spmv_warps<double>(cfg);
    const int64_t nu = spmv_warps<float>(cfg), nl = spmv_warps<double>(cfg);
    const int64_t wg = sms * ng, wu = sms * nu, wl = sms * nl;
    const bool fresh = !w->items_g.items || w->items_cb != cb;
    if (fresh || w->items_g.nw != wg) {
        upload_items(w->items_g, build_items(s.h_row_ptr, s.h_col, w->lay, false, cb, fp32, cfg), wg, ng);
        if (w->mm_part) cudaFree(w->mm_part);
        w->mm_part = nullptr;
        BA_CUDA_TRY(cudaMalloc(&w->mm_part, sizeof(double) * kMaxDirs * 9 * size_t(w->items_g.n > 0 ? w->items_g.n : 1)));
        ++w->epoch;
    }
    if (!s.h_row_ptr_u.empty() && (fresh || w->items_u.nw != wu)) {
        upload_items(w->items_u, build_items(s.h_row_ptr_u, s.h_col_u, w->lay, false, cb, fp32, cfg), wu, nu);
        ++w->epoch;
    }
    if (fresh) {
        w->items_l_dirs = -1;
        w->items_cb = cb;
    }
    if (n_dirs > 1 && (w->items_l_dirs != n_dirs || w->items_l.nw != wl)) {
        upload_items(w->items_l, build_items(s.h_row_ptr, s.h_col, w->lay, true, cb, fp32, cfg), wl, nl);
        w->items_l_dirs = n_dirs;
        ++w->epoch;
    }
    w->use_l = n_dirs > 1;
    w->col_lanes = n_dirs <= 8 ? 2 : 4;
    set_smem_attrs();
}

static int grid_for_host(int64_t n) {
    int64_t g = (n + kThreads - 1) / kThreads;
    int cap = num_sms() * 8;
    return int(g < 1 ? 1 : (g > cap ? cap : g));
}

// Per-problem layout of a solve and the grid widths; buffers grow to fit.
static void prepare(Solver* w, const Structure& s, const SolveArgs& a, int n_dirs, bool fp32) {
    const int nb = int(s.h_cam_off.size()) - 1;
    std::vector<Layout> lay(nb);
    int64_t hoff = 0, phoff = 0, boff = 0;
    int nc_max = 1;
    for (int b = 0; b < nb; ++b) {
        Layout& L = lay[b];
        L.c0 = s.h_cam_off[b];
        L.nc = s.h_cam_off[b + 1] - L.c0;
        nc_max = std::max(nc_max, L.nc);
        const int nd = a.mcg ? n_dirs : 1;
        L.sz = (L.nc + nd - 1) / nd;
        L.n_eff = (L.nc + L.sz - 1) / L.sz;
        L.K = (L.sz + kChunkCams - 1) / kChunkCams;
        int64_t cap = 1;
        if (a.mcg) {
            cap = a.max_history > 0 ? a.max_history : int64_t(a.max_iters) * L.n_eff + 1;
            if (cap < 1 + L.n_eff) cap = 1 + L.n_eff;
            if (cap > (int64_t(1) << 30)) throw Error(BA_ERR_INVALID_ARG, "direction history too large");
        }
        L.cap = int(cap);
        L.hoff = hoff;
        L.phoff = phoff;
        L.boff = boff;
        // (a problem that one CTA solves keeps its history in whole tiles of columns; 16-byte aligned)
        const int64_t cols = fp32 && solved_alone(L, true, a.mcg != 0) ? (cap + kOneTile - 1) / kOneTile * kOneTile : cap;
        hoff += (cols * 9 * int64_t(L.nc) + 3) / 4 * 4;
        phoff += cap * L.n_eff * L.K;
        boff += cap;
    }
    const int64_t n = 9 * int64_t(s.n_c);
    const size_t elt = fp32 ? 4 : 8;
    const int G = num_sms() * 2;
    w->nb = nb;
    w->n = n;
    w->mi1 = std::max(w->mi1, a.max_iters + 1);
    w->gx = int(std::min<int64_t>(std::max(1, 4 * G / nb), (9 * int64_t(nc_max) + kThreads - 1) / kThreads));
    if (nc_max > kMaxProblemCams) throw Error(BA_ERR_INVALID_ARG, "too many cameras in one problem");
    w->gu = (nc_max + kUpdCams - 1) / kUpdCams;
    w->gg = int(std::min<int64_t>(G, (9 * int64_t(nc_max) + kGramRows - 1) / kGramRows));
    w->gq = std::max(1, G / nb);
    w->gpq = int(std::max<int64_t>(1, std::min<int64_t>((9 * int64_t(nc_max) + 31) / 32, 4 * G / nb)));
    w->gphi = std::max(1, 4 * G / nb);
    w->gb = std::max(1, G / nb);
    w->phi_rows = 1;
    for (const Layout& L : lay) w->phi_rows = std::max(w->phi_rows, 9 * ((L.sz + L.K - 1) / L.K));
    w->gcol = std::min(nc_max, std::max(1, 16 * G / nb));
    if (!w->h_ctl || int(w->lay.size()) != nb) {
        if (w->h_ctl) cudaFreeHost(w->h_ctl);
        if (w->h_outer) cudaFreeHost(w->h_outer);
        w->h_ctl = nullptr;
        w->h_outer = nullptr;
        BA_CUDA_TRY(cudaMallocHost(&w->h_ctl, sizeof(Ctl) * nb));
        BA_CUDA_TRY(cudaMallocHost(&w->h_outer, sizeof(Outer) * nb));
    }
    if (!w->cap_stream) BA_CUDA_TRY(cudaStreamCreateWithFlags(&w->cap_stream, cudaStreamNonBlocking));
    if (!w->cap2) BA_CUDA_TRY(cudaStreamCreateWithFlags(&w->cap2, cudaStreamNonBlocking));
    if (!w->cap3) BA_CUDA_TRY(cudaStreamCreateWithFlags(&w->cap3, cudaStreamNonBlocking));
    if (!w->cap_side) BA_CUDA_TRY(cudaStreamCreateWithFlags(&w->cap_side, cudaStreamNonBlocking));
    if (!w->ev_fork) BA_CUDA_TRY(cudaEventCreateWithFlags(&w->ev_fork, cudaEventDisableTiming));
    if (!w->ev_join) BA_CUDA_TRY(cudaEventCreateWithFlags(&w->ev_join, cudaEventDisableTiming));
    if (!w->h_params) BA_CUDA_TRY(cudaMallocHost(&w->h_params, sizeof(Params)));
    if (!w->h_loops) BA_CUDA_TRY(cudaMallocHost(&w->h_loops, sizeof(Loops)));
    grow(w->P, size_t(hoff) * elt);
    grow(w->Q, size_t(hoff) * elt);
    grow(w->r, size_t(n) * elt);
    grow(w->z, size_t(n) * elt);
    grow(w->xw, size_t(n) * elt);
    grow(w->PT, size_t(n) * kMaxDirs * elt);
    grow(w->part_a, size_t(nb) * w->gg * kGramMax * sizeof(double));
    const size_t wide = fp32 ? sizeof(WideSlot<float>) : sizeof(WideSlot<double>);
    grow(w->part_b, size_t(nb) * w->gu * wide);
    grow(w->part_cam, size_t(s.n_c) * 3 * sizeof(double));
    grow(w->dpinv, size_t(nb) * w->mi1 * kMaxDirs * kMaxDirs * sizeof(double));
    grow(w->beta, size_t(boff) * kMaxDirs * sizeof(double));
    grow(w->phip, size_t(phoff) * wide);
    // the largest problem that k_one_cta (float32) or k_pcg_cluster (float64 PCG) solves
    w->one_cams = 0;
    w->all_small = true;
    for (const Layout& L : lay) {
        if (solved_alone(L, fp32, a.mcg != 0) && a.wait_polls > 0) w->one_cams = std::max(w->one_cams, L.nc);
        else w->all_small = false;
    }
    if (fp32 && w->one_cams > 0) grow(w->colblk, size_t(boff) * sizeof(int));
    grow(w->hist, size_t(nb) * w->mi1 * sizeof(double));
    grow(w->blk_off, size_t(nb) * w->mi1 * sizeof(int));
    grow(w->blk_w, size_t(nb) * w->mi1 * sizeof(int));
    grow(w->ctl, size_t(nb) * sizeof(Ctl));
    grow(w->outer, size_t(nb) * sizeof(Outer));
    grow(w->rt, size_t(n) * sizeof(double));
    const void* lay_p = w->lay_d.p;
    grow(w->lay_d, size_t(nb) * sizeof(Layout));
    grow(w->dpart, size_t(nb) * w->gu * 3 * wide);
    grow(w->dtot, size_t(nb) * 2 * sizeof(double));
    grow(w->camdot, size_t(s.n_c) * 2 * sizeof(double));
    grow(w->params, sizeof(Params));
    grow(w->loops, sizeof(Loops));
    if (w->h_hist_n < size_t(nb) * w->mi1) {
        if (w->h_hist) cudaFreeHost(w->h_hist);
        w->h_hist = nullptr;
        w->h_hist_n = 0;
        BA_CUDA_TRY(cudaMallocHost(&w->h_hist, sizeof(double) * size_t(nb) * w->mi1));
        w->h_hist_n = size_t(nb) * w->mi1;
    }
    // the layouts change with the solver and its options, not from solve to solve: the upload (a host wait of
    // about 10 us) is skipped when the device holds them already
    if (lay_p != w->lay_d.p || w->lay.size() != lay.size() ||
        std::memcmp(w->lay.data(), lay.data(), sizeof(Layout) * lay.size()) != 0) {
        w->lay.clear();
        BA_CUDA_TRY(cudaMemcpy(w->lay_d.p, lay.data(), sizeof(Layout) * nb, cudaMemcpyHostToDevice));
        w->lay = lay;
    }
    w->spmv_cfg = a.spmv_cfg >= 0 && a.spmv_cfg < kSpmvShapes ? a.spmv_cfg : 0;
    ensure_items(w, s, a.mcg ? n_dirs : 1, a.item_blocks, fp32, w->spmv_cfg);
    w->items_g.polls = a.wait_polls;
    w->items_l.polls = a.wait_polls;
    w->items_u.polls = a.wait_polls;
    if (fp32 && s.n_up > 0) grow(w->tb, size_t(s.n_up) * (kTbHead + 1) * sizeof(float));
}

static void free_buf(Buf& b) {
    if (b.p) cudaFree(b.p);
    b = Buf();
}

Solver* solver_create() { return new Solver(); }

// A warp whose tile wait gave up left its work item uncounted, so its group's arrival counter did not return to
// zero and the next product would take the last chunk too early (or never): a solve that timed out clears
// the counters of every list.
static void clear_counters(Solver* w, cudaStream_t st) {
    for (ItemList* l : {&w->items_g, &w->items_l, &w->items_u})
        if (l->cnt) BA_CUDA_TRY(cudaMemsetAsync(l->cnt, 0, sizeof(int) * l->ngrp, st));
}

void solver_interrupt_products(Solver* w, cudaStream_t st) {
    for (ItemList* l : {&w->items_g, &w->items_l, &w->items_u})
        if (l->cnt) BA_CUDA_TRY(cudaMemsetAsync(l->cnt, 1, sizeof(int) * l->ngrp, st));   // no group's count
    clear_counters(w, st);
    BA_CUDA_TRY(cudaStreamSynchronize(st));
}

void solver_destroy(Solver* w) {
    if (!w) return;
    Buf* bufs[] = {&w->P, &w->Q, &w->r, &w->z, &w->xw, &w->PT, &w->part_a, &w->part_b, &w->part_cam, &w->dpinv,
                   &w->beta, &w->colblk, &w->phip, &w->hist, &w->blk_off, &w->blk_w, &w->ctl, &w->outer, &w->rt,
                   &w->lay_d, &w->dpart, &w->dtot, &w->camdot, &w->params, &w->loops};
    for (Buf* b : bufs) free_buf(*b);
    for (SolveExec* e : w->execs) {
        cudaGraphExecDestroy(e->exec);
        delete e;
    }
    free_items(w->items_g);
    free_items(w->items_l);
    free_items(w->items_u);
    free_buf(w->tb);
    if (w->mm_part) cudaFree(w->mm_part);
    if (w->h_ctl) cudaFreeHost(w->h_ctl);
    if (w->h_outer) cudaFreeHost(w->h_outer);
    if (w->h_params) cudaFreeHost(w->h_params);
    if (w->h_loops) cudaFreeHost(w->h_loops);
    if (w->h_hist) cudaFreeHost(w->h_hist);
    if (w->ev0) cudaEventDestroy(w->ev0);
    if (w->ev1) cudaEventDestroy(w->ev1);
    if (w->cap_stream) cudaStreamDestroy(w->cap_stream);
    if (w->cap2) cudaStreamDestroy(w->cap2);
    if (w->cap3) cudaStreamDestroy(w->cap3);
    if (w->cap_side) cudaStreamDestroy(w->cap_side);
    if (w->ev_fork) cudaEventDestroy(w->ev_fork);
    if (w->ev_join) cudaEventDestroy(w->ev_join);
    delete w;
}

int solver_history(const Solver* w, int problem, const double** hist) {
    if (problem < 0 || problem >= int(w->host_hist.size())) {
        *hist = nullptr;
        return 0;
    }
    *hist = w->host_hist[problem].data();
    return static_cast<int>(w->host_hist[problem].size());
}

// One launch of k_spmv in shape `cfg` (one CTA per SM).
// Launch with programmatic stream serialization (the kernels of a solve iteration): the kernel may
// be scheduled while the previous kernel on the stream drains and waits for it in wait_prior_grid,
// its first statement, instead of starting only after the previous grid has retired.
template <typename... K, typename... A>
static void launch_chained(void (*kern)(K...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A&&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    BA_CUDA_TRY(cudaLaunchKernelEx(&cfg, kern, std::forward<A>(args)...));
}

template <typename T, int MODE, bool ZH, bool SYM, int CFG>
static void launch_spmv_cfg(cudaStream_t st, const int64_t* row_ptr, const int64_t* tile_ptr, const int32_t* col,
                            const T* S, const T* z, const ItemList& L, int sel, T* out, const T* rvec, double* camdot,
                            Ctl* ctl, T* tb, T* tb8, const int32_t* cslot) {
    launch_chained(k_spmv<T, MODE, ZH, SYM, CFG>, dim3(num_sms()), dim3(SpmvShape<T, CFG>::kWarps * 32),
                   spmv_smem<T, CFG>(), st, row_ptr, tile_ptr, col, S, z, L, sel, out, rvec, camdot, ctl, tb, tb8,
                   cslot);
}
template <typename T, int MODE, bool ZH, bool SYM>
static void launch_spmv(int cfg, cudaStream_t st, const int64_t* row_ptr, const int64_t* tile_ptr, const int32_t* col,
                        const T* S, const T* z, const ItemList& L, int sel, T* out, const T* rvec, double* camdot,
                        Ctl* ctl, T* tb, T* tb8 = nullptr, const int32_t* cslot = nullptr) {
    if (cfg == 1)
        launch_spmv_cfg<T, MODE, ZH, SYM, 1>(st, row_ptr, tile_ptr, col, S, z, L, sel, out, rvec, camdot, ctl, tb, tb8,
                                             cslot);
    else if (cfg == 2)
        launch_spmv_cfg<T, MODE, ZH, SYM, 2>(st, row_ptr, tile_ptr, col, S, z, L, sel, out, rvec, camdot, ctl, tb, tb8,
                                             cslot);
    else
        launch_spmv_cfg<T, MODE, ZH, SYM, 0>(st, row_ptr, tile_ptr, col, S, z, L, sel, out, rvec, camdot, ctl, tb, tb8,
                                             cslot);
}

// A one-column product y = S z, z a column of the direction history (modes of k_spmv).  With the upper
// triangle Su (float32) it is the symmetric product in two launches; float64 streams the full
// pattern (its products are bound by the float64 pipe, which halving the bytes would not relieve).
// Returns the launches.
template <typename T, int MODE>
static int enqueue_product(Solver* w, const Structure& s, const T* S, const T* Su, const T* zsrc, int sel, T* out,
                           const T* rvec, cudaStream_t st) {
    Ctl* ctl = ptr<Ctl>(w->ctl);
    double* camdot = MODE == 1 ? ptr<double>(w->camdot) : nullptr;
    if (Su) {
        T* tb = ptr<T>(w->tb);
        T* tb8 = tb + kTbHead * s.n_up;
        launch_spmv<T, MODE, true, true>(w->spmv_cfg, st, s.row_ptr_u, s.tile_ptr_u, s.col_u, Su, zsrc, w->items_u,
                                         sel, out, rvec, camdot, ctl, tb, tb8, s.cslot);
        launch_chained(k_spmv_col<T, MODE, true>, dim3(w->gcol, w->nb), dim3(kColWarps * 32), 0, st, s.qptr,
                       (const T*)tb, (const T*)tb8, zsrc, sel, out, rvec, camdot, ctl);
        return 2;
    }
    launch_spmv<T, MODE, true, false>(w->spmv_cfg, st, s.row_ptr, s.tile_ptr, s.col, S, zsrc, w->items_g, sel, out,
                                      rvec, camdot, ctl, nullptr);
    return 1;
}

// A batch of this many problems fills the chip with small CTAs; fewer problems are spread over large CTAs and
// clusters.  The results are the same bits.
static bool many_problems(int nb) { return kSmallCtas * nb > num_sms(); }

// Enqueue one iteration of the chosen algorithm for every problem on `st`; returns the launches.
template <typename T>
static int enqueue_iteration(Solver* w, const Structure& s, const T* S, const T* Su, const double* Dinv, T* x,
                             bool mcg, cudaStream_t st) {
    const int nb = w->nb;
    T* P = ptr<T>(w->P);
    T* Q = ptr<T>(w->Q);
    T* r = ptr<T>(w->r);
    T* z = ptr<T>(w->z);
    Ctl* ctl = ptr<Ctl>(w->ctl);
    const int Gt = num_sms();   // tile-streaming products: one CTA per SM
    if (!mcg) {
        const int np = enqueue_product<T, 1>(w, s, S, Su, P, kSelLive, Q, r, st);
        launch_chained(k_pcg_update<T>, dim3(w->gu, nb), dim3(kUpdThreads), 0, st, Dinv, P, Q, x, r, z,
                       ptr<double>(w->camdot), ptr<WideSlot<T>>(w->dpart), ptr<double>(w->dtot), ctl);
        launch_chained(k_pcg_dir<T>, dim3(w->gq, nb), dim3(kThreads), 0, st, z, P, ptr<WideSlot<T>>(w->dpart), w->gu,
                       ptr<double>(w->dtot), ptr<double>(w->hist), ctl);
        return np + 2;
    } else {
        if (many_problems(nb))
            launch_chained(k_mcg_gram<T, kGramFew>, dim3(w->gg, nb), dim3(kGramFew), 0, st, P, Q, r,
                           ptr<double>(w->part_a), w->gg, ctl);
        else
            launch_chained(k_mcg_gram<T, kGramThreads>, dim3(std::min(w->gg, std::max(1, 2 * num_sms() / nb)), nb),
                           dim3(kGramThreads), 0, st, P, Q, r, ptr<double>(w->part_a), w->gg, ctl);
        if (many_problems(nb) && w->gg <= kSmallGroups)
            launch_chained(k_mcg_small_few<T>, dim3(nb), dim3(kSmallFew), 0, st, ctl, ptr<double>(w->part_a), w->gg,
                           ptr<double>(w->dpinv), w->mi1);
        else
            launch_chained(k_mcg_small<T>, dim3(nb * kSmallCtas), dim3(kSmallThreads), 0, st, ctl, ptr<double>(w->part_a),
                           w->gg, ptr<double>(w->dpinv), w->mi1);
        launch_chained(k_mcg_update<T>, dim3(w->gu, nb), dim3(kUpdThreads), 0, st, Dinv, P, Q, x, r, z,
                       ptr<WideSlot<T>>(w->dpart), ctl);
        auto phi = w->phi_rows <= 64 ? k_mcg_phi<T, 2> : w->phi_rows <= 128 ? k_mcg_phi<T, 4> : k_mcg_phi<T, 8>;
        launch_chained(phi, dim3(w->gphi + 1, nb), dim3(kThreads), 0, st, Q, z, ptr<WideSlot<T>>(w->phip),
                       ptr<WideSlot<T>>(w->dpart), w->gu, ptr<double>(w->hist), ptr<int>(w->blk_off),
                       ptr<int>(w->blk_w), w->mi1, ctl);
        T* betat = ptr<T>(w->beta);
        launch_chained(k_mcg_beta<T>, dim3(w->gb, nb), dim3(kThreads), 0, st, ptr<WideSlot<T>>(w->phip),
                       ptr<double>(w->dpinv), ptr<int>(w->blk_off), ptr<int>(w->blk_w), betat, ctl, w->mi1);
        if constexpr (sizeof(T) == 8) {
            // Eq. 18: Q_{i+1} = S Z_{i+1} - sum_j Q_j beta_{i,j}; S Z over whole rows for the
            // problems forming a global block, over the subset segments for the local ones
            launch_spmv<T, 0, false, false>(w->spmv_cfg, st, s.row_ptr, s.tile_ptr, s.col, S, z, w->items_g,
                                            w->use_l ? kSelGlobal : kSelLive, Q, nullptr, nullptr, ctl, nullptr);
            if (w->use_l)
                launch_spmv<T, 0, false, false>(w->spmv_cfg, st, s.row_ptr, s.tile_ptr, s.col, S, z, w->items_l,
                                                kSelLocal, Q, nullptr, nullptr, ctl, nullptr);
            launch_chained(k_mcg_pq<T, 1>, dim3(w->gpq, nb), dim3(PqShape<T>::kSlices * 32), 0, st, P, Q, z, betat,
                           (T*)nullptr, ctl);
            return w->use_l ? 8 : 7;
        } else {
            // Algorithm 2: Q_{i+1} = S P_{i+1}
            // two rows per lane once they still give nearly every SM a CTA (a row's sum is the same either way)
            const bool many = many_problems(nb) && w->col_lanes == 2;   // up to 8 directions
            auto pq = many ? k_mcg_pq<T, 1, kPqFew> : w->n >= int64_t(48) * Gt ? k_mcg_pq<T, 2> : k_mcg_pq<T, 1>;
            launch_chained(pq, dim3(w->gpq, nb), dim3((many ? kPqFew : PqShape<T>::kSlices) * 32), 0, st, P, Q, z, betat,
                           ptr<T>(w->PT), ctl);
            const int np = enqueue_product<T, 2>(w, s, S, Su, P, kSelW1, Q, nullptr, st);
            auto mm = w->col_lanes == 2 ? k_spmm<T, 2> : k_spmm<T, 4>;
            launch_chained(mm, dim3(Gt), dim3(SpmmCfg::kWarps * 32), spmm_smem<T>(), st, s.row_ptr, s.tile_ptr,
                           s.col, S, ptr<T>(w->PT), w->items_g, static_cast<T*>(w->mm_part), Q, ctl);
            return 7 + np;
        }
    }
}

// x = 0, r = sign * rhs, z = D^{-1} r, P_0 = z and the control blocks (small: of problems solved alone too);
// returns the launches.
template <typename T>
static int krylov_init(Solver* w, const Structure& s, const T* S, const T* Su, const double* Dinv, const double* rhs,
                       double sign, const double* scale, T* x, const Outer* outer, cudaStream_t st, bool small) {
    const int nb = w->nb;
    k_init_vec<T><<<dim3(w->gu, nb), kUpdThreads, 0, st>>>(ptr<Layout>(w->lay_d), rhs, sign, scale, Dinv, outer, x,
                                                            ptr<T>(w->r), ptr<T>(w->z), ptr<T>(w->P),
                                                            ptr<WideSlot<T>>(w->part_b));
    k_init_ctl<T><<<nb, 32, 0, st>>>(ptr<Ctl>(w->ctl), ptr<Layout>(w->lay_d), ptr<WideSlot<T>>(w->part_b), w->gu,
                                  ptr<Params>(w->params), sizeof(T) == 4 ? kStagnation : 0.0, sizeof(T) == 4 ? 1 : 0,
                                  outer, ptr<int>(w->blk_off), ptr<int>(w->blk_w), w->mi1, small);
    return 2;
}

// The solves of the problems that one CTA or one cluster solves, right after krylov_init (x: the solution
// of a float64 solve); returns the launches.
static int enqueue_small(Solver* w, const Structure& s, const System& y, bool mcg, double* x, cudaStream_t st) {
    if (w->one_cams == 0) return 0;
    if (y.S) {
        k_pcg_cluster<<<w->nb * kSmallCtas, kCluThreads, clu_smem(w->one_cams), st>>>(
            s.row_ptr, s.tile_ptr, s.col, y.S, y.Dinv, x, ptr<double>(w->r), ptr<double>(w->z), ptr<double>(w->hist),
            ptr<Ctl>(w->ctl));
        return 1;
    }
    k_one_cta<<<w->nb, kOneThreads, one_smem(w->one_cams), st>>>(
        mcg, s.row_ptr, s.tile_ptr, s.col, y.S32, y.Dhat, ptr<float>(w->xw), ptr<float>(w->r), ptr<float>(w->z),
        ptr<float>(w->P), ptr<float>(w->Q), ptr<WideSlot<float>>(w->phip), ptr<double>(w->dpinv), ptr<float>(w->beta),
        ptr<int>(w->colblk), ptr<double>(w->hist), ptr<int>(w->blk_off), ptr<int>(w->blk_w), w->mi1, ptr<Ctl>(w->ctl));
    return 1;
}

// problems solved alone in a batch with others
static bool beside(const Solver* w) { return w->one_cams > 0 && !w->all_small; }
static void join_small(Solver* w, cudaStream_t st) {
    if (beside(w)) BA_CUDA_TRY(cudaStreamWaitEvent(st, w->ev_join));
}

// The start of a sweep: krylov_init, the problems that are solved whole, and Q_0 = S P_0 of the others, from
// which Algorithm 2 starts its iterations (Algorithm 1 forms Q = S P first in every one).  Problems that are
// solved whole form their own Q_0 and are done for everyone else: they take part in no tile-streaming
// product, so no tile wait can end them.  In a batch with larger problems they run on a branch of the graph
// (stream side, joined by join_small) beside the others' iterations: one after the other, 8 problems of 20
// cameras and 8 of 300 took 11.8 ms to 1e-9 (MCG, 8 directions), beside each other 9.9 ms; the 300s alone 8.9.
// Returns the launches.
template <typename T>
static int krylov_start(Solver* w, const Structure& s, const System& y, const T* S, const T* Su, const double* Dinv,
                        const double* rhs, double sign, const double* scale, T* x, const Outer* outer, bool mcg,
                        cudaStream_t st, cudaStream_t side) {
    int n = krylov_init<T>(w, s, S, Su, Dinv, rhs, sign, scale, x, outer, st, w->one_cams > 0);
    if (!beside(w)) side = nullptr;
    if (side) {
        BA_CUDA_TRY(cudaEventRecord(w->ev_fork, st));
        BA_CUDA_TRY(cudaStreamWaitEvent(side, w->ev_fork));
    }
    n += enqueue_small(w, s, y, mcg, sizeof(T) == 8 ? reinterpret_cast<double*>(x) : nullptr, side ? side : st);
    if (side) BA_CUDA_TRY(cudaEventRecord(w->ev_join, side));
    if (mcg && !w->all_small) n += enqueue_product<T, 0>(w, s, S, Su, ptr<T>(w->P), kSelLive, ptr<T>(w->Q), nullptr, st);
    return n;
}

// true residual t = -b~ - S x into out (may be null) and, per problem, its norms into ctl (true_rr,
// bb): explicit tiled S in float64 precision, the implicit operator (double-float arithmetic) in mixed precision.
static int true_residual(Solver* w, const Structure& s, const System& y, const double* x, double* out,
                         cudaStream_t st) {
    int n = 0, sums = 2;
    if (y.S) {
        k_true_residual<<<grid_for_host(int64_t(s.n_c) * 32), kThreads, 0, st>>>(
            s.n_c, s.row_ptr, s.tile_ptr, s.col, y.S, x, y.bt, out, ptr<double>(w->part_cam));
        n = 1;
    } else {
        n = launch_implicit_residual(s, y, x, out, ptr<double>(w->part_cam), st);
        sums = 3;
    }
    k_true_reduce<<<w->nb, 32 * sums, 0, st>>>(ptr<Ctl>(w->ctl), ptr<double>(w->part_cam), sums);
    return n + 1;
}

// ---- the solve graph: conditional WHILE nodes inserted into a stream capture ------------------

// A WHILE node on handle h after the current capture frontier of stream cs; the capture goes on after
// it.  Returns the (empty) body graph.
static cudaGraph_t capture_while(cudaStream_t cs, cudaGraphConditionalHandle h) {
    cudaStreamCaptureStatus stat;
    cudaGraph_t g = nullptr;
    const cudaGraphNode_t* deps = nullptr;
    size_t nd = 0;
    BA_CUDA_TRY(cudaStreamGetCaptureInfo(cs, &stat, nullptr, &g, &deps, nullptr, &nd));
    cudaGraphNodeParams np = {};
    np.type = cudaGraphNodeTypeConditional;
    np.conditional.handle = h;
    np.conditional.type = cudaGraphCondTypeWhile;
    np.conditional.size = 1;
    cudaGraphNode_t node;
    BA_CUDA_TRY(cudaGraphAddNode(&node, g, deps, nullptr, nd, &np));
    BA_CUDA_TRY(cudaStreamUpdateCaptureDependencies(cs, &node, nullptr, 1, cudaStreamSetCaptureDependencies));
    return np.conditional.phGraph_out[0];
}

// A conditional handle of the graph being captured on cs (no default: set before the node runs).
static cudaGraphConditionalHandle capture_handle(cudaStream_t cs) {
    cudaStreamCaptureStatus stat;
    cudaGraph_t g = nullptr;
    BA_CUDA_TRY(cudaStreamGetCaptureInfo(cs, &stat, nullptr, &g, nullptr, nullptr, nullptr));
    cudaGraphConditionalHandle h;
    BA_CUDA_TRY(cudaGraphConditionalHandleCreate(&h, g, 0, 0));
    return h;
}

// The Krylov loop of one sweep, captured on cs: the sweep's start, then WHILE(any problem running) {
// chunk iterations; loop condition } on the body stream cb.
// Sets *pre (launches before the loop) and *per_pass (launches per pass of the loop).
template <typename T>
static void capture_krylov(Solver* w, const Structure& s, const System& y, const T* S, const T* Su, const double* Dinv,
                           const double* rhs, double sign, const double* scale, T* x, const Outer* outer, bool mcg,
                           int chunk, cudaStream_t cs, cudaStream_t cb, int* pre, int* per_pass) {
    const cudaGraphConditionalHandle h = capture_handle(cs);
    *pre = krylov_start<T>(w, s, y, S, Su, Dinv, rhs, sign, scale, x, outer, mcg, cs, w->cap_side) + 1;
    k_loop_cond<<<1, kThreads, 0, cs>>>(h, 1, ptr<Ctl>(w->ctl), w->nb, ptr<Loops>(w->loops), 1, chunk,
                                        ptr<Params>(w->params));
    cudaGraph_t body = capture_while(cs, h);
    BA_CUDA_TRY(cudaStreamBeginCaptureToGraph(cb, body, nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal));
    *per_pass = 1;
    for (int k = 0; k < chunk; ++k) *per_pass += enqueue_iteration<T>(w, s, S, Su, Dinv, x, mcg, cb);
    launch_chained(k_loop_cond, dim3(1), dim3(kThreads), 0, cb, h, 1, ptr<Ctl>(w->ctl), w->nb, ptr<Loops>(w->loops), 0,
                   chunk, ptr<Params>(w->params));
    cudaGraph_t done = nullptr;
    cudaError_t e = cudaStreamEndCapture(cb, &done);
    if (e != cudaSuccess) throw Error(BA_ERR_CUDA, std::string("loop body capture: ") + cudaGetErrorString(e));
    join_small(w, cs);
}



// Capture and instantiate the whole solve: float64 (Krylov loop and the true residual) or mixed
// precision (WHILE(a problem refines) { float32 Krylov loop; float64 true residual; plan the next
// sweep }).
static cudaGraphExec_t build_solve_graph(Solver* w, const Structure& s, const System& y, const SolveArgs& a,
                                         double* x, GraphCounts& gc) {
    const bool fp32 = a.precision == BA_PRECISION_MIXED;
    const bool mcg = a.mcg != 0;
    const int nb = w->nb;
    const int64_t n = int64_t(s.n_c) * 9;
    cudaStream_t cs = w->cap_stream;
    gc = GraphCounts();
    BA_CUDA_TRY(cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal));
    try {
        if (!fp32) {
            capture_krylov<double>(w, s, y, y.S, nullptr, y.Dinv, y.bt, -1.0, nullptr, x, nullptr, mcg, a.chunk, cs,
                                   w->cap2, &gc.pre, &gc.body);
            gc.post = true_residual(w, s, y, x, nullptr, cs);
        } else {
            k_start_refine<<<grid_for_host(n), kThreads, 0, cs>>>(n, y.bt, x, ptr<double>(w->rt));
            k_outer_init<<<nb, kThreads, 0, cs>>>(ptr<Layout>(w->lay_d), y.bt, y.lam, ptr<Outer>(w->outer));
            const cudaGraphConditionalHandle ho = capture_handle(cs);
            k_refine_plan<<<1, kThreads, 0, cs>>>(ptr<Outer>(w->outer), nb, ptr<Params>(w->params), ho, 1,
                                                  ptr<Loops>(w->loops), 0);
            gc.pre = 3;
            cudaGraph_t body = capture_while(cs, ho);
            cudaStream_t c2 = w->cap2;
            BA_CUDA_TRY(cudaStreamBeginCaptureToGraph(c2, body, nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal));
            int kpre = 0;
            capture_krylov<float>(w, s, y, y.S32, y.S32u, y.Dhat, ptr<double>(w->rt), 1.0, y.lam, ptr<float>(w->xw),
                                  ptr<Outer>(w->outer), mcg, a.chunk, c2, w->cap3, &kpre, &gc.body);
            k_accumulate<<<dim3(w->gx, nb), kThreads, 0, c2>>>(ptr<Layout>(w->lay_d), ptr<Outer>(w->outer),
                                                               ptr<float>(w->xw), y.lam, x, y.xd);
            const int tr = true_residual(w, s, y, x, ptr<double>(w->rt), c2);
            k_refine_after<<<nb, 32, 0, c2>>>(ptr<Ctl>(w->ctl), ptr<Outer>(w->outer), ptr<Params>(w->params));
            k_refine_plan<<<1, kThreads, 0, c2>>>(ptr<Outer>(w->outer), nb, ptr<Params>(w->params), ho, 1,
                                                  ptr<Loops>(w->loops), 1);
            gc.sweep = kpre + 1 + tr + 2;
            cudaGraph_t done = nullptr;
            cudaError_t e = cudaStreamEndCapture(c2, &done);
            if (e != cudaSuccess) throw Error(BA_ERR_CUDA, std::string("refinement body capture: ") + cudaGetErrorString(e));
        }
    } catch (...) {
        cudaGraph_t junk = nullptr;
        cudaStreamEndCapture(cs, &junk);
        if (junk) cudaGraphDestroy(junk);
        cudaGetLastError();
        throw;
    }
    cudaGraph_t g = nullptr;
    cudaError_t e = cudaStreamEndCapture(cs, &g);
    if (e != cudaSuccess) throw Error(BA_ERR_CUDA, std::string("solve graph capture: ") + cudaGetErrorString(e));
    cudaGraphExec_t exec = nullptr;
    e = cudaGraphInstantiate(&exec, g, 0);
    cudaGraphDestroy(g);
    if (e != cudaSuccess) throw Error(BA_ERR_CUDA, std::string("solve graph instantiate: ") + cudaGetErrorString(e));
    return exec;
}

// Host-driven loops (ba_options.host_loop): a plain graph of chunk iterations and the pass counter,
// launched by the host until every problem is done.  gc.body receives its launches.
static cudaGraphExec_t build_chunk_graph(Solver* w, const Structure& s, const System& y, const SolveArgs& a,
                                         double* x, GraphCounts& gc) {
    const bool fp32 = a.precision == BA_PRECISION_MIXED;
    cudaStream_t cs = w->cap_stream;
    gc = GraphCounts();
    gc.body = 1;
    BA_CUDA_TRY(cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal));
    for (int k = 0; k < a.chunk; ++k)
        gc.body += fp32 ? enqueue_iteration<float>(w, s, y.S32, y.S32u, y.Dhat, ptr<float>(w->xw), a.mcg != 0, cs)
                        : enqueue_iteration<double>(w, s, y.S, nullptr, y.Dinv, x, a.mcg != 0, cs);
    k_loop_cond<<<1, kThreads, 0, cs>>>(cudaGraphConditionalHandle(), 0, ptr<Ctl>(w->ctl), w->nb,
                                        ptr<Loops>(w->loops), 0, a.chunk, ptr<Params>(w->params));
    cudaGraph_t g = nullptr;
    cudaError_t e = cudaStreamEndCapture(cs, &g);
    if (e != cudaSuccess) throw Error(BA_ERR_CUDA, std::string("chunk graph capture: ") + cudaGetErrorString(e));
    cudaGraphExec_t exec = nullptr;
    e = cudaGraphInstantiate(&exec, g, 0);
    cudaGraphDestroy(g);
    if (e != cudaSuccess) throw Error(BA_ERR_CUDA, std::string("chunk graph instantiate: ") + cudaGetErrorString(e));
    return exec;
}

// Launch the chunk graph until every problem's Ctl says done (at most the loop bound); returns the
// launches and counts the host waits.
static int64_t host_krylov_loop(Solver* w, cudaGraphExec_t chunk_exec, const GraphCounts& gc, const SolveArgs& a,
                                cudaStream_t st, int* waits) {
    const int nb = w->nb;
    const int bound = a.max_iters / a.chunk + 2;
    int64_t launches = 0;
    for (int c = 0; c <= bound; ++c) {
        BA_CUDA_TRY(cudaMemcpyAsync(w->h_ctl, w->ctl.p, sizeof(Ctl) * nb, cudaMemcpyDeviceToHost, st));
        BA_CUDA_TRY(cudaStreamSynchronize(st));
        ++*waits;
        bool all_done = true;
        for (int b = 0; b < nb && all_done; ++b) all_done = w->h_ctl[b].done != 0;
        if (all_done || c == bound) break;
        BA_CUDA_TRY(cudaGraphLaunch(chunk_exec, st));
        launches += gc.body;
    }
    return launches;
}

static void run_host_loops(Solver* w, const Structure& s, const System& y, const SolveArgs& a, double* x,
                           cudaGraphExec_t chunk_exec, const GraphCounts& gc, cudaStream_t st, int* waits) {
    const bool fp32 = a.precision == BA_PRECISION_MIXED;
    const int nb = w->nb;
    const int64_t n = int64_t(s.n_c) * 9;
    Loops* lp = ptr<Loops>(w->loops);
    const Params* prm = ptr<Params>(w->params);
    const cudaGraphConditionalHandle none = cudaGraphConditionalHandle();
    int64_t launches = 0;
    if (!fp32) {
        launches += krylov_start<double>(w, s, y, y.S, nullptr, y.Dinv, y.bt, -1.0, nullptr, x, nullptr, a.mcg != 0, st,
                                         nullptr);
        k_loop_cond<<<1, kThreads, 0, st>>>(none, 0, ptr<Ctl>(w->ctl), nb, lp, 1, a.chunk, prm);
        launches += 1 + host_krylov_loop(w, chunk_exec, gc, a, st, waits);
        launches += true_residual(w, s, y, x, nullptr, st);
    } else {
        k_start_refine<<<grid_for_host(n), kThreads, 0, st>>>(n, y.bt, x, ptr<double>(w->rt));
        k_outer_init<<<nb, kThreads, 0, st>>>(ptr<Layout>(w->lay_d), y.bt, y.lam, ptr<Outer>(w->outer));
        k_refine_plan<<<1, kThreads, 0, st>>>(ptr<Outer>(w->outer), nb, prm, none, 0, lp, 0);
        launches += 3;
        for (int sweep = 0; sweep <= a.max_refine; ++sweep) {
            BA_CUDA_TRY(cudaMemcpyAsync(w->h_outer, w->outer.p, sizeof(Outer) * nb, cudaMemcpyDeviceToHost, st));
            BA_CUDA_TRY(cudaStreamSynchronize(st));
            ++*waits;
            bool any = false;
            for (int b = 0; b < nb && !any; ++b) any = w->h_outer[b].swept != 0;
            if (!any) break;
            launches += krylov_start<float>(w, s, y, y.S32, y.S32u, y.Dhat, ptr<double>(w->rt), 1.0, y.lam,
                                            ptr<float>(w->xw), ptr<Outer>(w->outer), a.mcg != 0, st, nullptr);
            k_loop_cond<<<1, kThreads, 0, st>>>(none, 0, ptr<Ctl>(w->ctl), nb, lp, 1, a.chunk, prm);
            launches += 1 + host_krylov_loop(w, chunk_exec, gc, a, st, waits);
            k_accumulate<<<dim3(w->gx, nb), kThreads, 0, st>>>(ptr<Layout>(w->lay_d), ptr<Outer>(w->outer),
                                                               ptr<float>(w->xw), y.lam, x, y.xd);
            launches += 1 + true_residual(w, s, y, x, ptr<double>(w->rt), st);
            k_refine_after<<<nb, 32, 0, st>>>(ptr<Ctl>(w->ctl), ptr<Outer>(w->outer), prm);
            k_refine_plan<<<1, kThreads, 0, st>>>(ptr<Outer>(w->outer), nb, prm, none, 0, lp, 1);
            launches += 2;
        }
    }
    BA_CUDA_TRY(cudaGetLastError());
    w->launches = launches;
}

// The instantiated graph for this solve (kept for the next solve of the same kind; a few kinds are
// kept, e.g. PCG and MCG in turn, and graphs that hold freed buffers are dropped).
static cudaGraphExec_t solve_graph(Solver* w, const Structure& s, const System& y, const SolveArgs& a, double* x,
                                   GraphCounts& gc) {
    const bool fp32 = a.precision == BA_PRECISION_MIXED;
    GraphKey key;
    key.mcg = a.mcg;
    key.fp32 = fp32;
    key.chunk = a.chunk;
    key.mi1 = w->mi1;
    key.use_l = w->use_l;
    key.epoch = w->epoch;
    key.polls = a.wait_polls;
    key.nb = w->nb;
    key.host = a.host_loop;
    key.cfg = a.spmv_cfg;
    key.one = w->one_cams;
    key.all = w->all_small;
    key.phi = w->phi_rows;
    key.lanes = w->col_lanes;
    key.allocs = g_allocs.load();
    const void* ptrs[4] = {x, fp32 ? (const void*)y.S32 : (const void*)y.S, w->items_g.items, w->items_l.items};
    for (int i = 0; i < 4; ++i) key.ptrs[i] = ptrs[i];
    for (size_t i = 0; i < w->execs.size();) {
        if (w->execs[i]->key.allocs != key.allocs) {
            cudaGraphExecDestroy(w->execs[i]->exec);
            delete w->execs[i];
            w->execs.erase(w->execs.begin() + i);
        } else {
            ++i;
        }
    }
    for (SolveExec* e : w->execs)
        if (e->key == key) {
            gc = e->gc;
            return e->exec;
        }
    SolveExec* e = new SolveExec();
    e->key = key;
    try {
        e->exec = a.host_loop ? build_chunk_graph(w, s, y, a, x, e->gc) : build_solve_graph(w, s, y, a, x, e->gc);
    } catch (...) {
        delete e;
        throw;
    }
    if (w->execs.size() >= 6) {
        cudaGraphExecDestroy(w->execs.front()->exec);
        delete w->execs.front();
        w->execs.erase(w->execs.begin());
    }
    w->execs.push_back(e);
    gc = e->gc;
    return e->exec;
}

void solver_run(Solver* w, const Structure& s, const System& y, const SolveArgs& a, double* x, SolveOut& out,
                cudaStream_t st) {
    int n_dirs = a.mcg ? a.n_dirs : 1;
    if (n_dirs < 1) n_dirs = 1;
    if (n_dirs > kMaxDirs) throw Error(BA_ERR_INVALID_ARG, "n_dirs must be in [1, 16]");
    const bool fp32 = a.precision == BA_PRECISION_MIXED;
    prepare(w, s, a, n_dirs, fp32);
    const int nb = w->nb;
    w->launches = 0;
    w->host_hist.assign(nb, std::vector<double>());
    GraphCounts gc;
    cudaGraphExec_t exec = solve_graph(w, s, y, a, x, gc);

    // the solver's events, made once (on the device of the handle)
    if (!w->ev0) BA_CUDA_TRY(cudaEventCreate(&w->ev0));
    if (!w->ev1) BA_CUDA_TRY(cudaEventCreate(&w->ev1));
    const cudaEvent_t e0 = w->ev0, e1 = w->ev1;
    BA_CUDA_TRY(cudaEventRecord(e0, st));
    // the solve: its arguments in, one graph launch, the results out, one wait
    Params* hp = w->h_params;
    hp->tol = a.tol;
    hp->tau = a.tau;
    hp->inner_tol = a.inner_tol;
    hp->max_iters = a.max_iters;
    hp->max_refine = a.max_refine;
    hp->mcg = a.mcg;
    hp->pad = 0;
    BA_CUDA_TRY(cudaMemcpyAsync(w->params.p, hp, sizeof(Params), cudaMemcpyHostToDevice, st));
    BA_CUDA_TRY(cudaMemsetAsync(w->loops.p, 0, sizeof(Loops), st));
    int host_waits = 0;
    if (a.host_loop) run_host_loops(w, s, y, a, x, exec, gc, st, &host_waits);
    else BA_CUDA_TRY(cudaGraphLaunch(exec, st));
    BA_CUDA_TRY(cudaMemcpyAsync(w->h_ctl, w->ctl.p, sizeof(Ctl) * nb, cudaMemcpyDeviceToHost, st));
    if (fp32) BA_CUDA_TRY(cudaMemcpyAsync(w->h_outer, w->outer.p, sizeof(Outer) * nb, cudaMemcpyDeviceToHost, st));
    BA_CUDA_TRY(cudaMemcpyAsync(w->h_loops, w->loops.p, sizeof(Loops), cudaMemcpyDeviceToHost, st));
    BA_CUDA_TRY(cudaMemcpyAsync(w->h_hist, w->hist.p, sizeof(double) * size_t(nb) * w->mi1, cudaMemcpyDeviceToHost, st));
    BA_CUDA_TRY(cudaEventRecord(e1, st));
    BA_CUDA_TRY(cudaEventSynchronize(e1));
    ++host_waits;
    BA_CUDA_TRY(cudaGetLastError());
    float ms = 0.f;
    cudaEventElapsedTime(&ms, e0, e1);

    const Loops lp = *w->h_loops;
    if (!a.host_loop) w->launches = gc.pre + int64_t(lp.outer) * gc.sweep + int64_t(lp.inner) * gc.body + gc.post;
    out = SolveOut();
    out.probs.assign(nb, ProbOut());
    bool timed_out = false;
    for (int b = 0; b < nb; ++b) {
        ProbOut& o = out.probs[b];
        const Ctl& c = w->h_ctl[b];
        int steps = 0;
        if (!fp32) {
            o.status = c.done ? c.status : BA_ERR_NOT_CONVERGED;
            o.iters = c.it;
            o.local_steps = c.local_steps;
            o.pinv_steps = c.pinv_steps;
            o.history_cols = a.mcg ? c.cols : 1;
            o.rel_residual = c.rr0 > 0 ? std::sqrt(c.rr / c.rr0) : 0.0;
            o.refinements = 1;
            o.true_rel_residual = c.bb > 0 ? std::sqrt(c.true_rr / c.bb) : 0.0;
            steps = c.it;
        } else {
            const Outer& u = w->h_outer[b];
            o.status = u.status;
            o.iters = u.iters;
            o.local_steps = u.locals;
            o.pinv_steps = u.pinvs;
            o.history_cols = u.cols;
            o.refinements = u.sweeps;
            // tr is the float64 true residual of the problem's current x
            o.rel_residual = u.bb > 0 ? std::sqrt(u.tr / u.bb) : 0.0;
            o.true_rel_residual = o.rel_residual;
            steps = u.iters;
        }
        o.n_eff = w->lay[b].n_eff;
        timed_out = timed_out || o.status == BA_ERR_TIMEOUT;
        std::vector<double>& h = w->host_hist[b];
        h.resize(size_t(std::min(steps, w->mi1)));
        for (size_t i = 0; i < h.size(); ++i) h[i] = std::sqrt(w->h_hist[i * nb + b]);
    }
    if (timed_out) {
        clear_counters(w, st);
        BA_CUDA_TRY(cudaStreamSynchronize(st));
        ++host_waits;
    }
    out.launches = w->launches;
    out.host_waits = host_waits;
    out.ms = ms;
    // the batch's summary: the first failing problem's status, the largest counts and residuals
    out.status = BA_OK;
    out.n_eff = 1;
    for (int b = 0; b < nb; ++b) {
        const ProbOut& o = out.probs[b];
        if (out.status == BA_OK && o.status != BA_OK) out.status = o.status;
        out.iters = std::max(out.iters, o.iters);
        out.local_steps = std::max(out.local_steps, o.local_steps);
        out.pinv_steps = std::max(out.pinv_steps, o.pinv_steps);
        out.n_eff = std::max(out.n_eff, o.n_eff);
        out.refinements = std::max(out.refinements, o.refinements);
        out.history_cols = std::max(out.history_cols, o.history_cols);
        out.rel_residual = std::max(out.rel_residual, o.rel_residual);
        out.true_rel_residual = std::max(out.true_rel_residual, o.true_rel_residual);
    }
}

// Reads every 16 bytes of buf (n of them) and writes nothing unless they are all 0xff (never: the
// buffer is zeroed once): a read that the compiler cannot drop.
__global__ void k_l2_read(const uint4* __restrict__ buf, int64_t n, unsigned* sink) {
    const int64_t i0 = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    unsigned v = 0xffffffffu;
    for (int64_t i = i0; i < n; i += int64_t(gridDim.x) * blockDim.x) {
        const uint4 u = buf[i];
        v &= u.x & u.y & u.z & u.w;
    }
    if (i0 < n && v == 0xffffffffu) atomicAdd(sink, 1u);
}

// Evict L2 by reading a 256 MiB buffer (twice the cache).  A read leaves clean lines behind, so the
// timed kernel after it writes nothing back for earlier kernels (a written flush buffer would leave
// dirty lines whose write-back lands in the timed launch).
void flush_l2(cudaStream_t st) {
    static void* buf = nullptr;
    static unsigned* sink = nullptr;
    const size_t bytes = size_t(256) << 20;
    if (!buf) {
        BA_CUDA_TRY(cudaMalloc(&buf, bytes));
        BA_CUDA_TRY(cudaMalloc(&sink, sizeof(unsigned)));
        BA_CUDA_TRY(cudaMemset(buf, 0, bytes));
    }
    k_l2_read<<<num_sms() * 8, 256, 0, st>>>(static_cast<const uint4*>(buf), int64_t(bytes / 16), sink);
}

// a^T b as the float32 sweeps add it (for the tests): a chunk of `chunk` rows per warp as in k_mcg_phi, then the
// chunks as in k_mcg_beta.
__global__ void k_test_phi(const float* a, const float* b, int n, int chunk, WideSlot<float>* slots) {
    const int r0 = blockIdx.x * chunk;
    phi_columns<float, 1>(a, n, b, r0, min(r0 + chunk, n), slots + blockIdx.x, 1);
}
__global__ void k_test_phi_block(const WideSlot<float>* slots, int chunks, double* out) {
    phi_block<float>(slots, 0, 1, 1, chunks, 1, chunks, true, threadIdx.x, 32, out);
}

// a^T b as k_pcg_update and k_pcg_dir add it: a product per thread, kUpdThreads a CTA
__global__ void __launch_bounds__(kUpdThreads) k_test_update(const float* a, const float* b, int n,
                                                             WideSlot<float>* slots) {
    const int i = blockIdx.x * kUpdThreads + threadIdx.x;
    ExactSum<float> v[1];
    if (i < n) v[0].add(a[i], b[i]);
    cta_publish<float, 1>(v, slots);
}
// a^T b as k_one_cta adds it: 9 n9 values by one thread
__global__ void k_test_one_phi(const float* a, const float* b, int n9, double* out) {
    if (threadIdx.x == 0) *out = one_phi<1>(a, b, 0, 9 * n9);
}
__global__ void k_test_update_total(const WideSlot<float>* slots, int np, double* out) {
    const WideSum<float> s = total_of<float, 1>(slots, np, 0);
    if (threadIdx.x == 0) *out = s.value();
}

void test_float_sums(const float* a, const float* b, int n, int chunk, double* out) {
    const int chunks = (n + chunk - 1) / chunk;
    Buf ab, slots;
    grow(ab, sizeof(float) * 2 * size_t(n) + sizeof(double));
    const int ctas = (n + kUpdThreads - 1) / kUpdThreads, most = std::max(chunks, ctas);
    grow(slots, sizeof(WideSlot<float>) * size_t(most) + 3 * sizeof(double));
    float* da = ptr<float>(ab);
    double* d = reinterpret_cast<double*>(ptr<WideSlot<float>>(slots) + most);
    cudaError_t e = cudaMemcpy(da, a, sizeof(float) * n, cudaMemcpyDefault);
    if (e == cudaSuccess) e = cudaMemcpy(da + n, b, sizeof(float) * n, cudaMemcpyDefault);
    if (e == cudaSuccess) {
        k_test_phi<<<chunks, 32>>>(da, da + n, n, chunk, ptr<WideSlot<float>>(slots));
        k_test_phi_block<<<1, 32>>>(ptr<WideSlot<float>>(slots), chunks, d);
        k_test_update<<<ctas, kUpdThreads>>>(da, da + n, n, ptr<WideSlot<float>>(slots));
        k_test_update_total<<<1, 32>>>(ptr<WideSlot<float>>(slots), ctas, d + 1);
        k_test_one_phi<<<1, 32>>>(da, da + n, n / 9, d + 2);
        e = cudaMemcpy(out, d, 3 * sizeof(double), cudaMemcpyDefault);
    }
    free_buf(ab);
    free_buf(slots);
    BA_CUDA_TRY(e);
}

// The PCG product q = S p of every problem (k_spmv MODE 1, the kernel of Algorithm 1; in float32 the
// symmetric product, both of its launches), set up as at the start of a PCG solve (p = D^{-1} b~).
double solver_time_spmv(Solver* w, const Structure& s, const System& y, bool fp32, int reps, int item_blocks,
                        int spmv_cfg, cudaStream_t st) {
    SolveArgs a;
    a.mcg = 0;
    a.max_iters = 1;
    a.item_blocks = item_blocks;
    a.spmv_cfg = spmv_cfg;
    a.precision = fp32 ? BA_PRECISION_MIXED : BA_PRECISION_FP64;
    prepare(w, s, a, 1, fp32);
    Params* hp = w->h_params;
    *hp = Params();
    hp->tol = 1e-6;
    hp->max_iters = 1;
    BA_CUDA_TRY(cudaMemcpyAsync(w->params.p, hp, sizeof(Params), cudaMemcpyHostToDevice, st));
    if (fp32)
        krylov_init<float>(w, s, y.S32, y.S32u, y.Dhat, y.bt, -1.0, y.lam, ptr<float>(w->xw), nullptr, st, false);
    else
        krylov_init<double>(w, s, y.S, nullptr, y.Dinv, y.bt, -1.0, nullptr, ptr<double>(w->xw), nullptr, st, false);
    BA_CUDA_TRY(cudaGetLastError());
    cudaEvent_t e0, e1;
    BA_CUDA_TRY(cudaEventCreate(&e0));
    BA_CUDA_TRY(cudaEventCreate(&e1));
    double total = 0.0;
    for (int k = 0; k < reps; ++k) {
        flush_l2(st);
        BA_CUDA_TRY(cudaEventRecord(e0, st));
        if (fp32)
            enqueue_product<float, 1>(w, s, y.S32, y.S32u, ptr<float>(w->P), kSelLive, ptr<float>(w->Q),
                                      ptr<float>(w->r), st);
        else
            enqueue_product<double, 1>(w, s, y.S, nullptr, ptr<double>(w->P), kSelLive, ptr<double>(w->Q),
                                       ptr<double>(w->r), st);
        BA_CUDA_TRY(cudaEventRecord(e1, st));
        BA_CUDA_TRY(cudaEventSynchronize(e1));
        float ms = 0.f;
        BA_CUDA_TRY(cudaEventElapsedTime(&ms, e0, e1));
        total += ms;
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    return total / reps;
}

// Shape and item chunk chosen by timing the PCG product: every shape with every chunk of 32 .. 1024
// blocks per work item, `reps` launches each; ties keep the earlier candidate.  The lists are left
// built for the winner.
void solver_autotune(Solver* w, const Structure& s, const System& y, bool fp32, int reps, int* best_cfg,
                     int* best_cb, double* best_ms, cudaStream_t st) {
    const int cands[] = {32, 64, 128, 256, 512, 1024};
    int bcfg = 0, bcb = 0;
    double bms = 0.0;
    for (int cfg = 0; cfg < kSpmvShapes; ++cfg)
        for (int cb : cands) {
            if (cfg == 1 && !fp32) break;   // the same shape as 0
            const double ms = solver_time_spmv(w, s, y, fp32, reps, cb, cfg, st);
            if (bcb == 0 || ms < bms) {
                bcfg = cfg;
                bcb = cb;
                bms = ms;
            }
        }
    solver_time_spmv(w, s, y, fp32, 1, bcb, bcfg, st);
    *best_cfg = bcfg;
    *best_cb = bcb;
    *best_ms = bms;
}

}  // namespace ba
