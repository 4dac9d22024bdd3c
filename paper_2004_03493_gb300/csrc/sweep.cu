// Forward and reverse sweeps of Algorithm 1: pull-style sparse matrix-vector
// products over the device CSRs.
//
//   forward (Algorithm 1, forward loop):  pi^l(i) = sqrt(c) * sum_{j in Out(i)} x^{l-1}(j),
//           x^{l}(i) = pi^l(i) / din(i)            -- rows of the out-edge CSR
//   reverse (Algorithm 1, reverse loop; Eq. sL):
//           s^l(j) = sqrt(c) / din(j) * sum_{i in I(j)} s^{l-1}(i) + D^(j) pi^{L-l}(j) / a
//                                                   -- rows of the in-edge CSR
//
// (P pi)(i) = sum_j P(i,j) pi(j) with P(i,j) = 1/din(j) for i in I(j), so the
// forward product pulls along out-edges with the 1/din factor folded into the
// gathered vector x; (P^T s)(j) = (1/din(j)) sum_{i in I(j)} s(i) pulls along
// in-edges.  Both are atomic-free and deterministic: each row's sum is formed in
// a fixed order by one lane (short rows) or by fixed pieces, joined by one warp in a
// fixed order (long rows).
//
// Two arithmetic forms share the kernels through a value/accumulator policy:
//   FP64  -- the plain method: the history pi^l and the result s in FP64.  GB300's
//            scalar FP64 unit issues about 0.4 additions per SM per clock, so the
//            per-level arithmetic runs in two-float on the FP32 pipe: the gathered
//            vectors x^l and s^l are two-floats (float2, 8 bytes like a double), each
//            row sum is two-float, and the FP64 values are read and written through
//            integer conversions (f2conv.cuh).  Every stored value is within about
//            2^-46 relative of an FP64 computation of the same sums (the step and query
//            parity tests hold it to 1e-12 of the oracle).  The Lemma 5 sweeps of
//            Algorithm 3 take the same form; the sparse history keeps FP64 sums (Pol64);
//   FP32c -- the precision form: pi^l and x^l stored in FP32 with two-float
//            (compensated) row sums; s^l stored and summed as two-floats; FP64
//            only for the final s^L and the D^ ratio.  On GB300, whose FP64 issue
//            rate is a small fraction of FP32, this keeps the sweeps bound by
//            memory rather than by FP64 arithmetic.
#include "common.cuh"
#include "f2conv.cuh"
#include "internal.h"
#include "twofloat.cuh"

#include <type_traits>

namespace esim {

// ---------------------------------------------------------------- policies

struct Pol64 {  // FP64 values, FP64 sums
    using V = double;
    using A = double;
    static __device__ __forceinline__ A zero() { return 0.0; }
    static __device__ __forceinline__ A add(A a, V v) { return a + v; }
    static __device__ __forceinline__ A combine(A a, A b) { return a + b; }
    static __device__ __forceinline__ A shfl(A a, int o, int w) { return __shfl_down_sync(0xffffffffu, a, o, w); }
    static __device__ __forceinline__ A fresh(const A* p) { return __ldcg(p); }
};

struct Pol32c {  // FP32 values, two-float sums
    using V = float;
    using A = f2;
    static __device__ __forceinline__ A zero() { return f2{0.f, 0.f}; }
    static __device__ __forceinline__ A add(A a, V v) { return f2_add_f(a, v); }
    static __device__ __forceinline__ A combine(A a, A b) { return f2_add(a, b); }
    static __device__ __forceinline__ A shfl(A a, int o, int w) { return f2_shfl_down(a, o, w); }
    static __device__ __forceinline__ A fresh(const A* p) {  // past the L1: other SMs wrote it in this launch
        const float2 v = __ldcg(reinterpret_cast<const float2*>(p));
        return f2{v.x, v.y};
    }
};

struct Pol2f {  // two-float values (float2: hi, lo), two-float sums
    using V = float2;
    using A = f2;
    static __device__ __forceinline__ A zero() { return f2{0.f, 0.f}; }
    static __device__ __forceinline__ A add(A a, V v) { return f2_add(a, f2{v.x, v.y}); }
    static __device__ __forceinline__ A combine(A a, A b) { return f2_add(a, b); }
    static __device__ __forceinline__ A shfl(A a, int o, int w) { return f2_shfl_down(a, o, w); }
    static __device__ __forceinline__ A fresh(const A* p) {  // past the L1: other SMs wrote it in this launch
        const float2 v = __ldcg(reinterpret_cast<const float2*>(p));
        return f2{v.x, v.y};
    }
};

template <class Pol>
__device__ __forceinline__ typename Pol::A warp_combine(typename Pol::A v) {  // lane 0 has the result
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = Pol::combine(v, Pol::shfl(v, o, 32));
    return v;
}

// ---------------------------------------------------------------- row epilogues

struct ForwardOp {  // FP64
    double sc;
    const double* __restrict__ inv_din;
    const uint32_t* __restrict__ pos;
    double* __restrict__ pi_out;
    double* __restrict__ x_out;  // by position
    __device__ __forceinline__ void operator()(int64_t row, double acc) const {
        const double p = sc * acc;
        pi_out[row] = p;
        x_out[at_pos(pos, row)] = p * inv_din[row];
    }
};

struct ReverseSparseOp {  // FP64; the D^ pi^{L-l} / a term is scattered from the sparse history
    double sc;
    const double* __restrict__ inv_din;
    const uint32_t* __restrict__ pos;  // NULL for the last level, whose result is by node
    double* __restrict__ s_out;
    __device__ __forceinline__ void operator()(int64_t row, double acc) const {
        s_out[at_pos(pos, row)] = (sc * acc) * inv_din[row];
    }
};

struct ForwardOp32c {  // FP32 storage, two-float sum
    f2 sc;
    const uint32_t* __restrict__ in_rp;
    const uint32_t* __restrict__ pos;
    float* __restrict__ pi_out;
    float* __restrict__ x_out;  // by position
    __device__ __forceinline__ void operator()(int64_t row, f2 acc) const {
        const f2 p = f2_mul(acc, sc);
        const float pf = __fadd_rn(p.hi, p.lo);
        pi_out[row] = pf;
        const uint32_t d = in_rp[row + 1] - in_rp[row];
        x_out[at_pos(pos, row)] = d ? __fdiv_rn(pf, (float)d) : 0.f;
    }
};

// Reverse level in two-float: s^l = sqrt(c) (P^T s^{l-1}) + w pi^{L-l}, w = D^/a
// as a two-float; intermediate levels store float2, the last level FP64.
template <bool kFinal>
struct ReverseOp2f {
    f2 sc;
    const uint32_t* __restrict__ rp;
    const uint32_t* __restrict__ pos;
    const float2* w;
    const float* h;
    float2* __restrict__ s_out;  // by position
    double* __restrict__ s_final;
    __device__ __forceinline__ void operator()(int64_t row, f2 acc) const {
        const uint32_t d = rp[row + 1] - rp[row];
        f2 prop = f2{0.f, 0.f};
        if (d) prop = f2_div_f(f2_mul(acc, sc), (float)d);
        const float2 wv = w[row];
        const f2 s = f2_add(prop, f2_mul_f(f2{wv.x, wv.y}, h[row]));
        if (kFinal) s_final[row] = f2_to_double(s);
        else s_out[at_pos(pos, row)] = make_float2(s.hi, s.lo);
    }
};

// FP64 form, forward level: pi^l = sqrt(c) * row sum in two-float, stored as FP64;
// x^l = pi^l / din stored as a two-float for the next level's gathers.
struct ForwardOpD {
    f2 sc;
    const uint32_t* __restrict__ in_rp;
    const uint32_t* __restrict__ pos;
    double* __restrict__ pi_out;
    float2* __restrict__ x_out;  // by position
    __device__ __forceinline__ void operator()(int64_t row, f2 acc) const {
        const f2 p = f2_mul(acc, sc);
        pi_out[row] = f2_to_double_bits(p);
        const uint32_t d = in_rp[row + 1] - in_rp[row];
        const f2 x = d ? f2_div_f(p, (float)d) : f2{0.f, 0.f};
        x_out[at_pos(pos, row)] = make_float2(x.hi, x.lo);
    }
};

// FP64 form: D^(k) pi^{L-l}(k) / a in two-float from the FP64 values (exact quotient
// correction, so pi = a and D^ = 1 give 1 exactly)
__device__ __forceinline__ f2 diag_term(double dhat, double h, f2 a) {
    return f2_div(f2_mul(double_to_f2_bits(dhat), double_to_f2_bits(h)), a);
}

// FP64 form, reverse level: s^l = sqrt(c) (P^T s^{l-1}) + D^ pi^{L-l} / a in two-float,
// pi^{L-l} and D^ read in FP64; s^l stored as a two-float, the last level as FP64.
template <bool kFinal>
struct ReverseOpD {
    f2 sc;
    f2 a;
    const uint32_t* __restrict__ rp;
    const uint32_t* __restrict__ pos;
    const double* dhat;
    const double* h;
    float2* __restrict__ s_out;  // by position
    double* __restrict__ s_final;
    __device__ __forceinline__ void operator()(int64_t row, f2 acc) const {
        const uint32_t d = rp[row + 1] - rp[row];
        const f2 prop = d ? f2_div_f(f2_mul(acc, sc), (float)d) : f2{0.f, 0.f};
        const f2 s = f2_add(prop, diag_term(dhat[row], h[row], a));
        if (kFinal) s_final[row] = f2_to_double_bits(s);
        else s_out[at_pos(pos, row)] = make_float2(s.hi, s.lo);
    }
};

// ---------------------------------------------------------------- row kernel
//
// A sweep level is gather-bound: each entry reads one value x[col[p]] from a vector
// that sits in L2, and a random 4- or 8-byte gather costs a 32-byte sector whatever its
// width.  One warp takes one slice (32 rows of nearly equal length, one per lane; sell.cu):
// every lane adds its own row's entries one after another in two chains (even and odd
// ones), kU gathers in flight, the next kU column numbers loaded before the gathers
// are waited for.  No shared memory is used, so the L1 keeps the values of the nodes with
// many edges; an entry costs about 16 instructions instead of 54.
// Rows longer than row_cap (8 to 64, 64 from four million edges on: a lane's chain is most of
// a small level's time; capi.cu) are summed by a warp each, lanes side by side along the row,
// first in the grid; a row longer than 32 row_cap entries is cut into pieces, and the warp
// that counts in the last of them adds their sums.  Both joins are fixed shuffle trees.
// Every row's sum has a fixed order, so the sweeps are deterministic.
//
// n = 1e6, m = 1.75e7: 81 / 83 us a forward / reverse level in FP64 storage with eight gathers in
// flight (about a tenth less with four), against 128 / 137 on warp tiles staged in shared memory (54 instructions an entry, 9 % L1 hits); FP64 sums
// (sparse history) 98 against 316 on eight or sixteen lanes a row.  n = 1e5, m = 1e6: 11-12
// against 20-23.  What is left is the L2's rate of scattered sectors (tags 63 % busy, L1
// path 66 %).
// Gathers in flight per lane: eight where a level is one row's latency; four from four million edges on, where
// the warps, not the lanes, have to cover it (half the registers a lane, for two-floats seven
// blocks an SM).  n = 1e6, m = 1.75e7, L = 33, FP64 / FP32c sweeps: 4.60 / 4.08 ms with eight, 4.12 /
// 3.85 with four; the FP32c query at n = 1e5 415 us with eight, 447 with four.  Below the line, at a cap
// of 64 on both sides: random n = 100,000, m = 3.9e6 929 us with eight, 1092 with four.
template <class Pol, int kU>
constexpr int sell_min_blocks() {
    return kU == 4 && sizeof(typename Pol::V) == 8 && sizeof(typename Pol::A) == sizeof(f2) &&
                   !std::is_same<typename Pol::V, double>::value
               ? 7
               : 1;
}

template <class Pol, int kU, class Op>
__global__ void __launch_bounds__(kBlock, (sell_min_blocks<Pol, kU>())) sell_rows_kernel(const SellRows A, const uint32_t* __restrict__ rp,
                                                          const typename Pol::V* x, Op op,
                                                          typename Pol::A* __restrict__ partial,
                                                          unsigned* __restrict__ arrived) {
    using Acc = typename Pol::A;
    using V = typename Pol::V;
    const int lane = threadIdx.x & 31;
    const int64_t s = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    next_may_start();
    if (s >= A.nslices) return;
    const uint32_t o0 = __ldg(A.off + s), steps = __ldg(A.off + s + 1) - o0;
    const int2 r = __ldg(A.rows + s * 32 + lane);
    const uint32_t len = (uint32_t)r.y;
    const int32_t* __restrict__ c = A.col + (size_t)o0 * 32 + lane;
    int32_t j[kU];
#pragma unroll
    for (int u = 0; u < kU; ++u)
        if ((uint32_t)u < steps) j[u] = __ldg(c + u * 32);
    prior_done();  // until here only the graph is read; the level before wrote x
    Acc acc0 = Pol::zero(), acc1 = Pol::zero();
    for (uint32_t t = 0; t < steps; t += kU) {
        V g[kU];
#pragma unroll
        for (int u = 0; u < kU; ++u)
            if (t + u < len) g[u] = x[j[u]];
        c += kU * 32;
#pragma unroll
        for (int u = 0; u < kU; ++u)
            if (t + kU + u < steps) j[u] = __ldg(c + u * 32);
#pragma unroll
        for (int u = 0; u < kU; u += 2) {
            if (t + u < len) acc0 = Pol::add(acc0, g[u]);
            if (t + u + 1 < len) acc1 = Pol::add(acc1, g[u + 1]);
        }
    }
    const Acc acc = Pol::combine(acc0, acc1);
    if (s >= A.npieces) {
        if (r.x >= 0) op((int64_t)r.x, acc);
        return;
    }
    Acc sum = warp_combine<Pol>(acc);
    const uint32_t deg = __ldg(rp + r.x + 1) - __ldg(rp + r.x), piece = 32 * A.row_cap;
    if (deg > piece) {
        const uint32_t first = A.piece[s].first, count = (deg + piece - 1) / piece;
        unsigned last = 0;
        if (lane == 0) {
            partial[s] = sum;
            __threadfence();
            last = atomicInc(arrived + first, count - 1) == count - 1;  // wraps to 0 for the next sweep
            __threadfence();
        }
        if (!__shfl_sync(0xffffffffu, last, 0)) return;
        sum = Pol::zero();
        for (uint32_t i = (uint32_t)lane; i < count; i += 32) sum = Pol::combine(sum, Pol::fresh(partial + first + i));
        sum = warp_combine<Pol>(sum);
    }
    if (lane == 0) op((int64_t)r.x, sum);
}

// The same walk over the slices with 32-bit sets and OR: bit c of next(i) says that the walk
// distribution of candidate c reaches i one step later.  counts[c] gains the nodes with bit c:
// a warp's 32 sets are counted column by column with ballots.  One warp a row, which this
// replaces, left a hub's row to one warp: 29 us a level at n = 20,011 and 79 at n = 1e5, now
// 11.7 and 13.2 (serialised launches).
__global__ void __launch_bounds__(kBlock) reach_rows_kernel(const SellRows A, const uint32_t* __restrict__ rp,
                                                           const uint32_t* cur, uint32_t* __restrict__ next,
                                                           unsigned long long* __restrict__ counts,
                                                           unsigned long long* __restrict__ partial,
                                                           unsigned* __restrict__ arrived) {
    constexpr int kU = 8;
    __shared__ unsigned total[32];
    const int lane = threadIdx.x & 31;
    const int64_t s = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    next_may_start();
    if (threadIdx.x < 32) total[threadIdx.x] = 0u;
    __syncthreads();
    prior_done();
    if (s < A.nslices) {
        const uint32_t o0 = __ldg(A.off + s), steps = __ldg(A.off + s + 1) - o0;
        const int2 r = __ldg(A.rows + s * 32 + lane);
        const uint32_t len = (uint32_t)r.y;
        const int32_t* __restrict__ c = A.col + (size_t)o0 * 32 + lane;
        uint32_t set = 0u;
        for (uint32_t t = 0; t < steps; t += kU, c += kU * 32) {
            int32_t j[kU];
#pragma unroll
            for (int u = 0; u < kU; ++u)
                if (t + u < len) j[u] = __ldg(c + u * 32);
#pragma unroll
            for (int u = 0; u < kU; ++u)
                if (t + u < len) set |= cur[j[u]];
        }
        unsigned n = 0;  // lane c: the nodes of this warp with bit c
        if (s >= A.npieces) {
            if (r.x >= 0) next[at_pos(A.pos, r.x)] = set;
            if (__any_sync(0xffffffffu, set != 0u)) {
#pragma unroll
                for (int b = 0; b < 32; ++b) {
                    const unsigned m = __ballot_sync(0xffffffffu, set >> b & 1u);
                    if (lane == b) n = __popc(m);
                }
            }
        } else {
            uint32_t all = __reduce_or_sync(0xffffffffu, set);
            const uint32_t deg = __ldg(rp + r.x + 1) - __ldg(rp + r.x), piece = 32 * A.row_cap;
            bool done = true;
            if (deg > piece) {
                const uint32_t first = A.piece[s].first, count = (deg + piece - 1) / piece;
                unsigned last = 0;
                if (lane == 0) {
                    partial[s] = all;
                    __threadfence();
                    last = atomicInc(arrived + first, count - 1) == count - 1;  // wraps to 0 for the next sweep
                    __threadfence();
                }
                done = __shfl_sync(0xffffffffu, last, 0);
                if (done) {
                    uint32_t v = 0u;
                    for (uint32_t i = (uint32_t)lane; i < count; i += 32) v |= (uint32_t)__ldcg(partial + first + i);
                    all = __reduce_or_sync(0xffffffffu, v);
                }
            }
            if (done) {
                if (lane == 0) next[at_pos(A.pos, r.x)] = all;
                n = all >> lane & 1u;
            }
        }
        if (n) atomicAdd(&total[lane], n);
    }
    __syncthreads();
    if (threadIdx.x < 32 && total[threadIdx.x]) atomicAdd(counts + threadIdx.x, (unsigned long long)total[threadIdx.x]);
}

// ---------------------------------------------------------------- level 0

// A call's first launch: no count of arrivals is left from calls before it.
__device__ __forceinline__ void clear_counts(const CallCounts& c) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < c.n; i += (int64_t)gridDim.x * blockDim.x) c.p[i] = 0u;
}

__global__ void forward_init_kernel(int64_t n, const CallCounts counts, int64_t u, const uint32_t* __restrict__ pos, double a, const double* __restrict__ inv_din,
                                    double* __restrict__ pi0, double* __restrict__ x0) {
    clear_counts(counts);
    const int64_t pu = at_pos(pos, u);
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        pi0[i] = i == u ? a : 0.0;
        x0[i] = i == pu ? a * inv_din[u] : 0.0;
    }
}

// FP64 form, level 0: pi^0 = a e_u (FP64), x^0 = a / din(u) e_u as a two-float.
__global__ void forward_init_d_kernel(int64_t n, const CallCounts counts, int64_t u, const uint32_t* __restrict__ pos, double a,
                                      float xhi, float xlo,
                                      double* __restrict__ pi0, float2* __restrict__ x0) {
    prior_done();
    clear_counts(counts);
    const int64_t pu = at_pos(pos, u);
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        pi0[i] = i == u ? a : 0.0;
        x0[i] = i == pu ? make_float2(xhi, xlo) : make_float2(0.f, 0.f);
    }
}

// FP64 form: s^0 = D^ pi^L / a as a two-float (in FP64 when L = 0).
__global__ void reverse_init_d_kernel(int64_t n, const CallCounts counts, const uint32_t* __restrict__ pos, float a_hi, float a_lo,
                                      const double* dhat,
                                      const double* h, float2* __restrict__ s0,
                                      double* __restrict__ s_final) {
    prior_done();
    clear_counts(counts);
    const f2 a{a_hi, a_lo};
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const f2 s = diag_term(dhat[i], h[i], a);
        if (s_final) s_final[i] = f2_to_double_bits(s);
        else s0[at_pos(pos, i)] = make_float2(s.hi, s.lo);
    }
}

__global__ void forward_init32_kernel(int64_t n, const CallCounts counts, int64_t u, const uint32_t* __restrict__ pos, float a, float xv,
                                      float* __restrict__ pi0, float* __restrict__ x0) {
    prior_done();
    clear_counts(counts);
    const int64_t pu = at_pos(pos, u);
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        pi0[i] = i == u ? a : 0.f;
        x0[i] = i == pu ? xv : 0.f;
    }
}

// w = D^ / a as two-floats, and s^0 = w pi^L (float2, or FP64 when L = 0)
__global__ void reverse_init2f_kernel(int64_t n, const CallCounts counts, const uint32_t* __restrict__ pos, double inv_a,
                                      const double* dhat,
                                      const float* h, float2* __restrict__ w, float2* __restrict__ s0,
                                      double* __restrict__ s_final) {
    prior_done();
    clear_counts(counts);
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const f2 wv = f2_from_double(dhat[i] * inv_a);
        w[i] = make_float2(wv.hi, wv.lo);
        const f2 s = f2_mul_f(wv, h[i]);
        if (s_final) s_final[i] = f2_to_double(s);
        else s0[at_pos(pos, i)] = make_float2(s.hi, s.lo);
    }
}

// ---------------------------------------------------------------- launchers

namespace {

// Sparse linearization (Section 3.2): after forward level l, pi_run += pi^l (level
// order, as the dense sum) and the entries pi^l(k) > theta are appended to the
// sparse history as (k, pi^l(k)).  Warps take their slots with one atomic each; the
// order of entries within a level therefore varies, but each node appears at most
// once per level, so the reverse scatter gives the same values whatever the order.
// The last block to finish records the level's end (a ticket, no waiting).
__global__ void __launch_bounds__(kBlock) compact_level_kernel(int64_t n, const double* __restrict__ lev,
                                                               double* __restrict__ pi_run, int first, double theta,
                                                               SparseHist h, int level, Status* __restrict__ st) {
    const int lane = threadIdx.x & 31;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t base = (int64_t)blockIdx.x * blockDim.x; base < n; base += stride) {  // uniform per block
        const int64_t i = base + threadIdx.x;
        double v = 0.0;
        bool keep = false;
        if (i < n) {
            v = lev[i];
            pi_run[i] = first ? v : pi_run[i] + v;
            keep = v > theta;
        }
        const unsigned mask = __ballot_sync(0xffffffffu, keep);
        if (mask) {
            unsigned long long pos0 = 0ull;
            if (lane == 0) pos0 = atomicAdd(&st->hist_count, (unsigned long long)__popc(mask));
            pos0 = __shfl_sync(0xffffffffu, pos0, 0);
            if (keep) {
                const unsigned long long pos = pos0 + (unsigned long long)__popc(mask & ((1u << lane) - 1u));
                if (pos < h.cap) {
                    h.idx[pos] = (int32_t)i;
                    h.val[pos] = v;
                } else if (h.cap) {
                    atomicOr(&st->err, kErrCapacity);
                }  // cap = 0: counting pass
            }
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        const unsigned t = atomicAdd(&st->ticket, 1u);
        if (t == gridDim.x - 1) {
            const unsigned long long end = atomicAdd(&st->hist_count, 0ull);
            if (h.lvl) h.lvl[level + 1] = end < h.cap ? end : h.cap;
            st->ticket = 0u;
        }
    }
}

// s(k) += D^(k) pi^level(k) / a (times the host's 1/a) over the sparse entries of one
// level (unique nodes).
__global__ void __launch_bounds__(kBlock) scatter_level_kernel(const uint64_t* __restrict__ lvl, int level,
                                                               const int32_t* __restrict__ idx,
                                                               const double* __restrict__ val,
                                                               const double* __restrict__ dhat,
                                                               const uint32_t* __restrict__ pos, double inv_a,
                                                               double* __restrict__ s) {
    const uint64_t beg = lvl[level], end = lvl[level + 1];
    for (uint64_t p = beg + (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; p < end;
         p += (uint64_t)gridDim.x * blockDim.x) {
        const int32_t k = idx[p];
        const int64_t q = at_pos(pos, k);
        s[q] = s[q] + dhat[k] * val[p] * inv_a;
    }
}

int elementwise_blocks(const Graph& g, int64_t n) {
    int64_t b = (n + kBlock - 1) / kBlock;
    int64_t cap = (int64_t)g.sm_count * 8;
    if (b > cap) b = cap;
    return (int)(b < 1 ? 1 : b);
}

// The first launch of a call, over all nodes: kernel(n, counts, args...)
template <class... Params, class... Args>
cudaError_t each_node(const Graph& g, void (*kernel)(int64_t, CallCounts, Params...), Args&&... args) {
    return launch_after(g.stream, dim3((unsigned)elementwise_blocks(g, g.n)), kBlock, 0, kernel, g.n, call_counts(g),
                        args...);
}

template <class Pol, class Op>
cudaError_t sweep_level(const Graph& g, const DevCsr& A, const typename Pol::V* x, const Op& op) {
    using Acc = typename Pol::A;
    static_assert(sizeof(Acc) == 8, "piece sums are 8 bytes");
    Acc* partial = reinterpret_cast<Acc*>(g.partial);
    unsigned* arrived = call_counts(g).p;
    const int64_t blocks = (A.sell.nslices * 32 + kBlock - 1) / kBlock;
    auto* kernel = A.sell.few_in_flight ? sell_rows_kernel<Pol, 4, Op> : sell_rows_kernel<Pol, 8, Op>;
    return launch_after(g.stream, dim3((unsigned)blocks), kBlock, 0, kernel, A.sell, A.rp, x, op, partial, arrived);
}

f2 host_f2(double v) {
    const float h = (float)v;
    return f2{h, (float)(v - (double)h)};
}

}  // namespace

cudaError_t launch_forward(const Graph& g, int64_t u, double c, int32_t L, double* hist, double* xa, double* xb) {
    const double sc = sqrt(c);
    const double a = 1.0 - sc;
    const uint32_t din_u = (*g.din_host)[(size_t)u];
    const f2 x0 = din_u ? host_f2(a / (double)din_u) : f2{0.f, 0.f};
    float2* x[2] = {reinterpret_cast<float2*>(xa), reinterpret_cast<float2*>(xb)};
    cudaError_t e = each_node(g, forward_init_d_kernel, u, g.out.sell.pos, a, x0.hi, x0.lo, hist, x[0]);
    if (e != cudaSuccess) return e;
    const f2 sc2 = host_f2(sc);
    for (int32_t l = 1; l <= L; ++l) {
        ForwardOpD op{sc2, g.in.rp, g.out.sell.pos, hist + (size_t)l * (size_t)g.n, x[l & 1]};
        e = sweep_level<Pol2f>(g, g.out, x[(l - 1) & 1], op);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// Two-float vectors: s^l in sa and (as scratch) in s_out, alternating so that level L-1
// lands in sa and the last level reads sa and writes s_out in FP64.
cudaError_t launch_reverse(const Graph& g, const double* hist, int32_t L, double c, const double* dhat, double* s_out,
                           double* sa, double* /*sb*/) {
    const double sc = sqrt(c);
    const double a = 1.0 - sc;
    float2* A = reinterpret_cast<float2*>(sa);
    float2* S = reinterpret_cast<float2*>(s_out);
    auto buf = [&](int32_t l) { return ((L - 1 - l) & 1) == 0 ? A : S; };
    const f2 a2 = host_f2(a);
    cudaError_t e = each_node(g, reverse_init_d_kernel, g.in.sell.pos, a2.hi, a2.lo, dhat, hist + (size_t)L * g.n,
                              L > 0 ? buf(0) : nullptr, L == 0 ? s_out : nullptr);
    if (e != cudaSuccess) return e;
    const f2 sc2 = host_f2(sc);
    for (int32_t l = 1; l <= L; ++l) {
        const float2* sp = buf(l - 1);
        const double* h = hist + (size_t)(L - l) * g.n;
        if (l < L) {
            ReverseOpD<false> op{sc2, a2, g.in.rp, g.in.sell.pos, dhat, h, buf(l), nullptr};
            e = sweep_level<Pol2f>(g, g.in, sp, op);
        } else {
            ReverseOpD<true> op{sc2, a2, g.in.rp, g.in.sell.pos, dhat, h, nullptr, s_out};
            e = sweep_level<Pol2f>(g, g.in, sp, op);
        }
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// Forward sweeps with the sparse history: dense rolling vectors (lev = pi^l, x^l),
// pi = sum_l pi^l accumulated in level order, and only pi^l(k) > theta kept.  With
// h.cap = 0 and h.lvl = NULL the entries are only counted (into Status::hist_count).
cudaError_t launch_forward_sparse(const Graph& g, int64_t u, double c, int32_t L, double theta, const SparseHist& h,
                                  double* lev, double* pi_run, double* xa, double* xb) {
    const double sc = sqrt(c);
    const double a = 1.0 - sc;
    cudaError_t e = cudaSuccess;
    if (h.lvl && (e = cudaMemsetAsync(h.lvl, 0, sizeof(uint64_t) * (size_t)(L + 2), g.stream)) != cudaSuccess)
        return e;
    const int eb = elementwise_blocks(g, g.n);
    forward_init_kernel<<<eb, kBlock, 0, g.stream>>>(g.n, call_counts(g), u, g.out.sell.pos, a, g.inv_din, lev, xa);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    compact_level_kernel<<<eb, kBlock, 0, g.stream>>>(g.n, lev, pi_run, 1, theta, h, 0, g.status);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    double* x[2] = {xa, xb};
    for (int32_t l = 1; l <= L; ++l) {
        ForwardOp op{sc, g.inv_din, g.out.sell.pos, lev, x[l & 1]};
        if ((e = sweep_level<Pol64>(g, g.out, x[(l - 1) & 1], op)) != cudaSuccess) return e;
        compact_level_kernel<<<eb, kBlock, 0, g.stream>>>(g.n, lev, pi_run, 0, theta, h, l, g.status);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// Reverse sweeps with the sparse history: s^l = sqrt(c) P^T s^{l-1}, then the kept
// entries of pi^{L-l} add D^ pi^{L-l} / a.
cudaError_t launch_reverse_sparse(const Graph& g, const SparseHist& h, int32_t L, double c, const double* dhat,
                                  double* s_out, double* sa) {
    const double sc = sqrt(c);
    const double a = 1.0 - sc;
    double* buf[2] = {s_out, sa};
    const unsigned sb = (unsigned)g.sm_count * 4;
    cudaError_t e = launch_fill(g, g.n, 0.0, buf[L & 1]);
    if (e != cudaSuccess) return e;
    scatter_level_kernel<<<sb, kBlock, 0, g.stream>>>(h.lvl, L, h.idx, h.val, dhat, L > 0 ? g.in.sell.pos : nullptr, 1.0 / a,
                                                 buf[L & 1]);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    for (int32_t l = 1; l <= L; ++l) {
        double* sn = buf[(L - l) & 1];
        const uint32_t* pos = l < L ? g.in.sell.pos : nullptr;  // the last level's result is by node
        ReverseSparseOp op{sc, g.inv_din, pos, sn};
        if ((e = sweep_level<Pol64>(g, g.in, buf[(L - l + 1) & 1], op)) != cudaSuccess) return e;
        scatter_level_kernel<<<sb, kBlock, 0, g.stream>>>(h.lvl, L - l, h.idx, h.val, dhat, pos, 1.0 / a, sn);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// Algorithm 3 helpers: h_l = (P^T)^l(u, .), the distribution of a non-stop walk from
// u (no decay, no stop), for l = 0..steps, into H[(steps+1) * n] (FP64 storage), in the
// FP64 form's two-float arithmetic (x_l = h_l / din as two-floats in xa/xb, n 8-byte
// entries each).
cudaError_t launch_walk_distributions(const Graph& g, int64_t u, int steps, double* H, double* xa, double* xb) {
    const uint32_t din_u = (*g.din_host)[(size_t)u];
    const f2 x0 = din_u ? host_f2(1.0 / (double)din_u) : f2{0.f, 0.f};
    float2* x[2] = {reinterpret_cast<float2*>(xa), reinterpret_cast<float2*>(xb)};
    cudaError_t e = each_node(g, forward_init_d_kernel, u, g.out.sell.pos, 1.0, x0.hi, x0.lo, H, x[0]);
    if (e != cudaSuccess) return e;
    const f2 one{1.f, 0.f};
    for (int l = 1; l <= steps; ++l) {
        ForwardOpD op{one, g.in.rp, g.out.sell.pos, H + (size_t)l * (size_t)g.n, x[l & 1]};
        e = sweep_level<Pol2f>(g, g.out, x[(l - 1) & 1], op);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

struct PlainOpD {
    double* __restrict__ out;
    __device__ __forceinline__ void operator()(int64_t row, f2 acc) const { out[row] = f2_to_double_bits(acc); }
};

// out(i) = sum_{j in Out(i)} x(j): the pull product over out-edges without weights, x by
// position (g.out.sell.pos) as two-floats, the sums in two-float, out in FP64.
cudaError_t launch_pull_sum(const Graph& g, const float2* x, double* out) {
    return sweep_level<Pol2f>(g, g.out, x, PlainOpD{out});
}

cudaError_t launch_reach(const Graph& g, const uint32_t* cur, uint32_t* next, unsigned long long* counts) {
    unsigned long long* partial = reinterpret_cast<unsigned long long*>(g.partial);
    unsigned* arrived = call_counts(g).p;
    const int64_t blocks = (g.out.sell.nslices * 32 + kBlock - 1) / kBlock;
    return launch_after(g.stream, dim3((unsigned)blocks), kBlock, 0, reach_rows_kernel, g.out.sell, g.out.rp, cur, next,
                        counts, partial, arrived);
}

cudaError_t launch_forward32(const Graph& g, int64_t u, double c, int32_t L, float* hist, float* xa, float* xb) {
    const double sc = sqrt(c);
    const float a = (float)(1.0 - sc);
    const uint32_t din_u = (*g.din_host)[(size_t)u];
    cudaError_t e = each_node(g, forward_init32_kernel, u, g.out.sell.pos, a, din_u ? a / (float)din_u : 0.f, hist, xa);
    if (e != cudaSuccess) return e;
    float* x[2] = {xa, xb};
    const f2 sc2 = host_f2(sc);
    for (int32_t l = 1; l <= L; ++l) {
        ForwardOp32c op{sc2, g.in.rp, g.out.sell.pos, hist + (size_t)l * (size_t)g.n, x[l & 1]};
        e = sweep_level<Pol32c>(g, g.out, x[(l - 1) & 1], op);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t launch_reverse32(const Graph& g, const float* hist, int32_t L, double c, const double* dhat,
                             double* s_out, float2* w, float2* sa, float2* sb) {
    const double sc = sqrt(c);
    const double a = 1.0 - sc;
    float2* buf[2] = {sa, sb};
    cudaError_t e = each_node(g, reverse_init2f_kernel, g.in.sell.pos, 1.0 / a, dhat, hist + (size_t)L * g.n, w,
                              buf[0], L == 0 ? s_out : nullptr);
    if (e != cudaSuccess) return e;
    const f2 sc2 = host_f2(sc);
    for (int32_t l = 1; l <= L; ++l) {
        const float2* sp = buf[(l - 1) & 1];
        const float* h = hist + (size_t)(L - l) * g.n;
        if (l < L) {
            ReverseOp2f<false> op{sc2, g.in.rp, g.in.sell.pos, w, h, buf[l & 1], nullptr};
            e = sweep_level<Pol2f>(g, g.in, sp, op);
        } else {
            ReverseOp2f<true> op{sc2, g.in.rp, g.in.sell.pos, w, h, nullptr, s_out};
            e = sweep_level<Pol2f>(g, g.in, sp, op);
        }
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace esim
