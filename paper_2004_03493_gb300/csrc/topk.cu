// Top-k selection (Sec. 1: the k nodes with the highest similarity to the source).
//
// Each candidate node i gets a 96-bit key (ordered(score) << 32 | ~i): a larger
// key is a higher score, and among equal scores a smaller id.  Keys are unique,
// so the top-k set is unique.
//
// Two launches read the scores once each.  The first deals the nodes to slices (a few
// thousand in all, Deal below) and keeps each slice's largest key; its last block to finish finds
// the k-th largest of those by a radix select over 8-bit digits.  The slices' maxima are k
// different keys, so the k-th largest of all keys is no smaller: that is a bound below which
// nothing is selected.  The second launch collects the keys at or above the bound, little more
// than k of them, and its last block sorts them.  If they are more than its list holds (large
// scores in places chosen against the dealing), that block selects over all scores by radix itself.
//
// What bounds it: two passes over n scores (8 MB at n = 2^20: 1.2 us each at the HBM rate)
// and about five dependent small steps.  Histogram and select launches for every digit of
// the key, most of them with nothing left to do, took 142 us there for k = 100; this takes
// 26.
#include "common.cuh"
#include "internal.h"
#include "exactsim.h"
#include <cuda.h>

#include <algorithm>
#include <mutex>
#include <string>

namespace esim {

namespace {

constexpr int kTopkThreads = 1024;
constexpr int kMaxSlices = 16384;   // maxima per column
constexpr int kCandMax = 8192;      // collected keys per column, at most

struct TopkState {
    unsigned long long bound_hi;
    unsigned int bound_lo;
    unsigned int count;       // keys collected
};

struct Cand {
    unsigned long long hi;
    unsigned int lo;
    unsigned int pad;
};

__device__ __forceinline__ unsigned long long ordered_bits(double s) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(s);
    return (b >> 63) ? ~b : (b ^ 0x8000000000000000ull);
}

__device__ __forceinline__ double from_ordered(unsigned long long o) {
    const unsigned long long b = (o >> 63) ? (o ^ 0x8000000000000000ull) : ~o;
    return __longlong_as_double((long long)b);
}

__device__ __forceinline__ unsigned digit_of(unsigned long long hi, unsigned lo, int d) {
    return d < 8 ? (unsigned)((hi >> (56 - 8 * d)) & 0xFFu) : (unsigned)((lo >> (24 - 8 * (d - 8))) & 0xFFu);
}

// The prefix of a radix select over the keys' 8-bit digits, most significant first.
struct Prefix {
    unsigned long long hi;
    unsigned int lo;
    unsigned int k_rem;   // keys still to select within the prefix
    int done;
    int depth;            // digits fixed
};

// Whether the top `depth` digits of the key are the prefix's (-1, 0, +1).
__device__ __forceinline__ int cmp_prefix(unsigned long long hi, unsigned lo, const Prefix& s, int depth) {
    if (depth == 0) return 0;
    if (depth <= 8) {
        const int sh = 64 - 8 * depth;
        const unsigned long long a = hi >> sh, b = s.hi >> sh;
        return a < b ? -1 : (a > b ? 1 : 0);
    }
    if (hi != s.hi) return hi < s.hi ? -1 : 1;
    const int sh = 32 - 8 * (depth - 8);
    const unsigned a = lo >> sh, b = s.lo >> sh;
    return a < b ? -1 : (a > b ? 1 : 0);
}

// How nodes are dealt to slices.  Scores have order: ids of neighbours, communities or a crawl lie
// together, and all zeros tie in id order.  A slice of neighbouring ids would hold many of the k
// best keys, and the bound would let k times its length through (n = 2^20, k = 50: sorted
// scores took 1255 us, 37 non-zero ones 4612, with slices of 128 neighbours; 29 and 44 now, scores in
// random order 31).  So groups of 32
// ids, one coalesced load, are spread over the warps by a multiplication modulo their number, with
// a factor near the golden ratio of it: group q is dealt to place q * A mod groups, and a
// run of groups, or every s-th one, falls evenly over the places.  Within its group a lane takes
// an id rotated by a hash of q, so that one column of a grid of ids does not stay in one lane.
// A slice is G of the 32 warps of a block, one lane each: the ids of a group are in 32 slices.
struct Deal {
    uint32_t groups;   // ceil(n / 32)
    uint32_t back;     // 1 / A modulo groups: the group at place p is p * back mod groups
    uint64_t magic;    // floor((2^64 - 1) / groups)
    // x mod groups, x < 2^58: the quotient's estimate is at most one too small
    __device__ __forceinline__ uint32_t mod(uint64_t x) const {
        const uint64_t r = x - __umul64hi(x, magic) * groups;
        return (uint32_t)(r >= groups ? r - groups : r);
    }
};

Deal make_deal(int64_t n) {
    const int64_t m = (n + 31) / 32;
    for (int64_t A = (int64_t)((double)m * 0.6180339887498949) + 1;; ++A) {  // the next one with an inverse
        int64_t r0 = m, r1 = A % m, t0 = 0, t1 = 1;  // r = t A modulo m
        while (r1) {
            const int64_t q = r0 / r1, r2 = r0 - q * r1, t2 = t0 - q * t1;
            r0 = r1, r1 = r2, t0 = t1, t1 = t2;
        }
        if (r0 == 1) return Deal{(uint32_t)m, (uint32_t)(t0 < 0 ? t0 + m : t0), ~0ull / (uint64_t)m};
    }
}

// One block: fixes digits of `pre` until the keys of the prefix bucket are exactly those
// still needed, or until at most `slack` more than k keys lie at or above the prefix.
// key(i, hi, lo) gives key i < count, false where there is none.  Fewer than k keys in
// all: the prefix stays empty (depth 0), which every key reaches.  kRegs > 0: count is at most
// kRegs per thread, and the keys are read once, into registers.
template <int kRegs, class Key>
__device__ void radix_select(int64_t count, unsigned k, unsigned slack, Prefix& pre, unsigned* hist, const Key& key) {
    const int lane = threadIdx.x & 31;
    if (threadIdx.x == 0) pre = Prefix{0ull, 0u, k, 0, 0};
    unsigned long long rh[kRegs ? kRegs : 1];
    unsigned rl[kRegs ? kRegs : 1];
    bool there[kRegs ? kRegs : 1];
    if constexpr (kRegs > 0) {
#pragma unroll
        for (int u = 0; u < kRegs; ++u) {
            const int64_t i = threadIdx.x + (int64_t)u * blockDim.x;
            there[u] = i < count && key(i, rh[u], rl[u]);
        }
    }
    for (int d = 0; d < 12; ++d) {
        for (int b = threadIdx.x; b < 256; b += blockDim.x) hist[b] = 0;
        __syncthreads();
        const Prefix s = pre;
        if (s.done) break;
        auto count_key = [&](bool is, unsigned long long hi, unsigned lo) {  // every lane takes part
            const unsigned dig = is && cmp_prefix(hi, lo, s, d) == 0 ? digit_of(hi, lo, d) : 256u;
            const unsigned peers = __match_any_sync(0xffffffffu, dig);
            if (dig < 256u && lane == __ffs(peers) - 1) atomicAdd(&hist[dig], (unsigned)__popc(peers));
        };
        if constexpr (kRegs > 0) {
#pragma unroll
            for (int u = 0; u < kRegs; ++u)
                if (u * (int64_t)blockDim.x < count) count_key(there[u], rh[u], rl[u]);  // uniform
        } else {
            constexpr int kU = 8;  // keys in flight
            for (int64_t base = threadIdx.x & ~31; base < count; base += kU * (int64_t)blockDim.x) {  // warp-uniform
                unsigned long long hi[kU];
                unsigned lo[kU];
                bool is[kU];
#pragma unroll
                for (int u = 0; u < kU; ++u) {
                    const int64_t i = base + lane + u * (int64_t)blockDim.x;
                    is[u] = i < count && key(i, hi[u], lo[u]);
                }
#pragma unroll
                for (int u = 0; u < kU; ++u) count_key(is[u], hi[u], lo[u]);
            }
        }
        __syncthreads();
        if (threadIdx.x < 32) {  // lane l: bins 255 - 8l down to 248 - 8l
            unsigned mine = 0;
            for (int j = 0; j < 8; ++j) mine += hist[255 - 8 * lane - j];
            unsigned incl = mine;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned v = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += v;
            }
            const unsigned total = __shfl_sync(0xffffffffu, incl, 31);
            if (d == 0 && total <= s.k_rem) {
                if (lane == 0) pre.done = 1;
            } else if (incl >= s.k_rem && incl - mine < s.k_rem) {  // exactly one lane
                unsigned cum = incl - mine;
                int B = 255 - 8 * lane;
                while (cum + hist[B] < s.k_rem) cum += hist[B--];
                if (d < 8) pre.hi |= (unsigned long long)B << (56 - 8 * d);
                else pre.lo |= (unsigned)B << (24 - 8 * (d - 8));
                pre.k_rem = s.k_rem - cum;
                pre.depth = d + 1;
                pre.done = hist[B] <= pre.k_rem + slack;
            }
        }
        __syncthreads();
    }
    __syncthreads();
}

// Whether this block is the last of the column to get here (all threads call it); what the
// other blocks wrote before is then visible.
__device__ __forceinline__ bool last_block(unsigned* ticket) {
    __shared__ bool last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicInc(ticket, gridDim.x - 1) == gridDim.x - 1;
    __syncthreads();
    if (last) __threadfence();
    return last;
}

// Launch 1: the largest key of every slice; the last block's bound.  One column per blockIdx.y
// in both launches.
__global__ void __launch_bounds__(kTopkThreads) topk_bound_kernel(int64_t n, const Deal deal, const double* scores,
                                                                  int64_t exclude, TopkState* __restrict__ st,
                                                                  unsigned* __restrict__ tickets,
                                                                  unsigned long long* __restrict__ max_hi,
                                                                  unsigned* __restrict__ max_lo, int G, unsigned k,
                                                                  int64_t col_stride, const int64_t* excl) {
    __shared__ unsigned hist[256];
    __shared__ Prefix pre;
    scores += (int64_t)blockIdx.y * col_stride;
    st += blockIdx.y;
    max_hi += (size_t)blockIdx.y * kMaxSlices;
    max_lo += (size_t)blockIdx.y * kMaxSlices;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    unsigned long long hi = 0;
    unsigned lo = 0;  // 0: no element yet (~i is never 0)
    auto larger = [&](unsigned long long h, unsigned l) {
        if (h > hi || (h == hi && l > lo)) {
            hi = h;
            lo = l;
        }
    };
    prior_done();
    if (excl) exclude = excl[blockIdx.y];
    // places of this warp: its number, then every number of warps further
    const unsigned long long warps = (unsigned long long)gridDim.x * (kTopkThreads / 32);
    unsigned long long place = (unsigned long long)blockIdx.x * (kTopkThreads / 32) + wid;
    uint32_t q = deal.mod(place * deal.back);
    auto node = [&]() {
        const int64_t i = 32 * (int64_t)q + ((lane + (q * 0x9E3779B9u >> 27)) & 31);
        return i < n && i != exclude ? i : (int64_t)-1;
    };
    if (warps >= deal.groups) {  // one group a warp at most
        const int64_t i = place < deal.groups ? node() : -1;
        if (i >= 0) larger(ordered_bits(scores[i]), ~(unsigned)i);
    } else {
        const uint32_t step = deal.mod(warps * deal.back);
        constexpr int kU = 8;  // loads in flight
        for (; place < deal.groups; place += kU * warps) {
            double v[kU];
            int64_t id[kU];
#pragma unroll
            for (int u = 0; u < kU; ++u) {
                id[u] = place + u * warps < deal.groups ? node() : -1;
                if (id[u] >= 0) v[u] = scores[id[u]];
                q = q >= deal.groups - step ? q - (deal.groups - step) : q + step;
            }
#pragma unroll
            for (int u = 0; u < kU; ++u)
                if (id[u] >= 0) larger(ordered_bits(v[u]), ~(unsigned)id[u]);
        }
    }
    if (G > 1) {  // the maxima of 32 warps' same lane side by side, then of G of them
        __shared__ unsigned long long wh[32][33];
        __shared__ unsigned wl[32][33];
        wh[wid][lane] = hi;
        wl[wid][lane] = lo;
        __syncthreads();
        hi = wh[lane][wid];
        lo = wl[lane][wid];
        for (int o = 1; o < G; o <<= 1) {
            const unsigned long long h = __shfl_xor_sync(0xffffffffu, hi, o);
            larger(h, __shfl_xor_sync(0xffffffffu, lo, o));
        }
    }
    const int64_t tid = (int64_t)blockIdx.x * kTopkThreads + threadIdx.x;
    if ((threadIdx.x & (G - 1)) == 0) {
        max_hi[tid / G] = hi;
        max_lo[tid / G] = lo;
    }
    if (!last_block(tickets + 2 * blockIdx.y)) return;
    auto key = [&](int64_t i, unsigned long long& h, unsigned& l) {
        h = __ldcg(max_hi + i);
        l = __ldcg(max_lo + i);
        return l != 0u;
    };
    const int64_t slices = (int64_t)gridDim.x * kTopkThreads / G;
    if (slices <= 5 * kTopkThreads) radix_select<5>(slices, k, k / 8 + 32, pre, hist, key);
    else radix_select<0>(slices, k, k / 8 + 32, pre, hist, key);
    if (threadIdx.x == 0) {
        st->bound_hi = pre.hi;
        st->bound_lo = pre.lo;
        st->count = 0u;
    }
}

// Launch 2: the keys at or above the bound into cand (cap of them at most); the last block
// sorts them, descending, and writes the first k.  P, a power of two >= cap, keys fit its
// dynamic shared memory.
__global__ void __launch_bounds__(kTopkThreads) topk_pick_kernel(int64_t n, const double* scores,
                                                                 int64_t exclude, TopkState* __restrict__ st,
                                                                 unsigned* __restrict__ tickets,
                                                                 Cand* __restrict__ cand, unsigned cap, int k, int P,
                                                                 int64_t col_stride, const int64_t* excl,
                                                                 int32_t* __restrict__ ids_out,
                                                                 double* __restrict__ vals_out) {
    extern __shared__ unsigned long long sm_hi[];
    __shared__ unsigned hist[256];
    __shared__ Prefix pre;
    __shared__ unsigned found;
    unsigned* sm_lo = (unsigned*)(sm_hi + P);
    scores += (int64_t)blockIdx.y * col_stride;
    st += blockIdx.y;
    cand += (size_t)blockIdx.y * kCandMax;
    ids_out += (size_t)blockIdx.y * k;
    vals_out += (size_t)blockIdx.y * k;
    prior_done();
    if (excl) exclude = excl[blockIdx.y];
    const unsigned long long bh = st->bound_hi;
    const unsigned bl = st->bound_lo;
    const int lane = threadIdx.x & 31;
    const int64_t stride = (int64_t)gridDim.x * kTopkThreads;
    const int64_t tid = (int64_t)blockIdx.x * kTopkThreads + threadIdx.x;
    constexpr int kU = 4;
    for (int64_t i0 = tid - lane; i0 < n; i0 += stride * kU) {  // warp-uniform
        double v[kU];
#pragma unroll
        for (int u = 0; u < kU; ++u)
            if (i0 + lane + u * stride < n) v[u] = scores[i0 + lane + u * stride];
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            const int64_t i = i0 + lane + u * stride;
            unsigned long long h = 0;
            const unsigned l = ~(unsigned)i;
            bool take = i < n && i != exclude;
            if (take) {
                h = ordered_bits(v[u]);
                take = h > bh || (h == bh && l >= bl);
            }
            const unsigned mask = __ballot_sync(0xffffffffu, take);
            if (!mask) continue;
            unsigned slot = 0;
            if (lane == 0) slot = atomicAdd(&st->count, (unsigned)__popc(mask));
            slot = __shfl_sync(0xffffffffu, slot, 0) + (unsigned)__popc(mask & ((1u << lane) - 1u));
            if (take && slot < cap) cand[slot] = Cand{h, l, 0u};
        }
    }
    if (!last_block(tickets + 2 * blockIdx.y + 1)) return;
    unsigned cnt = *(volatile unsigned*)&st->count;
    if (cnt <= cap) {
        for (int i = threadIdx.x; i < (int)cnt; i += kTopkThreads) {
            sm_hi[i] = __ldcg(&cand[i].hi);
            sm_lo[i] = __ldcg(&cand[i].lo);
        }
    } else {
        radix_select<0>(n, (unsigned)k, 0u, pre, hist, [&](int64_t i, unsigned long long& h, unsigned& l) {
            h = ordered_bits(scores[i]);
            l = ~(unsigned)i;
            return i != exclude;
        });
        if (threadIdx.x == 0) found = 0u;
        __syncthreads();
        const Prefix s = pre;
        for (int64_t i = threadIdx.x; i < n; i += kTopkThreads) {
            if (i == exclude) continue;
            const unsigned long long h = ordered_bits(scores[i]);
            const unsigned l = ~(unsigned)i;
            if (cmp_prefix(h, l, s, s.depth) < 0) continue;
            const unsigned slot = atomicAdd(&found, 1u);
            if (slot < (unsigned)P) {  // k keys, or all of them where there are fewer
                sm_hi[slot] = h;
                sm_lo[slot] = l;
            }
        }
        __syncthreads();
        cnt = found < (unsigned)P ? found : (unsigned)P;
    }
    int Q = 1;
    while (Q < (int)cnt) Q <<= 1;
    for (int i = threadIdx.x; i < Q; i += kTopkThreads)
        if (i >= (int)cnt) {
            sm_hi[i] = 0ull;  // (0, 0) is below every real key (ids < 2^31)
            sm_lo[i] = 0u;
        }
    __syncthreads();
    for (int size = 2; size <= Q; size <<= 1) {
        for (int half = size >> 1; half > 0; half >>= 1) {
            for (int p = threadIdx.x; p < Q / 2; p += kTopkThreads) {
                const int i = 2 * p - (p & (half - 1)), j = i + half;
                const unsigned long long ah = sm_hi[i], bh2 = sm_hi[j];
                const unsigned al = sm_lo[i], bl2 = sm_lo[j];
                const bool a_less = ah < bh2 || (ah == bh2 && al < bl2);
                const bool desc = (i & size) == 0;  // overall order: descending
                if (desc ? a_less : !a_less) {
                    sm_hi[i] = bh2;
                    sm_hi[j] = ah;
                    sm_lo[i] = bl2;
                    sm_lo[j] = al;
                }
            }
            __syncthreads();
        }
    }
    for (int i = threadIdx.x; i < k; i += kTopkThreads) {
        if (i < (int)cnt) {
            ids_out[i] = (int32_t)(~sm_lo[i]);
            vals_out[i] = from_ordered(sm_hi[i]);
        } else {
            ids_out[i] = -1;
            vals_out[i] = 0.0;
        }
    }
}

// Workspace of B columns: states, tickets (two each), maxima (hi, lo), candidates.
constexpr size_t kStateBytes(size_t B) { return ((sizeof(TopkState) + 2 * sizeof(unsigned)) * B + 255) / 256 * 256; }
constexpr size_t kColumnBytes = (size_t)kMaxSlices * 12 + sizeof(Cand) * (size_t)kCandMax;

// B selections; column q of scores starts at scores + q * stride, and excl[q] (or exclude
// where excl is NULL, -1 for none) is left out of it.  tickets: the blocks of the two launches
// that have finished, two per column, zero before and after; NULL: the workspace's, cleared here.
cudaError_t topk_select(cudaStream_t stream, int sms, int64_t n, int32_t B, const double* scores, int64_t col_stride,
                        int64_t exclude, const int64_t* excl, int32_t k, int32_t* ids_out, double* vals_out, void* ws,
                        unsigned* tickets) {
    TopkState* st = (TopkState*)ws;
    unsigned long long* max_hi = (unsigned long long*)((char*)ws + kStateBytes((size_t)B));
    unsigned* max_lo = (unsigned*)(max_hi + (size_t)B * kMaxSlices);
    Cand* cand = (Cand*)(max_lo + (size_t)B * kMaxSlices);
    // Slices: enough of them that their k-th maximum is a tight bound (with 4 k of them about
    // 1.15 k keys reach it), few enough for one block to select from, five registers a thread.
    // One element per thread until the chip is full, with one block per SM where its slices (32)
    // are enough, two otherwise; over all columns together two, and what a column's slices need.
    const int64_t want = 4 * (int64_t)k < 2048 ? 2048 : (4 * (int64_t)k > 8192 ? 8192 : 4 * (int64_t)k);
    int64_t most = std::max<int64_t>((2 * (int64_t)sms + B - 1) / B, want / kTopkThreads);
    if (B == 1 && want <= 32 * (int64_t)sms) most = sms;
    most = std::min<int64_t>(most, kMaxSlices / 32);  // slices of 32 warps always fit
    const int64_t blocks = std::min<int64_t>((n + kTopkThreads - 1) / kTopkThreads, most);
    const int64_t threads = blocks * kTopkThreads;
    int G = 1;
    while (G < 32 && threads / (2 * G) >= want) G <<= 1;
    const unsigned cap = (unsigned)(2 * k + 1024 < kCandMax ? 2 * k + 1024 : kCandMax);
    int P = 1;
    while (P < (int)cap) P <<= 1;
    const size_t smem = (size_t)P * 12;
    cudaError_t e = cudaSuccess;
    if (!tickets) {
        tickets = (unsigned*)(st + B);
        if ((e = cudaMemsetAsync(tickets, 0, 2 * sizeof(unsigned) * (size_t)B, stream)) != cudaSuccess) return e;
    }
    // the limit is the process's, for all handles and threads: always the same value, never a lower one
    if (smem > 48 * 1024 - 2048 &&
        (e = cudaFuncSetAttribute(topk_pick_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kCandMax * 12)) !=
            cudaSuccess)
        return e;
    const dim3 grid((unsigned)blocks, (unsigned)B);
    e = launch_after(stream, grid, kTopkThreads, 0, topk_bound_kernel, n, make_deal(n), scores, exclude, st, tickets, max_hi, max_lo, G,
                     (unsigned)k, col_stride, excl);
    if (e != cudaSuccess) return e;
    return launch_after(stream, grid, kTopkThreads, smem, topk_pick_kernel, n, scores, exclude, st, tickets, cand, cap, k, P,
                        col_stride, excl, ids_out, vals_out);
}

}  // namespace

size_t topk_batch_workspace_bytes(int32_t B) { return kStateBytes((size_t)B) + kColumnBytes * (size_t)B + 256; }

size_t topk_workspace_bytes(int64_t /*n*/) { return topk_batch_workspace_bytes(1); }

cudaError_t launch_topk(const Graph& g, const double* scores, int64_t exclude, int32_t k, int32_t* ids_out,
                        double* vals_out, void* ws) {
    return topk_select(g.stream, g.sm_count, g.n, 1, scores, 0, exclude, nullptr, k, ids_out, vals_out, ws,
                       topk_tickets(g));
}

cudaError_t launch_topk_batch(const Graph& g, int32_t B, const double* scores, const int64_t* exclude, int32_t k,
                              int32_t* ids_out, double* vals_out, void* ws) {
    return topk_select(g.stream, g.sm_count, g.n, B, scores, g.n, -1, exclude, k, ids_out, vals_out, ws, nullptr);
}

}  // namespace esim

// ---------------------------------------------------------------------------
// Top-k selection that allocates nothing (esim_select_topk_static).
//
// Some callers cannot call cudaMalloc: code that runs inside a host framework
// which owns every byte of device memory (a fixed arena or a memory-capped
// serving process), and latency-critical threads that must not pay the device
// synchronisation cudaMalloc/cudaFree may cause.  For them the selection's
// scratch (the slices' maxima and the candidate list, about 328 KB) lives in
// the file-scope array below instead of a library or caller allocation.  Every
// GPU that loads the library holds this array until the process exits.
//
// In host code the symbol `g_topk_static_scratch` is only a host-side stand-in:
// passing it to a kernel would fault or, where the GPU can reach host memory,
// silently use the wrong memory.  The device address is taken once per device
// with cudaGetSymbolAddress (the first call on a device does this, with that
// device current; make that first call before any stream capture) and passed to
// the kernels.  The address is remembered together with the unique id of the CUDA
// context it was taken in: after a device reset the device has a new context (and
// the array a new address), so the next call takes the address again.  All calls
// share the array and it keeps the last call's contents; its tickets are cleared every call.
// Calls whose work overlaps on the GPU (different streams, or several host threads) race on
// the array.
// ---------------------------------------------------------------------------

namespace {

constexpr size_t kStaticTopkScratchBytes = esim::kStateBytes(1) + esim::kColumnBytes;

static __device__ __align__(256) unsigned char g_topk_static_scratch[kStaticTopkScratchBytes];

constexpr int kStaticMaxDevices = 64;
std::mutex g_static_mu;
void* g_static_ptr[kStaticMaxDevices] = {};
int g_static_sms[kStaticMaxDevices] = {};
unsigned long long g_static_ctx[kStaticMaxDevices] = {};  // context id the address belongs to

typedef CUresult (*CtxGetCurrentFn)(CUcontext*);
typedef CUresult (*CtxGetIdFn)(CUcontext, unsigned long long*);

// Unique id of the CUDA context current on this thread, from the driver's entry points.
// With no context current yet, the device's primary context is made current first (the
// context the runtime would use); a context the caller made current is left alone.
cudaError_t current_context_id(int dev, unsigned long long* id) {
    static CtxGetCurrentFn get_current = nullptr;
    static CtxGetIdFn get_id = nullptr;
    if (!get_current || !get_id) {
        void* f0 = nullptr;
        void* f1 = nullptr;
        cudaDriverEntryPointQueryResult q0, q1;
        cudaError_t e = cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &f0, 12000, cudaEnableDefault, &q0);
        if (e != cudaSuccess) return e;
        e = cudaGetDriverEntryPointByVersion("cuCtxGetId", &f1, 12000, cudaEnableDefault, &q1);
        if (e != cudaSuccess) return e;
        if (q0 != cudaDriverEntryPointSuccess || q1 != cudaDriverEntryPointSuccess || !f0 || !f1)
            return cudaErrorNotSupported;
        get_current = (CtxGetCurrentFn)f0;
        get_id = (CtxGetIdFn)f1;
    }
    CUcontext ctx = nullptr;
    if (get_current(&ctx) != CUDA_SUCCESS) return cudaErrorDeviceUninitialized;
    if (!ctx) {
        cudaError_t e = cudaSetDevice(dev);
        if (e != cudaSuccess) return e;
        if (get_current(&ctx) != CUDA_SUCCESS || !ctx) return cudaErrorDeviceUninitialized;
    }
    if (get_id(ctx, id) != CUDA_SUCCESS) return cudaErrorDeviceUninitialized;
    return cudaSuccess;
}

// Device address of the scratch array and the SM count of the current device, taken
// again whenever the device's context differs from the one they were taken in.
cudaError_t static_scratch(int dev, void** ptr, int* sms) {
    std::lock_guard<std::mutex> lock(g_static_mu);
    unsigned long long ctx = 0;
    cudaError_t e = current_context_id(dev, &ctx);
    if (e != cudaSuccess) return e;
    if (!g_static_ptr[dev] || g_static_ctx[dev] != ctx) {
        void* p = nullptr;
        e = cudaGetSymbolAddress(&p, g_topk_static_scratch);
        if (e != cudaSuccess) return e;
        int s = 0;
        e = cudaDeviceGetAttribute(&s, cudaDevAttrMultiProcessorCount, dev);
        if (e != cudaSuccess) return e;
        g_static_sms[dev] = s;
        g_static_ptr[dev] = p;
        g_static_ctx[dev] = ctx;
    }
    *ptr = g_static_ptr[dev];
    *sms = g_static_sms[dev];
    return cudaSuccess;
}

esim_status static_fail(esim_status status, const std::string& message) {
    esim::set_error((int)status, message);
    return status;
}

}  // namespace

extern "C" __attribute__((visibility("default"))) esim_status esim_select_topk_static(
    const double* scores, int64_t n, int64_t exclude, int32_t k, int32_t* ids_out, double* vals_out, void* stream) {
    using namespace esim;
    if (!scores || !ids_out || !vals_out) return static_fail(ESIM_EINVAL, "NULL argument");
    if (n < 1 || n >= ((int64_t)1 << 31)) return static_fail(ESIM_EINVAL, "need 1 <= n < 2^31");
    if (k < 1) return static_fail(ESIM_EINVAL, "k must be >= 1");
    if (k > kTopkMax)
        return static_fail(ESIM_ENOTSUP, "k above 4096: the static top-k scratch holds at most 4096 candidates");
    if (exclude < -1 || exclude >= n) return static_fail(ESIM_EINVAL, "exclude out of range");
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return static_fail(ESIM_ECUDA, std::string("cudaGetDevice: ") + cudaGetErrorString(e));
    if (dev < 0 || dev >= kStaticMaxDevices) return static_fail(ESIM_ENOTSUP, "device ordinal above 63");
    void* ws = nullptr;
    int sms = 0;
    e = static_scratch(dev, &ws, &sms);
    if (e != cudaSuccess)
        return static_fail(ESIM_ECUDA, std::string("static scratch set-up: ") + cudaGetErrorString(e));
    e = topk_select((cudaStream_t)stream, sms, n, 1, scores, 0, exclude, nullptr, k, ids_out, vals_out, ws, nullptr);
    if (e != cudaSuccess) return static_fail(ESIM_ECUDA, std::string("static top-k launch: ") + cudaGetErrorString(e));
    return ESIM_OK;
}
