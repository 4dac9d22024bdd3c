// Sample allocation, walk-pair sampler and diagonal estimate.
//
//   allocation (Lemma 4, "Sampling according to pi(k)^2"; Algorithm 1 for the
//   basic form): pi(k) = sum_l pi^l(k); R(k) = ceil(R_b * pi(k)^2) or
//   ceil(R_b * pi(k)), at least 1 where pi(k) > 0; off = exclusive prefix sum
//   of R (uint64).
//
//   sampler (Algorithm 2, walk semantics of Eq. scwwalk): R(k) pairs of
//   independent sqrt(c)-walks from each node k; nonmeet(k) counts the pairs that
//   never visit the same node at the same step.  Pair r of node k draws its
//   randomness from Philox-4x32-10 with counter (r_lo, r_hi, k, t) at step t, so
//   the result is independent of how pairs are spread over threads.  In-neighbour
//   choices are exactly uniform (Lemire's multiply-shift with rejection, ACM TOMS
//   2019; rejected words are replaced from a side stream with counter
//   (r_lo, r_hi, k, 2^31 | W 2^30 | j 2^16 | t), W = 0 for walk A, 1 for walk B).
//
//   D^(k) = nonmeet(k) / R(k) (Algorithm 2).
#include "common.cuh"
#include "internal.h"
#include "philox.cuh"
#include "twofloat.cuh"

#include <math.h>

namespace esim {

// Nodes per thread of the allocation's and the scans' tiles: one where the nodes then fill the
// chip anyway and a thread's chain of loads is what the kernel takes, eight from there on, so
// that the tile sums stay few enough for one block to scan.
constexpr int kScanItems = 8;
constexpr int64_t kOneItemUpTo = 1 << 18;
static int scan_items(int64_t n) { return n <= kOneItemUpTo ? 1 : kScanItems; }
constexpr uint32_t kWalkMaxSteps = 65536;

int64_t allocate_blocks(int64_t n) {
    const int64_t tile = (int64_t)kBlock * scan_items(n);
    return (n + tile - 1) / tile;
}

uint32_t walk_threshold(double c) {
    double v = floor(sqrt(c) * 4294967296.0);
    if (v >= 4294967295.0) return 0xFFFFFFFFu;
    if (v <= 0.0) return 0u;
    return (uint32_t)v;
}

// Block-wide exclusive scan of one uint64 per thread; *total gets the block sum.
__device__ __forceinline__ unsigned long long block_exclusive_scan(unsigned long long v, unsigned long long* smem,
                                                                   unsigned long long* total) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int nw = (blockDim.x + 31) >> 5;
    unsigned long long x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        unsigned long long y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) smem[wid] = x;
    __syncthreads();
    if (wid == 0) {
        unsigned long long w = lane < nw ? smem[lane] : 0ull;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            unsigned long long y = __shfl_up_sync(0xffffffffu, w, o);
            if (lane >= o) w += y;
        }
        smem[lane] = w;
    }
    __syncthreads();
    const unsigned long long warp_off = wid ? smem[wid - 1] : 0ull;
    *total = smem[nw - 1];
    __syncthreads();
    return warp_off + x - v;
}

// pi(k) = sum over levels of hist, in level order: FP64 sums for an FP64 history,
// two-float sums (rounded to FP64) for an FP32 history.  kU levels are loaded at a time: they
// are n apart, and one after another their latencies would add up to most of a small query.
template <typename H, class Add>
__device__ __forceinline__ void each_level(const H* __restrict__ hist, int64_t n, int64_t k, int32_t L, const Add& add) {
    constexpr int kU = 8;
    for (int32_t l0 = 0; l0 <= L; l0 += kU) {
        H v[kU];
#pragma unroll
        for (int u = 0; u < kU; ++u)
            if (l0 + u <= L) v[u] = hist[(size_t)(l0 + u) * (size_t)n + (size_t)k];
#pragma unroll
        for (int u = 0; u < kU; ++u)
            if (l0 + u <= L) add(v[u]);
    }
}

__device__ __forceinline__ double level_sum(const double* __restrict__ hist, int64_t n, int64_t k, int32_t L) {
    double p = 0.0;
    each_level(hist, n, k, L, [&](double v) { p += v; });
    return p;
}

__device__ __forceinline__ double level_sum(const float* __restrict__ hist, int64_t n, int64_t k, int32_t L) {
    f2 p = f2{0.f, 0.f};
    each_level(hist, n, k, L, [&](float v) { p = f2_add_f(p, v); });
    return f2_to_double(p);
}

// The last block of a grid to get here: exclusive scan of the tile sums (in place), the total
// into off[n] and the status block, the budget check.  The ticket wraps to zero.
struct TileSums {
    unsigned long long* R;   // gridDim.x
    double* Rd;              // gridDim.x: the same in double, or NULL
    double* norm;            // gridDim.x sums of pi^2, or NULL
    unsigned* ticket;        // zero before the launch
};

__device__ __forceinline__ void finish_tiles(const TileSums& t, double budget, uint64_t* __restrict__ off_n,
                                             Status* __restrict__ st) {
    __shared__ bool last;
    __shared__ unsigned long long su[32];
    __shared__ double sd[32];
    if (threadIdx.x == 0) {  // it wrote this block's sums
        __threadfence();
        last = atomicInc(t.ticket, gridDim.x - 1) == gridDim.x - 1;
        __threadfence();
    }
    __syncthreads();
    if (!last) return;
    const int64_t nblocks = gridDim.x;
    const int64_t per = (nblocks + blockDim.x - 1) / blockDim.x;
    const int64_t b0 = (int64_t)threadIdx.x * per;
    const int64_t b1 = b0 + per < nblocks ? b0 + per : nblocks;
    unsigned long long local = 0;
    double nrm = 0.0, rd = 0.0;
    for (int64_t b = b0; b < b1; ++b) {
        local += __ldcg(t.R + b);
        if (t.norm) nrm += __ldcg(t.norm + b);
        if (t.Rd) rd += __ldcg(t.Rd + b);
    }
    unsigned long long total;
    unsigned long long run = block_exclusive_scan(local, su, &total);
    for (int64_t b = b0; b < b1; ++b) {
        const unsigned long long v = __ldcg(t.R + b);
        t.R[b] = run;
        run += v;
    }
    nrm = block_sum(nrm, sd);
    rd = block_sum(rd, sd);
    if (threadIdx.x == 0) {
        *off_n = total;
        if (st) {  // NULL: an auxiliary scan that records nothing
            st->sum_R = total;
            if (t.norm) st->pi_norm2 = nrm;
            if (rd > budget || rd >= 1.8e19) atomicOr(&st->err, kErrBudget);
        }
    }
}

// pi(k), R(k) per node; per-tile sums of R (exact and in double) and of pi^2, and their scan.
// Bound by the history's bytes on large graphs (n = 1e6, L = 33, FP64: 272 MB), by the chain
// of loads on small ones (n = 2000, L = 11: 29 us with eight nodes a thread and one load at a
// time and the tile sums' scan in a launch of its own, 10 now with that scan in its last block).
template <typename H, int kItems>
__global__ void __launch_bounds__(kBlock) alloc_reduce_kernel(int64_t n, const H* __restrict__ hist, int32_t L,
                                                              double R_b, int mode, const uint32_t* __restrict__ exact_din,
                                                              double* __restrict__ pi_out,
                                                              uint64_t* __restrict__ R_out, const TileSums tiles,
                                                              double budget, uint64_t* __restrict__ off_n,
                                                              Status* __restrict__ st) {
    __shared__ unsigned long long red_u[kBlock / 32];
    __shared__ double red_d[kBlock / 32];
    const int64_t base = (int64_t)blockIdx.x * kBlock * kItems;
    unsigned long long sum_r = 0;
    double norm = 0.0, sum_rd = 0.0;
    bool overflow = false;
#pragma unroll 1
    for (int i = 0; i < kItems; ++i) {
        const int64_t k = base + (int64_t)i * kBlock + threadIdx.x;
        if (k >= n) break;
        const double p = level_sum(hist, n, k, L);
        if (pi_out) pi_out[k] = p;
        const double v = mode == 0 ? R_b * (p * p) : R_b * p;
        unsigned long long r = 0;
        if (v >= 9.2e18 || v != v) {
            overflow = true;
        } else {
            r = (unsigned long long)ceil(v);
            if (r == 0ull && p > 0.0) r = 1ull;  // every reached node gets a pair
            // Algorithm 3: D is exact for din <= 1, so those nodes need no pairs
            if (exact_din && exact_din[k + 1] - exact_din[k] <= 1u) r = 0ull;
        }
        R_out[k] = r;
        sum_r += r;
        sum_rd += (double)r;
        norm += p * p;
    }
    if (overflow) atomicOr(&st->err, kErrBudget);
    sum_r = block_sum(sum_r, red_u);
    norm = block_sum(norm, red_d);
    sum_rd = block_sum(sum_rd, red_d);
    if (threadIdx.x == 0) {
        tiles.R[blockIdx.x] = sum_r;
        tiles.norm[blockIdx.x] = norm;
        tiles.Rd[blockIdx.x] = sum_rd;
    }
    finish_tiles(tiles, budget, off_n, st);
}

// off[k] = tile offset + exclusive prefix of R within the tile.
template <int kItems>
__global__ void __launch_bounds__(kBlock) alloc_scan_kernel(int64_t n, const uint64_t* R,
                                                            const unsigned long long* tile_off,
                                                            uint64_t* __restrict__ off) {
    __shared__ unsigned long long su[32];
    const int64_t base = ((int64_t)blockIdx.x * kBlock + threadIdx.x) * kItems;
    prior_done();
    unsigned long long v[kItems];
    unsigned long long local = 0;
#pragma unroll
    for (int i = 0; i < kItems; ++i) {
        const int64_t k = base + i;
        v[i] = k < n ? R[k] : 0ull;
        local += v[i];
    }
    unsigned long long total;
    unsigned long long run = tile_off[blockIdx.x] + block_exclusive_scan(local, su, &total);
#pragma unroll
    for (int i = 0; i < kItems; ++i) {
        const int64_t k = base + i;
        if (k < n) off[k] = run;
        run += v[i];
    }
}

static cudaError_t scan_offsets(const Graph& g, int64_t N, const uint64_t* R, const unsigned long long* tile_off,
                                uint64_t* off) {
    const unsigned nb = (unsigned)allocate_blocks(N);
    return scan_items(N) == 1
               ? launch_after(g.stream, dim3(nb), kBlock, 0, alloc_scan_kernel<1>, N, R, tile_off, off)
               : launch_after(g.stream, dim3(nb), kBlock, 0, alloc_scan_kernel<kScanItems>, N, R, tile_off, off);
}

template <typename H>
cudaError_t launch_allocate_t(const Graph& g, const H* hist, int32_t L, double R_b, int mode, double* pi_out,
                              uint64_t* R_out, uint64_t* off) {
    const int64_t nb = allocate_blocks(g.n);
    const TileSums tiles{g.scan_part, g.norm_part + nb, g.norm_part, scan_ticket(g)};
    auto* kernel = scan_items(g.n) == 1 ? alloc_reduce_kernel<H, 1> : alloc_reduce_kernel<H, kScanItems>;
    kernel<<<(unsigned)nb, kBlock, 0, g.stream>>>(g.n, hist, L, R_b, mode, g.alg3 ? g.in.rp : nullptr, pi_out, R_out,
                                                  tiles, g.pair_budget, off + g.n, g.status);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    return scan_offsets(g, g.n, R_out, g.scan_part, off);
}

cudaError_t launch_allocate(const Graph& g, const double* hist, int32_t L, double R_b, int mode, double* pi_out,
                            uint64_t* R_out, uint64_t* off) {
    return launch_allocate_t<double>(g, hist, L, R_b, mode, pi_out, R_out, off);
}

cudaError_t launch_allocate32(const Graph& g, const float* hist, int32_t L, double R_b, int mode, double* pi_out,
                              uint64_t* R_out, uint64_t* off) {
    return launch_allocate_t<float>(g, hist, L, R_b, mode, pi_out, R_out, off);
}

// Exactly uniform index in [0, d) from word x (Lemire); rejections (probability
// below d / 2^32) redraw from the walk's side stream.
__device__ __forceinline__ uint32_t pick_redraw(uint32_t d, unsigned long long m, uint32_t rlo, uint32_t rhi, uint32_t k,
                                             uint32_t tag, const PhiloxKeys& K) {
    const uint32_t thr = (0u - d) % d;
    uint32_t l = (uint32_t)m;
    uint32_t j = 0;
    int used = 4;
    uint4 z = make_uint4(0, 0, 0, 0);
    while (l < thr) {
        if (used == 4) {
            if (j == (1u << 14)) break;
            z = philox4x32_10(make_uint4(rlo, rhi, k, tag | (j << 16)), K);
            ++j;
            used = 0;
        }
        const uint32_t x = used == 0 ? z.x : (used == 1 ? z.y : (used == 2 ? z.z : z.w));
        ++used;
        m = (unsigned long long)x * d;
        l = (uint32_t)m;
    }
    return (uint32_t)(m >> 32);
}

// Walks shared across the columns of a batch: segment s covers pairs
// [rbase[s], rbase[s] + len) of node s / B (node-major, B segments per node).
struct SharedSegs {
    int B;                  // 0: segments are (column, node) = (s / n, s % n)
    const uint64_t* rbase;  // first pair index of each segment (NULL unless shared)
};

__device__ __forceinline__ uint32_t segment_node(unsigned long long seg, unsigned long long n_nodes,
                                                 const SharedSegs& sh) {
    if (sh.B) return (uint32_t)(seg / (unsigned long long)sh.B);
    return (uint32_t)(seg < n_nodes ? seg : seg % n_nodes);
}

// ---------------------------------------------------------------- sampler
//
// Graph form: a walk's position is the pair (first in-edge, din) of its node, and
// walk[p] holds that pair for the node behind in-edge p, so a step is one dependent
// 8-byte load per walk.  A node without in-edges has (node id, 0): (first, din) is unique
// per node either way, so two walks meet iff both words agree, and reading walk[first] of
// such a node stays inside the array (it has max(m, n) entries).
//
// A warp takes a chunk of consecutive pair indices at a time from a counter (the first
// one by its own number).  A segment is the run of pairs of one (column, node): in a
// single query segment k is node k; in a batch of B columns segment q*n + k is node k of
// column q; with shared walks segment k*B + i is interval i of node k.
//
// Long runs of one segment (run_one): node, depth and the first Philox round are the
// warp's, a lane whose pair ended takes the next pair number by a ballot and a prefix
// count, and the counts are added once per run.  Short segments (run_many): the lanes hold
// the offsets of 32 consecutive segments and find their pair's segment by shuffles; the
// window moves on while other lanes' pairs still run.
//
// What bounds it: the generator.  A Philox block is 20 wide multiplies, 4 cycles each on a
// scheduler's multiply pipe, and 40 three-input XORs, 2 cycles each on its integer pipe;
// alone it reaches 426 G blocks/s on this chip.  run_one needs 17 of the multiplies, 95
// instructions per warp and step in all, and runs at 282 G pair-steps/s (9.5e8 pairs on the
// n = 2000 graph at the paper's kappa: 8.0 ms; the multiply pipe 78 % busy).  One pair
// stream per thread over a (rowptr, col) CSR, which this replaces, took 130 instructions and
// two dependent loads per walk and step, and a fixed share of the pairs per thread: 11.8 ms
// there, and 207 against 122 ms on a batch of 64 sources.
// Eight blocks of 192 threads fill an SM as six of 256 do (8.32 and 8.36 ms).  The smaller ones
// leave the planning room beside four or five of them: with five, the n = 1e5 top-50 query
// takes 39.0 against 43.4 ms, with four 38.5 against 39.0.
constexpr int kWalkBlock = 192;
constexpr uint32_t kRunMin = 128;        // shortest run of one segment that gets a loop of its own
constexpr uint32_t kChunkMin = 256;      // pairs per chunk where there are many
constexpr uint32_t kChunkMax = 16384;    // few enough that the warps finish together
constexpr uint32_t kChunksPerWarp = 8;
constexpr int kSparseRuns = 8;           // segments of 32 with pairs
constexpr uint32_t kPhiloxM0 = 0xD2511F53u, kPhiloxM1 = 0xCD9E8D57u;

struct WalkArgs {
    const uint2* __restrict__ row;    // n: (first in-edge, din), or (node, 0); positions times 8 if narrow
    const uint2* __restrict__ walk;   // max(m, n): the same of the node behind each in-edge
    const uint64_t* __restrict__ off; // nseg + 1
    const uint8_t* __restrict__ depth;
    unsigned long long* __restrict__ counts;
    uint64_t nseg;
    uint64_t n;
    SharedSegs sh;
    uint32_t T;
};

__device__ __forceinline__ uint32_t lanes_below() {
    uint32_t m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

// Rounds first..9 of Philox-4x32-10.
template <int kFirst>
__device__ __forceinline__ uint4 philox_rounds(uint4 x, const PhiloxKeys& K) {
#pragma unroll
    for (int i = kFirst; i < 10; ++i) {
        const unsigned long long p0 = (unsigned long long)kPhiloxM0 * x.x;
        const unsigned long long p1 = (unsigned long long)kPhiloxM1 * x.z;
        x = make_uint4((uint32_t)(p1 >> 32) ^ x.y ^ K.k0[i], (uint32_t)p1, (uint32_t)(p0 >> 32) ^ x.w ^ K.k1[i],
                       (uint32_t)p0);
    }
    return x;
}

// The table entry i places after a row's first one.  kNarrow: positions are byte offsets
// of 32 bits (a table below 4 GiB), which the load adds to its uniform base.
template <bool kNarrow>
__device__ __forceinline__ uint2 walk_entry(const uint2* __restrict__ walk, uint32_t first, uint32_t i) {
    if constexpr (kNarrow)
        return __ldg(reinterpret_cast<const uint2*>(reinterpret_cast<const char*>(walk) + (first + (i << 3))));
    else return __ldg(walk + (first + i));
}

// Whether two walks stand on the same node.
template <bool kNarrow>
__device__ __forceinline__ bool same_node(uint2 A, uint2 B) {
    return kNarrow ? A.x == B.x : A.x == B.x && A.y == B.y;
}

// The move of both walks on the words w of step t; false when the pair does not go on
// (a walk stops or has nowhere to go).  forced: the step is taken without the draw.
template <bool kNarrow>
__device__ __forceinline__ bool walk_move(uint4 w, bool forced, uint32_t T, uint2& A, uint2& B, uint32_t rlo, uint32_t rhi,
                                          uint32_t k, uint32_t t, const uint2* __restrict__ walk, const PhiloxKeys& K) {
    const bool cont = (forced | ((w.x < T) & (w.z < T))) & (A.y != 0u) & (B.y != 0u);
    const unsigned long long ma = (unsigned long long)w.y * A.y;
    const unsigned long long mb = (unsigned long long)w.w * B.y;
    uint32_t ia = (uint32_t)(ma >> 32), ib = (uint32_t)(mb >> 32);
    if (__builtin_expect(cont & (((uint32_t)ma < A.y) | ((uint32_t)mb < B.y)), 0)) {
        if ((uint32_t)ma < A.y) ia = pick_redraw(A.y, ma, rlo, rhi, k, 0x80000000u | t, K);
        if ((uint32_t)mb < B.y) ib = pick_redraw(B.y, mb, rlo, rhi, k, 0xC0000000u | t, K);
    }
    if (cont) {
        A = walk_entry<kNarrow>(walk, A.x, ia);
        B = walk_entry<kNarrow>(walk, B.x, ib);
    }
    return cont;
}

// len pairs (r0, r0 + 1, ...; no carry into the high word) of node k, depth d (kForced:
// d > 0), by the whole warp.  Adds this lane's steps; returns its count: Algorithm 2 counts
// pairs that never meet, Algorithm 3 pairs that first meet after their d forced steps.
template <bool kForced, bool kNarrow>
__device__ __forceinline__ uint32_t run_one(const WalkArgs& a, uint32_t k, uint2 home, uint32_t d, uint32_t rlo0,
                                            uint32_t rhi, uint32_t len, const PhiloxKeys& K, uint32_t& steps) {
    const uint32_t lane = threadIdx.x & 31;
    // round 0 multiplies k and r only; of round 1 the product of the first word is the run's
    const unsigned long long q1 = (unsigned long long)kPhiloxM1 * k;
    const uint32_t x0 = (uint32_t)(q1 >> 32) ^ rhi ^ K.k0[0];
    const uint32_t y0 = (uint32_t)q1 ^ K.k0[1];
    const unsigned long long q0 = (unsigned long long)kPhiloxM0 * x0;
    const uint32_t z1 = (uint32_t)(q0 >> 32) ^ K.k1[1], w1 = (uint32_t)q0;
    uint32_t next = 32, rlo = rlo0 + lane, t = 0, cnt = 0;
    unsigned long long p = (unsigned long long)kPhiloxM0 * rlo;
    uint32_t ph = (uint32_t)(p >> 32) ^ K.k1[0], pl = (uint32_t)p ^ z1;
    uint2 A = home, B = home;
    auto words = [&]() {
        const unsigned long long p1 = (unsigned long long)kPhiloxM1 * (ph ^ t);
        return philox_rounds<2>(make_uint4((uint32_t)(p1 >> 32) ^ y0, (uint32_t)p1, pl, w1), K);
    };
    auto restart = [&](uint32_t i) {
        rlo = rlo0 + i;
        p = (unsigned long long)kPhiloxM0 * rlo;
        ph = (uint32_t)(p >> 32) ^ K.k1[0];
        pl = (uint32_t)p ^ z1;
        t = 0;
        A = B = home;
    };
    // While 32 more pairs are left every lane has one, and before iteration 65535 no pair is
    // that long: neither is tested here.
    uint32_t it = 0;
    auto step = [&]() {
        const uint4 w = words();
        const bool cont = walk_move<kNarrow>(w, kForced && t < d, a.T, A, B, rlo, rhi, k, t, a.walk, K);
        const bool go = cont & !same_node<kNarrow>(A, B);
        if (kForced) cnt += (cont & !go & (t >= d)) ? 1u : 0u;
        else cnt += cont ? 0u : 1u;
        const uint32_t done = __ballot_sync(0xffffffffu, !go);
        ++t;
        if (!go) restart(next + __popc(done & lanes_below()));
        next += __popc(done);
    };
    if (!kForced)  // two steps a turn: 1.5 % less (forced pairs are slower for it)
        for (; next + 64 <= len && it < kWalkMaxSteps - 2; it += 2) {
            step();
            step();
        }
    for (; next + 32 <= len && it < kWalkMaxSteps - 1; ++it) step();
    steps += it;
    bool active = rlo - rlo0 < len;
    while (__any_sync(0xffffffffu, active)) {
        const uint4 w = words();
        const bool cont = active && walk_move<kNarrow>(w, kForced && t < d, a.T, A, B, rlo, rhi, k, t, a.walk, K);
        const bool meet = cont & same_node<kNarrow>(A, B);
        const bool ended = active & !(cont & !meet & (t + 1u < kWalkMaxSteps));
        steps += active ? 1u : 0u;
        cnt += (ended & (kForced ? meet & (t >= d) : !meet)) ? 1u : 0u;
        const uint32_t done = __ballot_sync(0xffffffffu, ended);
        ++t;
        if (ended) {
            const uint32_t i = next + __popc(done & lanes_below());
            active = i < len;
            restart(i);
        }
        next += __popc(done);
    }
    return cnt;
}

// Index of the segment that holds pair g (off[seg] <= g < off[seg+1]), seg >= lo, by the
// whole warp: each round splits the interval in 32.
__device__ __forceinline__ uint64_t find_segment(const uint64_t* __restrict__ off, uint64_t lo, uint64_t hi,
                                                 unsigned long long g) {
    const uint32_t lane = threadIdx.x & 31;
    while (hi - lo > 1) {  // off[lo] <= g < off[hi]
        const uint64_t step = (hi - lo + 31) >> 5;
        const uint64_t at = lo + (uint64_t)(lane + 1) * step;
        const bool below = at < hi && __ldg(off + at) <= g;
        const int c = __popc(__ballot_sync(0xffffffffu, below));  // the lanes below are the first c
        const uint64_t nlo = lo + (uint64_t)c * step;
        hi = nlo + step < hi ? nlo + step : hi;
        lo = nlo;
    }
    return lo;
}

// The pairs from g on, up to g1 or to the first segment with kRunMin pairs or more of the
// chunk, over many segments; seg holds g.  Returns where it stopped (seg likewise).
// A window of 32 segments with fewer than 32 pairs in fewer than kSparseRuns of them is one of
// 32 pairs instead, and each lane finds the segment of its own: in a batch whose sources share an
// eps most of a node's 64 segments have no pairs, and windows of segments took a turn for every
// one or two of them (64 sources on a random graph of 50,000 nodes, eps = 1e-2: walks 572 us,
// 107 now; one pair in every 64th of 4e6 nodes 98 and 34).  The registers it takes cost the windows of
// segments 2 % (random n = 400,003, m = 4,000,001, eps = 3e-4: walks 410 and 418 us).  Not inlined 2 % more; a
// kernel without depths beside this one gets half of it back and loses 0.6 % on long runs (8.23 and 8.28 ms).
template <bool kNarrow>
__device__ __forceinline__ unsigned long long run_many(const WalkArgs& a, unsigned long long g, unsigned long long g1,
                                                    uint64_t& seg_io, const PhiloxKeys& K, uint32_t& steps) {
    const uint32_t lane = threadIdx.x & 31;
    uint64_t wseg = seg_io;        // the window: segments wseg .. wseg + 31, one per lane
    uint32_t wend = 0, next = 0;   // pairs g + [next, wend) of the window are not taken yet
    uint32_t start = 0;            // pair number (from g) at which this lane's segment starts
    bool sparse = false;           // the window is 32 pairs, start the segment (from wseg) of the lane's pair
    bool last = false;             // no window after this one
    bool active = false;
    uint32_t k = 0, rlo = 0, rhi = 0, t = 0, d = 0;
    uint64_t seg = 0;
    uint2 A = make_uint2(0u, 0u), B = A;
    bool first = true;
    for (;;) {
        const uint32_t idle = __ballot_sync(0xffffffffu, !active);
        if (idle && next >= wend && !last) {  // the next window (uniform)
            if (!first) {
                wseg += sparse ? __shfl_sync(0xffffffffu, start, (int)wend - 1) : 32u;
                g += wend;
                next = wend = 0;
            }
            first = false;
            if (g >= g1 || wseg >= a.nseg) {
                last = true;
            } else {
                uint64_t e = wseg + lane + 1 <= a.nseg ? wseg + lane + 1 : a.nseg;
                unsigned long long hi = __ldg(a.off + e);
                if (!__any_sync(0xffffffffu, hi > g)) {  // a stretch without pairs: to the one that holds g
                    wseg = find_segment(a.off, wseg + 32, a.nseg, g);
                    e = wseg + lane + 1 <= a.nseg ? wseg + lane + 1 : a.nseg;
                    hi = __ldg(a.off + e);
                }
                if (hi > g1) hi = g1;
                if (hi < g) hi = g;
                unsigned long long lo = __shfl_up_sync(0xffffffffu, hi, 1);
                if (lane == 0) lo = g;
                const uint32_t large = __ballot_sync(0xffffffffu, hi - lo >= kRunMin);
                const int upto = large ? __ffs(large) - 1 : 32;  // segments of the window to run here
                start = (uint32_t)(lo - g);
                const uint32_t all = (uint32_t)(__shfl_sync(0xffffffffu, hi, 31) - g);
                wend = upto < 32 ? __shfl_sync(0xffffffffu, start, upto & 31) : all;
                sparse = upto == 32 && all < 32 && all < g1 - g &&
                         __popc(__ballot_sync(0xffffffffu, hi > lo)) < kSparseRuns;
                if (sparse) {
                    const unsigned long long p = g + lane;
                    uint64_t width = 32;  // probes this far apart, until they reach past the 32 pairs
                    unsigned long long probe;
                    for (;; width *= 8) {
                        const uint64_t at = wseg + width * (lane + 1);
                        probe = at < a.nseg ? __ldg(a.off + at) : ~0ull;
                        if (__shfl_sync(0xffffffffu, probe, 31) > g + 31) break;
                    }
                    uint32_t below = 0;  // probes at or before p
#pragma unroll
                    for (uint32_t s = 16; s > 0; s >>= 1)
                        if (__shfl_sync(0xffffffffu, probe, below + s - 1) <= p) below += s;
                    uint64_t in = wseg + width * below;  // off[in] <= p
                    uint64_t end = in + width < a.nseg ? in + width : a.nseg;
                    while (end - in > 1) {
                        const uint64_t mid = (in + end) >> 1;
                        if (__ldg(a.off + mid) <= p) in = mid; else end = mid;
                    }
                    // the first lane's segment lies in the window, or was searched for above
                    const uint32_t out = __ballot_sync(0xffffffffu, p >= g1 || in - wseg > 0xffffffffull);
                    start = (uint32_t)(in - wseg);
                    wend = out ? (uint32_t)__ffs(out) - 1u : 32u;
                }
                if (upto < 32) {
                    last = true;
                    if ((int)lane >= upto) start = 0xffffffffu;
                    seg_io = wseg + (uint32_t)upto;
                }
            }
        }
        // idle lanes take pairs: the segment is the last one that starts at or before it, or the found one
        if (idle) {
            const uint32_t i = next + __popc(idle & lanes_below());
            const bool take = !active && i < wend;
            uint32_t j = 0;
            if (sparse) {
                j = __shfl_sync(0xffffffffu, start, i & 31u);
            } else {
#pragma unroll
                for (int s = 16; s > 0; s >>= 1) {
                    const uint32_t v = __shfl_sync(0xffffffffu, start, j + s);
                    if (v <= i) j += s;
                }
            }
            next += __popc(idle);
            if (next > wend) next = wend;
            if (take) {
                seg = wseg + j;
                k = segment_node(seg, a.n, a.sh);
                const unsigned long long r = (a.sh.rbase ? __ldg(a.sh.rbase + seg) : 0ull) + (g + i - __ldg(a.off + seg));
                rlo = (uint32_t)r;
                rhi = (uint32_t)(r >> 32);
                d = a.depth ? a.depth[k] : 0u;
                A = B = __ldg(a.row + k);
                t = 0;
                active = true;
            }
        }
        if (!__any_sync(0xffffffffu, active)) {
            if (last) break;
            continue;
        }
        const uint4 w = philox_rounds<0>(make_uint4(rlo, rhi, k, t), K);
        const bool cont = active && walk_move<kNarrow>(w, t < d, a.T, A, B, rlo, rhi, k, t, a.walk, K);
        const bool meet = cont & same_node<kNarrow>(A, B);
        const bool go = cont & !meet & (t + 1u < kWalkMaxSteps);
        steps += active ? 1u : 0u;
        if (active & !go) {
            if (d ? (meet & (t >= d)) : !meet) atomicAdd(a.counts + seg, 1ull);
            active = false;
        }
        ++t;
    }
    return g + wend;
}

// Persistent walk-pair sampler (see above).  taken: the chunks taken beyond every warp's first,
// zero before the launch and this launch's alone while it runs; or NULL, and each block takes a
// fixed share of the chunks, for launches that may run several times at once (a captured
// graph's).  The fixed shares end unevenly: 64 sources on R-MAT 2^17 115 against 100 ms.
// kSide: the launch beside the planning's kernels, a function of its own for its carve-out.  An SM
// divides its L1 and shared memory when a block comes to it idle, and a block that needs more
// shared memory than the division gives waits until the SM is idle again.  The sampler uses
// next to none and stays for the whole launch, so with the division left to it every planning
// kernel with tables in shared memory waited for its end and nothing overlapped.
template <bool kNarrow, bool kSide>
__global__ void __launch_bounds__(kWalkBlock, 8) sample_pairs_kernel(const __grid_constant__ WalkArgs a, const __grid_constant__ PhiloxKeys K,
                                                                 double budget,
                                                                 unsigned long long* __restrict__ steps_out,
                                                                 Status* __restrict__ st,
                                                                 unsigned long long* __restrict__ taken) {
    __shared__ unsigned long long wsteps[kWalkBlock / 32];
    __shared__ unsigned long long own;  // taken of this block's chunks (no counter)
    unsigned long long total = __ldg(a.off + a.nseg);
    if ((double)total > budget || (st->err & kErrBudget)) {
        if (blockIdx.x == 0 && threadIdx.x == 0) atomicOr(&st->err, kErrBudget);
        total = 0ull;  // no walks
    }
    const uint32_t lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const unsigned long long nwarps = (unsigned long long)gridDim.x * (kWalkBlock / 32);
    // A few pairs are spread over all warps, 32 or more each: the launch then lasts as long as
    // its longest pair (18,000 pairs: the query takes 329 us, 370 with chunks of 256).  Many go
    // in chunks of at least kChunkMin, which pay for the search for their segment, about
    // kChunksPerWarp for each warp (24 instead of 8: 8.50 against 8.39 ms).
    unsigned long long size = total / nwarps < kChunkMin ? total / nwarps : kChunkMin;
    if (total / (nwarps * kChunksPerWarp) > size) size = total / (nwarps * kChunksPerWarp);
    size = size < 32 ? 32 : (size > kChunkMax ? kChunkMax : size);
    const unsigned long long nchunks = (total + size - 1) / size;
    if (lane == 0) wsteps[wid] = 0ull;
    if (threadIdx.x == 0) own = kWalkBlock / 32;
    __syncthreads();
    // consecutive chunks go to different blocks, so that a few chunks use all SMs
    unsigned long long c = (unsigned long long)wid * gridDim.x + blockIdx.x;
    while (c < nchunks) {
        unsigned long long g = c * size;
        const unsigned long long g1 = g + size < total ? g + size : total;
        uint64_t seg = find_segment(a.off, 0, a.nseg, g);
        uint32_t steps = 0;
        while (g < g1) {
            const unsigned long long sb = __ldg(a.off + seg), se = __ldg(a.off + seg + 1);
            unsigned long long end = se < g1 ? se : g1;
            // a long run, or what is left of the chunk lies in one segment
            if (end - g >= kRunMin || end == g1) {
                const uint32_t k = segment_node(seg, a.n, a.sh);
                const unsigned long long r = (a.sh.rbase ? __ldg(a.sh.rbase + seg) : 0ull) + (g - sb);
                const unsigned long long carry = (1ull << 32) - (r & 0xffffffffull);  // pairs to the next high word
                if (end - g > carry) end = g + carry;
                const uint32_t d = a.depth ? a.depth[k] : 0u, len = (uint32_t)(end - g);
                const uint2 home = __ldg(a.row + k);
                uint32_t cnt = d ? run_one<true, kNarrow>(a, k, home, d, (uint32_t)r, (uint32_t)(r >> 32), len, K, steps)
                                 : run_one<false, kNarrow>(a, k, home, 0u, (uint32_t)r, (uint32_t)(r >> 32), len, K, steps);
                cnt = __reduce_add_sync(0xffffffffu, cnt);
                if (lane == 0 && cnt) atomicAdd(a.counts + seg, (unsigned long long)cnt);
                g = end;
                if (g == se) ++seg;
                if (g < g1 && __ldg(a.off + seg + 1) <= g) seg = find_segment(a.off, seg, a.nseg, g);
            } else {
                g = run_many<kNarrow>(a, g, g1, seg, K, steps);
            }
        }
        steps = __reduce_add_sync(0xffffffffu, steps);
        if (lane == 0) {
            wsteps[wid] += steps;
            c = taken ? nwarps + atomicAdd(taken, 1ull) : atomicAdd(&own, 1ull) * gridDim.x + blockIdx.x;
        }
        c = __shfl_sync(0xffffffffu, c, 0);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned long long s = 0;
        for (int w = 0; w < kWalkBlock / 32; ++w) s += wsteps[w];
        if (s) atomicAdd(steps_out, s);
    }
}

__global__ void dhat_kernel(int64_t n, const uint64_t* nonmeet, const uint64_t* off,
                            double* __restrict__ dhat) {
    prior_done();
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x) {
        dhat[k] = pair_ratio(nonmeet[k], off[k + 1] - off[k]);
    }
}

__global__ void fill_kernel(int64_t n, double value, double* __restrict__ out) {
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x)
        out[k] = value;
}

__global__ void mask_R_kernel(int64_t n, const uint64_t* __restrict__ R, const uint8_t* __restrict__ keep,
                              uint8_t want_mask, uint64_t* __restrict__ R_out) {
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x)
        R_out[k] = ((want_mask >> keep[k]) & 1u) ? R[k] : 0ull;
}

__global__ void merge_counts_kernel(int64_t n, const uint8_t* __restrict__ cand, const uint64_t* __restrict__ side,
                                    uint64_t* __restrict__ counts) {
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x)
        if (cand[k] != 1) counts[k] = side[k];
}

__global__ void plan_scatter_kernel(const PlanEntry* __restrict__ plan, int count, uint64_t* __restrict__ R,
                                    uint8_t* __restrict__ depth, uint8_t* __restrict__ cand) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < count; i += gridDim.x * blockDim.x) {
        const PlanEntry e = plan[i];
        if (e.depth) {
            R[e.k] = e.R;
            depth[e.k] = e.depth;
        }
        if (e.early) cand[e.k] = 2;
    }
}

__global__ void mark_kernel(const int32_t* __restrict__ ids, int count, uint8_t* __restrict__ mark) {
    for (int i = threadIdx.x; i < count; i += blockDim.x) mark[ids[i]] = 1u;
}

// (first in-edge, din) of every node, or (node, 0) without in-edges; positions times 8 in
// a narrow table; and 1/din and floor((2^64 - 1) / din)
__global__ void walk_rows_kernel(int64_t n, const uint32_t* __restrict__ rp, int shift, uint2* __restrict__ row,
                                 double* __restrict__ inv_din, unsigned long long* __restrict__ magic) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t b = rp[i], d = rp[i + 1] - b;
        row[i] = make_uint2(((d ? b : (uint32_t)i) << shift) | (d || !shift ? 0u : 4u), d);
        inv_din[i] = d ? 1.0 / (double)d : 0.0;
        magic[i] = d >= 2 ? ~0ull / d : 0ull;
    }
}

// the same of the node behind every in-edge
__global__ void walk_edges_kernel(int64_t m, const int32_t* __restrict__ col, const uint2* __restrict__ row,
                                  uint2* __restrict__ walk) {
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < m; p += (int64_t)gridDim.x * blockDim.x)
        walk[p] = row[col[p]];
}

static int eb_cap(const Graph& g, int64_t n) {
    int64_t b = (n + kBlock - 1) / kBlock;
    if (b > (int64_t)g.sm_count * 8) b = (int64_t)g.sm_count * 8;
    return (int)(b < 1 ? 1 : b);
}

// 32-bit byte offsets reach the whole walk table
static bool walk_narrow(const Graph& g) { return (g.m > g.n ? g.m : g.n) < ((int64_t)1 << 29); }

cudaError_t launch_walk_table(const Graph& g) {
    walk_rows_kernel<<<eb_cap(g, g.n), kBlock, 0, g.stream>>>(g.n, g.in.rp, walk_narrow(g) ? 3 : 0, g.in.info, g.inv_din,
                                                               g.din_magic);
    walk_edges_kernel<<<eb_cap(g, g.m), kBlock, 0, g.stream>>>(g.m, g.in.col, g.in.info, g.in.walk);
    return cudaGetLastError();
}

cudaError_t launch_mask_R(const Graph& g, const uint64_t* R, const uint8_t* keep, uint8_t want_mask, uint64_t* R_out) {
    mask_R_kernel<<<eb_cap(g, g.n), kBlock, 0, g.stream>>>(g.n, R, keep, want_mask, R_out);
    return cudaGetLastError();
}

cudaError_t launch_merge_counts(const Graph& g, const uint8_t* cand, const uint64_t* side, uint64_t* counts) {
    merge_counts_kernel<<<eb_cap(g, g.n), kBlock, 0, g.stream>>>(g.n, cand, side, counts);
    return cudaGetLastError();
}

cudaError_t launch_plan_scatter(const Graph& g, const PlanEntry* plan, int count, uint64_t* R, uint8_t* depth,
                                uint8_t* cand) {
    if (count <= 0) return cudaSuccess;
    plan_scatter_kernel<<<1, kBlock, 0, g.stream>>>(plan, count, R, depth, cand);
    return cudaGetLastError();
}

cudaError_t launch_mark(const Graph& g, const int32_t* ids, int count, uint8_t* mark) {
    mark_kernel<<<1, kBlock, 0, g.stream>>>(ids, count, mark);
    return cudaGetLastError();
}

static int g_sample_blocks_per_sm = 0;

cudaError_t launch_sample(const Graph& g, const uint64_t* off, double c, uint64_t seed, uint64_t* nonmeet,
                          uint64_t* pair_steps, const uint8_t* depth, unsigned long long* taken) {
    return launch_sample_segments(g, g.n, off, c, seed, nonmeet, taken, pair_steps, depth);
}

cudaError_t launch_sample_segments(const Graph& g, int64_t nseg, const uint64_t* off, double c, uint64_t seed,
                                   uint64_t* nonmeet, unsigned long long* taken, uint64_t* pair_steps,
                                   const uint8_t* depth, int shared_B,
                                   const uint64_t* rbase, bool zero_counts) {
    cudaError_t e = cudaSuccess;
    if (zero_counts && (e = cudaMemsetAsync(nonmeet, 0, sizeof(uint64_t) * (size_t)nseg, g.stream)) != cudaSuccess)
        return e;
    unsigned long long* steps = pair_steps ? (unsigned long long*)pair_steps : &g.status->pair_steps;
    if (pair_steps) {
        e = cudaMemsetAsync(pair_steps, 0, sizeof(uint64_t), g.stream);
        if (e != cudaSuccess) return e;
    }
    if (g_sample_blocks_per_sm == 0) {
        int b = 0;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, (sample_pairs_kernel<true, false>), kWalkBlock, 0);
        if (e != cudaSuccess) return e;
        g_sample_blocks_per_sm = b > 0 ? b : 1;
    }
    const int per_sm = g.sample_block_cap > 0 && g.sample_block_cap < g_sample_blocks_per_sm ? g.sample_block_cap
                                                                                              : g_sample_blocks_per_sm;
    const unsigned blocks = (unsigned)(g.sm_count * per_sm);
    const WalkArgs a{g.in.info, g.in.walk, off, depth, (unsigned long long*)nonmeet, (uint64_t)nseg, (uint64_t)g.n,
                     SharedSegs{rbase ? shared_B : 0, rbase}, walk_threshold(c)};
    const bool side = steps == &g.status->pair_steps_side;  // it may run beside a launch on the query's own stream
    auto* kernel = walk_narrow(g) ? (side ? sample_pairs_kernel<true, true> : sample_pairs_kernel<true, false>)
                                  : (side ? sample_pairs_kernel<false, true> : sample_pairs_kernel<false, false>);
    if (side && (e = cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout,
                                          cudaSharedmemCarveoutMaxShared)) != cudaSuccess)
        return e;
    kernel<<<blocks, kWalkBlock, 0, g.stream>>>(a, philox_keys(seed), g.pair_budget, steps, g.status, taken);
    return cudaGetLastError();
}

cudaError_t launch_dhat(const Graph& g, const uint64_t* nonmeet, const uint64_t* off, double* dhat) {
    return launch_dhat_segments(g, g.n, nonmeet, off, dhat);
}

cudaError_t launch_fill(const Graph& g, int64_t n, double value, double* out) {
    int64_t b = (n + kBlock - 1) / kBlock;
    if (b > (int64_t)g.sm_count * 8) b = (int64_t)g.sm_count * 8;
    fill_kernel<<<(unsigned)(b < 1 ? 1 : b), kBlock, 0, g.stream>>>(n, value, out);
    return cudaGetLastError();
}

cudaError_t launch_dhat_segments(const Graph& g, int64_t nseg, const uint64_t* nonmeet, const uint64_t* off,
                                 double* dhat) {
    int64_t b = (nseg + kBlock - 1) / kBlock;
    if (b > (int64_t)g.sm_count * 8) b = (int64_t)g.sm_count * 8;
    return launch_after(g.stream, dim3((unsigned)(b < 1 ? 1 : b)), kBlock, 0, dhat_kernel, nseg, nonmeet, off, dhat);
}

// Scan of a ready R array of N segments (batches): tile sums and their scan, then off[].
template <int kItems>
__global__ void __launch_bounds__(kBlock) tile_sums_kernel(int64_t N, const uint64_t* __restrict__ R,
                                                           const TileSums tiles, double budget,
                                                           uint64_t* __restrict__ off_n, Status* __restrict__ st) {
    __shared__ unsigned long long red_u[kBlock / 32];
    __shared__ double red_d[kBlock / 32];
    const int64_t base = (int64_t)blockIdx.x * kBlock * kItems;
    unsigned long long su = 0;
    double sd = 0.0;
    for (int i = 0; i < kItems; ++i) {
        const int64_t k = base + (int64_t)i * kBlock + threadIdx.x;
        if (k < N) {
            su += R[k];
            sd += (double)R[k];
        }
    }
    su = block_sum(su, red_u);
    sd = block_sum(sd, red_d);
    if (threadIdx.x == 0) {
        tiles.R[blockIdx.x] = su;
        tiles.Rd[blockIdx.x] = sd;
    }
    finish_tiles(tiles, budget, off_n, st);
}

cudaError_t launch_scan_R(const Graph& g, int64_t N, const uint64_t* R, uint64_t* off, unsigned long long* part_R,
                          double* part_Rd, unsigned* ticket, bool record) {
    const int64_t nb = allocate_blocks(N);
    const TileSums tiles{part_R, part_Rd, nullptr, ticket};  // the scan of a ready R leaves the recorded ||pi||^2 as it is
    auto* kernel = scan_items(N) == 1 ? tile_sums_kernel<1> : tile_sums_kernel<kScanItems>;
    kernel<<<(unsigned)nb, kBlock, 0, g.stream>>>(N, R, tiles, g.pair_budget, off + N, record ? g.status : nullptr);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    return scan_offsets(g, N, R, part_R, off);
}

// The nodes with h != 0, ascending, into ids, and their number: tile counts and their scan,
// then the ids.
template <int kItems>
__global__ void __launch_bounds__(kBlock) support_tiles_kernel(int64_t n, const double* h,
                                                               const TileSums tiles, uint64_t* __restrict__ count) {
    __shared__ unsigned long long red[kBlock / 32];
    prior_done();
    const int64_t base = ((int64_t)blockIdx.x * kBlock + threadIdx.x) * kItems;
    unsigned long long c = 0;
#pragma unroll
    for (int i = 0; i < kItems; ++i) c += base + i < n && h[base + i] != 0.0;
    c = block_sum(c, red);
    if (threadIdx.x == 0) tiles.R[blockIdx.x] = c;
    finish_tiles(tiles, 0.0, count, nullptr);
}

template <int kItems>
__global__ void __launch_bounds__(kBlock) support_ids_kernel(int64_t n, const double* h,
                                                             const unsigned long long* tile_off,
                                                             int32_t* __restrict__ ids) {
    __shared__ unsigned long long su[32];
    prior_done();
    const int64_t base = ((int64_t)blockIdx.x * kBlock + threadIdx.x) * kItems;
    unsigned set = 0;
#pragma unroll
    for (int i = 0; i < kItems; ++i) set |= base + i < n && h[base + i] != 0.0 ? 1u << i : 0u;
    unsigned long long total;
    unsigned long long at = tile_off[blockIdx.x] + block_exclusive_scan((unsigned long long)__popc(set), su, &total);
#pragma unroll
    for (int i = 0; i < kItems; ++i)
        if (set >> i & 1u) ids[at++] = (int32_t)(base + i);
}

cudaError_t launch_support(const Graph& g, const double* h, int32_t* ids, uint64_t* count) {
    const unsigned nb = (unsigned)allocate_blocks(g.n);
    const TileSums tiles{g.scan_part, nullptr, nullptr, scan_ticket(g)};
    const bool one = scan_items(g.n) == 1;
    const cudaError_t e = one ? launch_after(g.stream, dim3(nb), kBlock, 0, support_tiles_kernel<1>, g.n, h, tiles, count)
                              : launch_after(g.stream, dim3(nb), kBlock, 0, support_tiles_kernel<kScanItems>, g.n, h,
                                             tiles, count);
    if (e != cudaSuccess) return e;
    return one ? launch_after(g.stream, dim3(nb), kBlock, 0, support_ids_kernel<1>, g.n, h, g.scan_part, ids)
               : launch_after(g.stream, dim3(nb), kBlock, 0, support_ids_kernel<kScanItems>, g.n, h, g.scan_part, ids);
}

}  // namespace esim
