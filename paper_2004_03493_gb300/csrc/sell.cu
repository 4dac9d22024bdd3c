// The sliced layout of a CSR that the single-vector sweeps read (internal.h, SellRows):
// planned on the host and filled on the device when a graph is loaded.
//
// Rows are sorted by length, longest first, within windows of kSellWindow consecutive
// rows, so the 32 rows of a slice have nearly the same length and stay close together in
// every vector that is indexed by row.  The entries of a slice are stored step by step:
// the 32 rows' t-th entries side by side, so a warp reads them with one coalesced load.
// Rows of more than row_cap entries take slices of their own, before all others, the lanes
// side by side along the row.
// The layout is SELL-C-sigma (M. Kreutzer, G. Hager, G. Wellein, H. Fehske, A. R. Bishop, SIAM
// J. Sci. Comput. 36(5), 2014) with C = 32 and sigma = kSellWindow; the cut rows are added to it.
#include "common.cuh"
#include "internal.h"

#include <algorithm>
#include <vector>

namespace esim {

namespace {

// Hubs.  A gathered value occupies a whole 128-byte line of the L1, about 1800 lines; side by
// side the hubs share lines of 16 (FP32c: 32) values.  n = 1e6, m = 1.75e7, L = 33, forward and
// reverse, FP64 / FP32c: 4.75 / 4.36 ms without, 4.61 / 4.07 with 8192 hubs, 4.67 / 4.10 with
// 16384, 4.76 / 4.19 with 32768.  Loads that keep the hubs and pass the others by the L1 are
// two instructions a gather and lose (4.87 / 4.19).
constexpr uint32_t kSellHubs = 8192;

// What the device fills of one CSR, and of both: blockIdx.y picks.  Two launches for the two CSRs
// instead of six: a small graph's load is mostly calls of a fixed cost (random n = 2000, m = 20,000
// 0.306 -> 0.281 ms a load, n = 500, m = 3001 0.194 -> 0.172).
struct Fill {
    int64_t windows, npieces, nslices;
    uint32_t row_cap;
    const uint32_t* rp;
    const int32_t* col;
    const uint32_t* off;
    const uint32_t* pos;
    const Segment* piece;
    int2* rows;
    int32_t* out;
};
struct Fills {
    Fill of[2];
};

// One window per block: sorts its rows by (length descending, row ascending) and writes
// their (row, length).  Cut rows get no place; the blocks past the windows write the rows of
// their pieces, one slice per piece and warp.
__global__ void __launch_bounds__(kSellWindow) sell_rows_of_slices_kernel(int64_t n, const __grid_constant__ Fills fills) {
    const Fill& f = fills.of[blockIdx.y];
    __shared__ uint32_t key[kSellWindow];
    const int t = threadIdx.x;
    if ((int64_t)blockIdx.x >= f.windows) {
        const int64_t s = ((int64_t)blockIdx.x - f.windows) * (kSellWindow / 32) + (t >> 5);
        const uint32_t lane = t & 31;
        if (s < f.npieces) {
            const uint32_t len = f.piece[s].end - f.piece[s].beg;
            f.rows[s * 32 + lane] = make_int2(f.piece[s].row, (int)(len > lane ? (len - lane + 31) / 32 : 0u));
        }
        return;
    }
    const int64_t base = (int64_t)blockIdx.x * kSellWindow;
    uint32_t mine = 0;  // no row here
    if (base + t < n) {
        const uint32_t len = f.rp[base + t + 1] - f.rp[base + t];
        if (len <= f.row_cap) mine = ((len + 1) << 10) | (uint32_t)(kSellWindow - 1 - t);
    }
    key[t] = mine;
    __syncthreads();
    for (int size = 2; size <= kSellWindow; size <<= 1)
        for (int half = size >> 1; half > 0; half >>= 1) {
            const int j = t ^ half;
            if (j > t) {
                const uint32_t a = key[t], b = key[j];
                if ((t & size) == 0 ? a < b : a > b) {
                    key[t] = b;
                    key[j] = a;
                }
            }
            __syncthreads();
        }
    const uint32_t k = key[t];
    f.rows[f.npieces * 32 + base + t] =
        k ? make_int2((int)(base + kSellWindow - 1 - (int64_t)(k & (kSellWindow - 1))), (int)(k >> 10) - 1) : make_int2(-1, 0);
}

// The entries, slice by slice: one warp per slice.
__global__ void __launch_bounds__(kBlock) sell_fill_kernel(const __grid_constant__ Fills fills) {
    const Fill& f = fills.of[blockIdx.y];
    const int lane = threadIdx.x & 31;
    for (int64_t s = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; s < f.nslices;
         s += ((int64_t)gridDim.x * blockDim.x) >> 5) {
        const int2 r = f.rows[s * 32 + lane];
        const uint32_t o0 = f.off[s], o1 = f.off[s + 1];
        const bool wide = s < f.npieces;
        const uint32_t beg = wide ? f.piece[s].beg + lane : (r.x < 0 ? 0u : f.rp[r.x]);
        for (uint32_t t = 0; t < o1 - o0; ++t)
            f.out[((size_t)o0 + t) * 32 + lane] =
                t < (uint32_t)r.y ? (int32_t)at_pos(f.pos, f.col[beg + (wide ? 32 * t : t)]) : 0;
    }
}

// Positions of the gathered vector: the at most kSellHubs nodes with the most uses (node i has
// uses_rp[i+1] - uses_rp[i] of them, the row lengths of the transpose) first.  Empty where
// that would gain nothing: every node is one, or they have no more than twice their share.
std::vector<uint32_t> hub_positions(int64_t n, const std::vector<uint32_t>& uses_rp) {
    if (n <= (int64_t)kSellHubs) return {};
    constexpr uint32_t kTop = 1u << 16;  // uses above this are alike
    auto uses = [&](int64_t i) { return std::min(uses_rp[(size_t)i + 1] - uses_rp[(size_t)i], kTop); };
    uint32_t most = 0;
    for (int64_t i = 0; i < n; ++i) most = std::max(most, uses(i));
    std::vector<uint32_t> count((size_t)most + 1, 0);
    for (int64_t i = 0; i < n; ++i) ++count[uses(i)];
    uint32_t least = most + 1, h = 0;  // hubs: the nodes with at least this many uses
    uint64_t share = 0;
    while (least > 1 && h + count[least - 1] <= kSellHubs) {
        h += count[--least];
        share += (uint64_t)count[least] * least;
    }
    if (h == 0 || (double)share * (double)n < 2.0 * (double)h * (double)uses_rp[(size_t)n]) return {};
    std::vector<uint32_t> pos((size_t)n);
    uint32_t hub = 0, other = h;
    for (int64_t i = 0; i < n; ++i) pos[(size_t)i] = uses(i) >= least ? hub++ : other++;
    return pos;
}

}  // namespace

void plan_sell(int64_t n, const std::vector<uint32_t>& rp, const std::vector<Segment>& pieces,
               const std::vector<uint32_t>& uses_rp, SellRows& out, std::vector<uint32_t>& off,
               std::vector<uint32_t>& pos) {
    pos = hub_positions(n, uses_rp);
    out.npieces = (int64_t)pieces.size();
    const int64_t windows = (n + kSellWindow - 1) / kSellWindow;
    out.nslices = out.npieces + windows * (kSellWindow / 32);
    off.clear();
    off.reserve((size_t)out.nslices + 1);
    uint64_t total = 0;  // below 2^32: a step holds at least one entry, and m < 2^32
    auto slice = [&](uint32_t steps) {
        off.push_back((uint32_t)total);
        total += steps;
    };
    for (const Segment& p : pieces) slice((p.end - p.beg + 31) / 32);
    std::vector<uint32_t> count((size_t)out.row_cap + 1);
    for (int64_t w = 0; w < windows; ++w) {  // a slice's steps: the longest of its 32 rows, the first in sorted order
        std::fill(count.begin(), count.end(), 0u);
        const int64_t end = std::min(n, (w + 1) * kSellWindow);
        for (int64_t r = w * kSellWindow; r < end; ++r) {
            const uint32_t len = rp[(size_t)r + 1] - rp[(size_t)r];
            if (len <= out.row_cap) ++count[len];
        }
        uint32_t rows = 0, next = 0;
        for (int64_t len = out.row_cap; len >= 0; --len) {
            rows += count[(size_t)len];
            for (; next < rows; next += 32) slice((uint32_t)len);
        }
        for (; next < (uint32_t)kSellWindow; next += 32) slice(0);
    }
    off.push_back((uint32_t)total);
}

cudaError_t fill_sell(int64_t n, const DevCsr& in, const DevCsr& out, cudaStream_t stream) {
    const int64_t windows = (n + kSellWindow - 1) / kSellWindow;
    auto fill = [&](const DevCsr& d) {
        return Fill{windows, d.sell.npieces, d.sell.nslices, d.sell.row_cap, d.rp,   d.col,
                    d.sell.off, d.sell.pos,   d.sell.piece,  d.sell.rows,    d.sell.col};
    };
    const Fills fills{{fill(in), fill(out)}};
    const int64_t pieces = std::max(in.sell.npieces, out.sell.npieces), slices = std::max(in.sell.nslices, out.sell.nslices);
    sell_rows_of_slices_kernel<<<dim3((unsigned)(windows + (pieces * 32 + kSellWindow - 1) / kSellWindow), 2), kSellWindow, 0,
                                 stream>>>(n, fills);
    const int64_t blocks = std::min<int64_t>((slices * 32 + kBlock - 1) / kBlock, 65536);
    sell_fill_kernel<<<dim3((unsigned)blocks, 2), kBlock, 0, stream>>>(fills);
    return cudaGetLastError();
}

}  // namespace esim
