// C ABI of the library (include/exactsim.h): graph loading, options, the whole
// query pipeline (Algorithm 1 with Algorithm 2 and the Lemma 4 allocation) and
// the step entry points.
#include "exactsim.h"
#include "internal.h"

#include <math.h>
#include <stddef.h>
#include <stdio.h>
#include <string.h>

#include <algorithm>
#include <atomic>
#include <memory>
#include <new>
#include <string>
#include <thread>
#include <vector>

using namespace esim;

struct esim_graph {
    Graph g;
};

namespace {

thread_local std::string t_err;

esim_status fail(esim_status st, const std::string& msg) {
    t_err = msg;
    return st;
}

esim_status cuda_fail(cudaError_t e, const char* where) {
    return fail(ESIM_ECUDA, std::string(where) + ": " + cudaGetErrorString(e));
}

#define ESIM_CUDA_TRY(expr, where)                        \
    do {                                                  \
        cudaError_t _e = (expr);                          \
        if (_e != cudaSuccess) return cuda_fail(_e, where); \
    } while (0)

template <typename T>
cudaError_t dev_alloc(T** p, size_t count) {
    *p = nullptr;
    if (count == 0) count = 1;
    return cudaMalloc((void**)p, sizeof(T) * count);
}

constexpr uint32_t kSegLen = 4096;         // probe sweeps: entries a block adds, an eighth of them each warp
constexpr uint32_t kProbeLongMin = 512;    // shortest row of a block; 1024/64, 2048/128, 1024/256 measured the same
// From this many edges on a level is no longer one row's latency: rows of up to 64 entries a lane, four
// gathers in flight.  Forward + reverse, L = 20, FP64, eight / four gathers at the rule's cap below the line
// and at 64 above it: skewed (Chung-Lu, mean degree 10, exponent 2.2) m = 3e6 809 / 736 us, 4.1e6 983 / 968,
// 6e6 1341 / 1289, 8e6 1766 / 1653, 1.2e7 2833 / 2397, 1.75e7 4053 / 3297; R-MAT n = 2^18 4.1e6 918 / 862,
// 8e6 1335 / 1218; random of mean degree 10 2e6 538 / 684, 4.1e6 880 / 939, 8e6 1540 / 1571, 1.75e7 3371 /
// 3301, of mean degree 40 3e6 684 / 707, 6e6 1006 / 1391, 8e6 1424 / 1816, 1.2e7 1908 / 1900.  The
// skewed graphs decide.  The cap above the line, four gathers, 32 / 64: skewed 4.1e6 912 / 968, 8e6
// 1629 / 1653, 1.75e7 3479 / 3297, random of mean degree 40 8e6 2987 / 1816.
constexpr int64_t kLongRowsFrom = 4000000;

// The longest row that one lane sums (SellRows, internal.h).  A lane's chain of gathers is most of
// a small level's time and a warp per row shortens it, as long as all warps of the level are on
// the chip at once: the smallest cap that leaves no more of them than that.  Forward, allocation and
// reverse at eps = 1e-4 in FP64, with caps of 32 / 16 / 8: random n = 2001, m = 16,009 174 / 160 / 138 us
// (877 warps at 8), n = 20,001, m = 160,009 209 / 189 / 275 (709 and 8854), m = 400,021
// 252 / 442 / 484 (16,303); skewed n = 20,001, m = 200,011 302 / 268 / 259 (4577), n = 50,001, m = 500,011
// 345 / 313 / 423 (5940 and 11,381), n = 100,003, m = 1,000,031 397 / 441 / 627 (11,446).
// Where 32 leaves many more warps than that and 64 clearly fewer, the warps are what takes the time:
// forward + reverse, L = 20, FP64 with 32 / 64: random n = 50,000, m = 2.5e6 1175 / 764 us (51,500
// and 2500 warps), n = 100,000, m = 3.9e6 1985 / 929, R-MAT n = 2^17, m = 3.75e6 937 / 739; but
// R-MAT n = 2^16, m = 1.5e6 468 / 505 (14,000), random n = 20,000, m = 1.9e6 525 / 690 (nearly all rows
// above 64: the few below it are the level's longest chains).
uint32_t sell_row_cap(int64_t n, const std::vector<uint32_t>& rp, int sm_count) {
    const int64_t resident = (int64_t)sm_count * 40;  // warps, at 48 registers a thread
    if ((int64_t)rp[n] >= kLongRowsFrom) return kLargeRowCap;
    static_assert(kSmallRowCap == 4 * kLeastRowCap && kLargeRowCap == 2 * kSmallRowCap, "a cap between would be left out");
    int64_t warps[4];
    for (int64_t& w : warps) w = (n + kSellWindow - 1) / kSellWindow * (kSellWindow / 32);
    for (int64_t r = 0; r < n; ++r) {  // one pass without branches; lengths are below kLongRowsFrom
        const uint32_t len = rp[r + 1] - rp[r];
        for (int i = 0; i < 4; ++i) {
            const uint32_t cap = kLeastRowCap << i;
            warps[i] += len > cap ? (len + 32 * cap - 1) / (32 * cap) : 0u;
        }
    }
    for (int i = 0; i < 3; ++i)
        if (warps[i] <= resident) return kLeastRowCap << i;
    return warps[2] > 4 * resident && 4 * warps[3] <= 3 * warps[2] ? kLargeRowCap : kSmallRowCap;
}

// Entries that a lane group of the batched sweeps adds one after another, at most: 64, so that a hub
// is not a level's longest chain; more on dense graphs, where cutting every row doubles the launches and
// only adds partial sums, but never so much that there are fewer than 8192 pieces of that length, about
// what the chip works on at once.  Sweeps of a query, 64 columns, forward + reverse, with 64 / 256:
// random n = 20,000, m = 3.9e6 4.18 / 2.64 ms; R-MAT n = 2^17, m = 3.75e6 (mean degree 28; five columns)
// 1.57 / 1.95, n = 3000, m = 9e5 with 64 / 128 0.92 / 1.04.
uint32_t batch_seg_len(int64_t n, int64_t m) {
    const int64_t most = std::min(4 * m / n, m / 8192);
    uint32_t len = 64;
    while (len < 4096 && 2 * (int64_t)len <= most) len *= 2;
    return len;
}

// A CSR's tables on the host.
struct CsrTables {
    std::vector<Segment> seg, bseg, pieces;
    std::vector<int32_t> long_rows, long_first, blong_rows, blong_first;
    std::vector<uint32_t> off, pos;
};

CsrTables plan_csr(int64_t n, const std::vector<uint32_t>& rp, const std::vector<uint32_t>& uses_rp, int sm_count,
                   DevCsr& d) {
    CsrTables t;
    const int64_t m = (int64_t)rp[n];
    d.long_min = kProbeLongMin;
    d.seg_len = kSegLen;
    d.bseg_len = batch_seg_len(n, m);
    d.sell.row_cap = sell_row_cap(n, rp, sm_count);
    d.sell.few_in_flight = m >= kLongRowsFrom;
    auto cut = [&](int64_t r, uint32_t len, std::vector<Segment>& sg) {
        const uint32_t first = (uint32_t)sg.size(), end = rp[r + 1];
        for (uint32_t s = rp[r]; s < end; s += len) sg.push_back(Segment{(int32_t)r, s, std::min(end, s + len), first});
    };
    const uint32_t cap = d.sell.row_cap, shortest = std::min(d.long_min, d.bseg_len);
    int64_t wide = 0, longer = 0;  // rows above the cap, and those of the other tables
    for (int64_t r = 0; r < n; ++r) {
        const uint32_t len = rp[r + 1] - rp[r];
        wide += len > cap;
        longer += len >= shortest;
    }
    t.pieces.reserve((size_t)(wide + m / (32 * (int64_t)cap)));
    if (wide)
        for (int64_t r = 0; r < n; ++r)
            if (rp[r + 1] - rp[r] > cap) cut(r, 32 * cap, t.pieces);
    if (longer)
        for (int64_t r = 0; r < n; ++r) {
            const uint32_t len = rp[r + 1] - rp[r];
            if (len < shortest) continue;
            if (len > kSegLen) {
                t.long_rows.push_back((int32_t)r);
                t.long_first.push_back((int32_t)t.seg.size());
            }
            if (len >= d.long_min) cut(r, kSegLen, t.seg);
            if (len >= d.bseg_len) {
                t.blong_rows.push_back((int32_t)r);
                t.blong_first.push_back((int32_t)t.bseg.size());
                cut(r, d.bseg_len, t.bseg);
            }
        }
    t.long_first.push_back((int32_t)t.seg.size());
    t.blong_first.push_back((int32_t)t.bseg.size());
    d.nseg = (int64_t)t.seg.size();
    d.nlong = (int64_t)t.long_rows.size();
    d.bnseg = (int64_t)t.bseg.size();
    d.bnlong = (int64_t)t.blong_rows.size();
    plan_sell(n, rp, t.pieces, uses_rp, d.sell, t.off, t.pos);
    return t;
}

// Up to here a CSR's entries go with the small tables in one copy: m = 20,000 0.281 -> 0.263 ms a load, 80,001
// 0.547 and 0.546; above, the copy through the stage costs as much as the calls (156,071 0.794 -> 0.803).
constexpr size_t kStagedEdges = 1 << 16;

size_t topk_stage_offset(int64_t n) { return (topk_workspace_bytes(n) + 255) / 256 * 256; }

// The graph's device memory: one allocation, one copy of the small tables, and what the device
// fills, both CSRs' slices in one launch each: a load makes few calls of a size-independent cost.  With
// allocations, copies and waits per table, 1/din and its inverse made on the host, and repeated in-edges
// looked up by a mark per node, the sliced rows had made it slower: Chung-Lu n = 2000, m = 20,000 0.40 ms
// (0.30 without them, 0.26 now), n = 8000, m = 80,001 0.89 (0.59, 0.55), n = 100,003, m = 1,000,003 7.4
// (6.3, 5.9); random n = 2863, m = 22,047 0.35 (0.27, 0.28).
esim_status upload_graph(Graph& g, const std::vector<uint32_t>& in_rp, const int32_t* in_col,
                         const std::vector<uint32_t>& out_rp, const int32_t* out_col) {
    const size_t n = (size_t)g.n, m = (size_t)g.m;
    const CsrTables tables[2] = {plan_csr(g.n, in_rp, out_rp, g.sm_count, g.in), plan_csr(g.n, out_rp, in_rp, g.sm_count, g.out)};
    struct Part {
        void** to;
        size_t at;
        const void* from;
        size_t bytes;
    };
    std::vector<Part> parts;
    size_t bytes = 0;
    auto take = [&](auto*& to, size_t count, const void* from = nullptr) {
        const size_t b = sizeof(*to) * count;
        parts.push_back({(void**)&to, bytes, from, b});
        bytes += (b + 255) / 256 * 256;
    };
    DevCsr* const csr[2] = {&g.in, &g.out};
    for (int i = 0; i < 2; ++i) {
        const CsrTables& t = tables[i];
        DevCsr& d = *csr[i];
        take(d.seg, t.seg.size(), t.seg.data());
        take(d.long_rows, t.long_rows.size(), t.long_rows.data());
        take(d.long_first, t.long_first.size(), t.long_first.data());
        take(d.bseg, t.bseg.size(), t.bseg.data());
        take(d.blong_rows, t.blong_rows.size(), t.blong_rows.data());
        take(d.blong_first, t.blong_first.size(), t.blong_first.data());
        take(d.sell.off, t.off.size(), t.off.data());
        take(d.sell.piece, t.pieces.size(), t.pieces.data());
        if (!t.pos.empty()) take(d.sell.pos, n, t.pos.data());
    }
    take(g.in.rp, n + 1, in_rp.data());
    take(g.out.rp, n + 1, out_rp.data());
    const bool stage_cols = m <= kStagedEdges;
    const int32_t* const cols[2] = {in_col, out_col};
    for (int i = 0; i < 2; ++i)
        if (stage_cols) take(csr[i]->col, m, cols[i]);
    const size_t staged = bytes;
    for (int i = 0; i < 2; ++i) {
        if (!stage_cols) take(csr[i]->col, m);
        take(csr[i]->sell.rows, 32 * (size_t)csr[i]->sell.nslices);
        take(csr[i]->sell.col, 32 * (size_t)tables[i].off.back());
    }
    take(g.in.info, n);                  // filled on the device, as the next three (launch_walk_table)
    take(g.in.walk, std::max(m, n));     // the tail past m is never a position
    take(g.inv_din, n);
    take(g.din_magic, n);
    take(g.status, 1);
    take(g.sample_taken, kSampleSlots);
    char* partial = nullptr;
    char* topk = nullptr;
    take(partial, scratch_bytes(g));
    take(g.scan_part, (size_t)allocate_blocks(g.n));
    take(g.norm_part, 2 * (size_t)allocate_blocks(g.n));
    take(topk, topk_stage_offset(g.n) + (sizeof(double) + sizeof(int32_t)) * kTopkMax);
    if (cudaMalloc((void**)&g.memory, bytes) != cudaSuccess) {
        cudaGetLastError();
        g.memory = nullptr;
        return fail(ESIM_ENOMEM, "cudaMalloc(graph tables of " + std::to_string(bytes) + " bytes)");
    }
    for (const Part& p : parts) *p.to = g.memory + p.at;
    g.partial = partial;
    g.topk_ws = topk;
    const std::unique_ptr<char[]> stage(new char[staged]);
    for (const Part& p : parts)
        if (p.from && p.bytes) memcpy(stage.get() + p.at, p.from, p.bytes);
    const cudaStream_t stream = g.stream;
    ESIM_CUDA_TRY(cudaMemcpyAsync(g.memory, stage.get(), staged, cudaMemcpyHostToDevice, stream), "upload graph tables");
    for (int i = 0; i < 2; ++i)
        if (!stage_cols)
            ESIM_CUDA_TRY(cudaMemcpyAsync(csr[i]->col, cols[i], sizeof(int32_t) * m, cudaMemcpyHostToDevice, stream),
                          "upload col");
    ESIM_CUDA_TRY(fill_sell(g.n, g.in, g.out, stream), "sliced rows");
    ESIM_CUDA_TRY(launch_walk_table(g), "walk table");
    ESIM_CUDA_TRY(cudaMemsetAsync(g.status, 0, sizeof(Status), stream), "reset status");
    ESIM_CUDA_TRY(cudaStreamSynchronize(stream), "graph tables");  // the host tables are this call's
    return ESIM_OK;
}

// The scratch of work on one stream (call_counts), and the allocation's and the scans' tile sums.
bool alloc_scratch(const Graph& g, void** partial, unsigned long long** part, double** norm) {
    const size_t nb = (size_t)allocate_blocks(g.n);
    return cudaMalloc(partial, scratch_bytes(g)) == cudaSuccess && dev_alloc(part, nb) == cudaSuccess &&
           dev_alloc(norm, 2 * nb) == cudaSuccess;
}

void free_a3workers(Graph& g) {
    for (auto& wk : g.a3workers) {
        if (wk.stream) {
            cudaStreamSynchronize(wk.stream);
            cudaStreamDestroy(wk.stream);
        }
        cudaFree(wk.ws);
        cudaFree(wk.partial);
        cudaFree(wk.scan_part);
        cudaFree(wk.norm_part);
    }
    g.a3workers.clear();
    g.a3worker_ws_bytes = 0;
}

// Up to `extra` workers beside the query's stream; returns how many exist (fewer when
// the device cannot hold more: the computation then uses fewer, never fails for it).
int ensure_a3workers(Graph& g, int extra) {
    const size_t need = alg3_workspace_bytes(g);
    if (g.a3worker_ws_bytes < need) free_a3workers(g);
    while ((int)g.a3workers.size() < extra) {
        Graph::A3Worker wk;
        const bool ok = cudaStreamCreateWithFlags(&wk.stream, cudaStreamNonBlocking) == cudaSuccess &&
                        cudaMalloc(&wk.ws, need) == cudaSuccess &&
                        alloc_scratch(g, &wk.partial, &wk.scan_part, &wk.norm_part);
        if (!ok) {
            cudaGetLastError();
            if (wk.stream) cudaStreamDestroy(wk.stream);
            cudaFree(wk.ws);
            cudaFree(wk.partial);
            cudaFree(wk.scan_part);
            cudaFree(wk.norm_part);
            break;
        }
        g.a3workers.push_back(wk);
        g.a3worker_ws_bytes = need;
    }
    return std::min<int>(extra, (int)g.a3workers.size());
}

void release(Graph& g) {
    cudaSetDevice(g.device);
    // no work of this handle may still use its buffers: its own streams drain first (a
    // caller's stream set by esim_set_stream is the caller's to drain)
    if (g.own_stream) cudaStreamSynchronize(g.own_stream);
    if (g.side_stream) cudaStreamSynchronize(g.side_stream);
    free_a3workers(g);
    cudaFree(g.memory);
    for (auto& ev : g.sample_ev)
        if (ev) cudaEventDestroy(ev);
    if (g.status_host) cudaFreeHost(g.status_host);
    cudaFree(g.ws);
    cudaFree(g.bws);
    cudaFree(g.a3ws);
    cudaFree(g.a3pws);
    cudaFree(g.zstage);
    for (auto& ev : g.ev)
        if (ev) cudaEventDestroy(ev);
    if (g.own_stream) cudaStreamDestroy(g.own_stream);
    if (g.side_stream) cudaStreamDestroy(g.side_stream);
    for (auto& ev : g.side_ev)
        if (ev) cudaEventDestroy(ev);
    for (auto& ev : g.side_tev)
        if (ev) cudaEventDestroy(ev);
    g = Graph{};
}

bool valid_c_eps(double c, double eps) { return c > 0.0 && c < 1.0 && eps > 0.0 && eps < 1.0; }

double kappa_of(const Graph& g, double c) {
    if (g.kappa > 0.0) return g.kappa;
    const double a = 1.0 - sqrt(c);
    return 6.0 / (a * a * a * a);
}

// Query workspace (one device arena per graph handle, grown on demand).  The
// FP64 form uses hist/xa/xb; the FP32c form uses hist32/xa32/xb32 and the
// two-float buffers w/sa2/sb2.  Every buffer starts on a 256-byte boundary.
struct Ws {
    double* hist;      // (L+1) n  FP64 history
    double* xa;        // n        forward x, then reverse ping-pong (FP64)
    double* xb;        // n
    float* hist32;     // (L+1) n  FP32 history
    float* xa32;       // n
    float* xb32;       // n
    float2* w2;        // n        D^/a as two-floats
    float2* sa2;       // n        reverse ping-pong (two-float)
    float2* sb2;       // n
    double* pi;        // n
    uint64_t* R;       // n
    uint64_t* off;     // n+1
    uint64_t* nonmeet; // n
    double* dhat;      // n
    double* s;         // n
    uint8_t* depth;    // n  Algorithm 3 depth per node (0: Algorithm 2)
    double* zsum;      // n  Algorithm 3: sum of the exact Z_l(k)
    uint8_t* cand;     // n  Algorithm 3: 0 other node, 1 candidate walked after the plan, 2 early candidate
    uint64_t* R2;      // n  R of the side sampler's nodes, then of the other candidates
    uint64_t* off2;    // n+1  offsets of the side sampler's walks (read by the side stream)
    uint64_t* offc;    // n+1  offsets of the candidates' walks
    uint64_t* nm2;     // n  counts of the other nodes
    int32_t* cand_ids; // 4096
    PlanEntry* plan;   // 4096  the cost model's plan, staged for the scatter
    // sparse linearization (FP64): rolling pi^l, the running pi, the kept entries
    double* lev;       // n
    double* pirun;     // n
    SparseHist sh;     // cap entries, L+2 level ends
};

size_t round256(size_t b) { return (b + 255) / 256 * 256; }

// Lay out the arena at `base` (or only measure it when base is null); returns bytes.
// Capacity of the sparse history: fewer than 1/theta entries exceed theta, because
// the pi^l(k) over all levels and nodes sum to at most 1 (pigeonhole, Section 3.2);
// never more than the dense (L+1) n.
uint64_t sparse_capacity(int64_t n, int32_t L, double theta) {
    const double bound = floor(1.000001 / theta) + 1.0;
    const double dense = (double)(L + 1) * (double)n;
    return (uint64_t)(bound < dense ? bound : dense);
}

size_t ws_layout(int64_t n_, int32_t L, int precision, char* base, Ws* w, uint64_t sparse_cap = 0) {
    const size_t n = (size_t)n_;
    size_t o = 0;
    auto take = [&](size_t bytes) -> char* {
        char* p = base ? base + o : nullptr;
        o += round256(bytes);
        return p;
    };
    Ws t{};
    if (precision == 0 && sparse_cap > 0) {  // the entries themselves go last (see below)
        t.lev = (double*)take(8 * n);
        t.pirun = (double*)take(8 * n);
        t.xa = (double*)take(8 * n);
        t.xb = (double*)take(8 * n);
    } else if (precision == 0) {
        t.hist = (double*)take(8 * n * (size_t)(L + 1));
        t.xa = (double*)take(8 * n);
        t.xb = (double*)take(8 * n);
    } else {
        t.hist32 = (float*)take(4 * n * (size_t)(L + 1));
        t.xa32 = (float*)take(4 * n);
        t.xb32 = (float*)take(4 * n);
        t.w2 = (float2*)take(8 * n);
        t.sa2 = (float2*)take(8 * n);
        t.sb2 = (float2*)take(8 * n);
        t.xa = (double*)t.sa2;  // FP64 scratch for step calls that need one (aliases sa2)
        t.xb = (double*)t.sb2;
    }
    t.pi = (double*)take(8 * n);
    t.R = (uint64_t*)take(8 * n);
    t.off = (uint64_t*)take(8 * (n + 1));
    t.nonmeet = (uint64_t*)take(8 * n);
    t.dhat = (double*)take(8 * n);
    t.s = (double*)take(8 * n);
    t.depth = (uint8_t*)take(n);
    t.zsum = (double*)take(8 * n);
    t.cand = (uint8_t*)take(n);
    t.R2 = (uint64_t*)take(8 * n);
    t.off2 = (uint64_t*)take(8 * (n + 1));
    t.offc = (uint64_t*)take(8 * (n + 1));
    t.nm2 = (uint64_t*)take(8 * n);
    t.cand_ids = (int32_t*)take(4 * 4096);
    t.plan = (PlanEntry*)take(sizeof(PlanEntry) * 4096);
    if (precision == 0 && sparse_cap > 0) {
        // last, so that the layout for a smaller capacity is a prefix of this one
        t.sh.lvl = (uint64_t*)take(8 * (size_t)(L + 2));
        t.sh.idx = (int32_t*)take(4 * (size_t)sparse_cap);
        t.sh.val = (double*)take(8 * (size_t)sparse_cap);
        t.sh.cap = sparse_cap;
    }
    if (w) *w = t;
    return o;
}

esim_status ensure_ws(Graph& g, int32_t L, int precision, Ws& w, uint64_t sparse_cap = 0) {
    const size_t need = ws_layout(g.n, L, precision, nullptr, nullptr, sparse_cap);
    g.last_ws_bytes = need;
    if (need > g.ws_bytes) {
        cudaStreamSynchronize(g.stream);
        cudaFree(g.ws);
        g.ws = nullptr;
        g.ws_bytes = 0;
        if (cudaMalloc(&g.ws, need) != cudaSuccess) {
            cudaGetLastError();
            return fail(ESIM_ENOMEM, "cudaMalloc(query workspace of " + std::to_string(need) + " bytes)");
        }
        g.ws_bytes = need;
    }
    ws_layout(g.n, L, precision, (char*)g.ws, &w, sparse_cap);
    return ESIM_OK;
}

esim_status check_graph(const esim_graph* h) {
    if (!h) return fail(ESIM_EINVAL, "graph handle is NULL");
    return ESIM_OK;
}

esim_status ensure_a3ws(Graph& g) {
    const size_t need = alg3_workspace_bytes(g);
    if (g.a3ws && g.a3ws_bytes >= need) return ESIM_OK;
    cudaStreamSynchronize(g.stream);
    cudaFree(g.a3ws);
    g.a3ws = nullptr;
    g.a3ws_bytes = 0;
    g.a3ws_clean = 0;
    if (cudaMalloc(&g.a3ws, need) != cudaSuccess) {
        cudaGetLastError();
        return fail(ESIM_ENOMEM, "cudaMalloc(Algorithm 3 workspace of " + std::to_string(need) + " bytes)");
    }
    g.a3ws_bytes = need;
    return ESIM_OK;
}

// Algorithm 3's depth choice under option alg3_rule = 1.  The paper grows l(k) until the
// explored edges reach 2 R(k) / sqrt(c), the walk work they replace.  Here the
// exploitation is done with dense sweeps, so the depth d of node k minimises an
// estimate of the GPU work, in walk pair-steps of the sampler:
//   walks      R_d (d + 1/(1-c)),  R_d = max(1, ceil(v c^(2d)))  (v = R_b pi(k)^2)
//   Lemma 5    2d-1 single-vector sweeps of m+n entries (h_1..h_d and the P~ sweeps);
//              sum_{i=1}^{d-4} |supp h_i| (d-i) probe column-sweeps for the deeper probe
//              levels; the last two probe levels (i = d-2 and d-3, two and three steps)
//              run one warp per node over its two- and three-hop neighbourhood and dense
//              probes only for the nodes too large for that, charged as
//              w_last (d-i) |supp h_i| column-sweeps; and the launches;
// d = 0 is Algorithm 2 alone.  The weights (options alg3_w_sweep, alg3_w_probe,
// alg3_w_launch, alg3_w_last: pair-steps per entry of a single sweep, per entry and
// column of a probe sweep, per launch, and the last level's share of a dense probe) are
// calibrated by timing whole queries on GB300.
double alg3_cost(int d, double v, double c, const uint64_t* supp, int64_t n, int64_t m, double w_sweep,
                 double w_probe, double w_launch, double w_last) {
    double r = d == 0 ? ceil(v) : ceil(v * pow(c, (double)(2 * d)));
    if (r < 1.0) r = 1.0;
    double cost = r * ((double)d + 1.0 / (1.0 - c));
    if (d > 0) {
        const double edges = (double)(m + n);
        uint64_t probe = 0, launches = 3 * (uint64_t)(2 * d - 1);
        for (int i = 1; i <= d - 4; ++i) {
            probe += supp[i] * (uint64_t)(d - i);
            launches += (supp[i] + 31) / 32 * (uint64_t)(3 * (d - i) + 2);
        }
        double last = 0.0;
        for (int i = std::max(1, d - 3); i <= d - 2; ++i) {
            last += w_last * ((double)(d - i) * (double)supp[i]);
            launches += 2;
        }
        cost += w_sweep * edges * (double)(2 * d - 1);
        cost += w_probe * edges * ((double)probe + last);
        cost += w_launch * (double)launches;
    }
    return cost;
}

// The depth of least estimated work, 0..max_depth (the first on ties).
int alg3_depth(double v, double c, const uint64_t* supp, int max_depth, int64_t n, int64_t m, double w_sweep,
               double w_probe, double w_launch, double w_last) {
    int d = 0;
    double best = alg3_cost(0, v, c, supp, n, m, w_sweep, w_probe, w_launch, w_last);
    for (int dd = 1; dd <= max_depth; ++dd) {
        const double cost = alg3_cost(dd, v, c, supp, n, m, w_sweep, w_probe, w_launch, w_last);
        if (cost < best) {
            best = cost;
            d = dd;
        }
    }
    return d;
}

// Algorithm 3 for the heaviest nodes (by pi, at most alg3_max_nodes, with din >= 2
// and an Algorithm 2 count of at least alg3_min_pairs): the depth by alg3_cost (at
// most alg3_max_depth), exact Z_1..Z_d (Lemma 5) on the GPU, and the pair count
// max(1, ceil(R_b pi(k)^2 c^(2d))) (pi(k) for the basic allocation): the tail
// estimator's variance and range are c^(2d) and c^d of Algorithm 2's.  Nodes with
// din <= 1 already got no pairs from the allocation.  Then the offsets are rescanned.
// The sampler on the side stream after the work queued so far on g.stream: offsets off,
// counts nm2, pair-steps to the status block's side counter; at most alg3_overlap
// blocks per SM, leaving room for the planning's kernels.  Records side_ev[1] at its end.
esim_status launch_side_walks(Graph& g, const Ws& w, const uint64_t* off, double c, uint64_t seed,
                              const uint8_t* depth) {
    ESIM_CUDA_TRY(cudaEventRecord(g.side_ev[0], g.stream), "record");
    ESIM_CUDA_TRY(cudaStreamWaitEvent(g.side_stream, g.side_ev[0], 0), "side wait");
    Graph view = g;
    view.stream = g.side_stream;
    view.sample_block_cap = g.alg3_overlap;
    if (g.timing) {
        for (auto& ev : g.side_tev)
            if (!ev) ESIM_CUDA_TRY(cudaEventCreate(&ev), "cudaEventCreate");
        cudaEventRecord(g.side_tev[0], g.side_stream);
    }
    ESIM_CUDA_TRY(launch_sample(view, off, c, seed, w.nm2, (uint64_t*)&g.status->pair_steps_side, depth,
                                &g.status->taken[1]),
                  "side walk pairs");
    if (g.timing) cudaEventRecord(g.side_tev[1], g.side_stream);
    ESIM_CUDA_TRY(cudaEventRecord(g.side_ev[1], g.side_stream), "record");
    return ESIM_OK;
}

// Starts, on the side stream, the walks of every node that is not an Algorithm 3
// candidate and of the early candidates (cand = 2), in one launch: their R(k) and depths
// are final, and the walk spec keys a pair by (seed, k, r), so splitting the nodes
// between sampler launches changes no count.  One launch, not one per group, so that
// the planning's kernels keep their share of every SM.
esim_status start_side_walks(Graph& g, const Ws& w, double c, uint64_t seed, int* launches) {
    ESIM_CUDA_TRY(launch_mask_R(g, w.R, w.cand, (1u << 0) | (1u << 2), w.R2), "side nodes' R");
    const int64_t nb = allocate_blocks(g.n);
    ESIM_CUDA_TRY(launch_scan_R(g, g.n, w.R2, w.off2, g.scan_part, g.norm_part + nb, scan_ticket(g), false), "side nodes' scan");
    esim_status st = launch_side_walks(g, w, w.off2, c, seed, w.depth);
    if (st != ESIM_OK) return st;
    *launches += 4;
    return ESIM_OK;
}

esim_status ensure_a3pws(Graph& g) {
    if (!alg3_paper_fits(g.n))
        return fail(ESIM_ENOTSUP, "the paper's Algorithm 3 depth rule keeps n x n support bit sets; n = " +
                                      std::to_string(g.n) + " is above its 4 GiB budget (option alg3_rule = 1 "
                                      "chooses depths by the cost model)");
    if (g.a3pws) return ESIM_OK;
    size_t need = 0;
    for (bool least : {false, true}) {  // the levels that are not kept are made twice
        need = alg3_paper_bytes(g.n, least);
        if (cudaMalloc(&g.a3pws, need) == cudaSuccess) {
            g.a3pws_bytes = need;
            return ESIM_OK;
        }
        cudaGetLastError();
        g.a3pws = nullptr;
    }
    return fail(ESIM_ENOMEM, "cudaMalloc(Algorithm 3 depth-rule workspace of " + std::to_string(need) + " bytes)");
}

// zsum(k) = sum_{l <= depth(k)} Z_l(k) for the nodes of the given depths (every other
// entry 0): Z_1 = c/din(k) for every node of depth 1 in depth_dev, the closed form of
// depth 2 (alg3_paper.cu) for the nodes in d2, and Z_1..Z_d from alg3_first_meeting, one
// node at a time, for the nodes in deep and for the depth-2 nodes whose two-hop
// neighbourhood is too large for the closed form's table.  Synchronises g.stream.
esim_status alg3_zsums_of(Graph& g, const uint8_t* depth_dev, const std::vector<int32_t>& d2,
                          std::vector<std::pair<int32_t, int>> deep, double c, double* zsum, int* launches) {
    ESIM_CUDA_TRY(cudaMemsetAsync(zsum, 0, sizeof(double) * (size_t)g.n, g.stream), "reset zsum");
    ESIM_CUDA_TRY(alg3_paper_z1(g, depth_dev, c, zsum), "Algorithm 3 Z_1");
    *launches += 1;
    if (!d2.empty()) {
        const int cnt = (int)d2.size();
        const size_t need = round256(4 * d2.size()) + 8 * d2.size();  // ids, then the gathered values
        if (g.zstage_bytes < need) {
            cudaStreamSynchronize(g.stream);
            cudaFree(g.zstage);
            g.zstage = nullptr;
            g.zstage_bytes = 0;
            const size_t want = round256(4 * (size_t)g.n) + 8 * (size_t)g.n;
            if (cudaMalloc(&g.zstage, want) != cudaSuccess) {
                cudaGetLastError();
                return fail(ESIM_ENOMEM, "cudaMalloc(Algorithm 3 staging of " + std::to_string(want) + " bytes)");
            }
            g.zstage_bytes = want;
        }
        int32_t* stage_ids = (int32_t*)g.zstage;
        double* stage_vals = (double*)((char*)g.zstage + round256(4 * d2.size()));
        std::vector<double> v2((size_t)cnt);
        ESIM_CUDA_TRY(cudaMemcpyAsync(stage_ids, d2.data(), sizeof(int32_t) * d2.size(), cudaMemcpyHostToDevice,
                                      g.stream),
                      "upload depth-2 nodes");
        ESIM_CUDA_TRY(alg3_paper_z2(g, stage_ids, cnt, c, zsum), "Algorithm 3 Z_1 + Z_2");
        ESIM_CUDA_TRY(alg3_gather_f64(g, stage_ids, cnt, zsum, stage_vals), "gather depth-2 terms");
        ESIM_CUDA_TRY(cudaMemcpyAsync(v2.data(), stage_vals, sizeof(double) * d2.size(), cudaMemcpyDeviceToHost,
                                      g.stream),
                      "copy depth-2 terms");
        ESIM_CUDA_TRY(cudaStreamSynchronize(g.stream), "Algorithm 3 depth-2 terms");  // d2 and v2 are locals
        *launches += 2;
        for (int i = 0; i < cnt; ++i)
            if (v2[(size_t)i] != v2[(size_t)i]) deep.emplace_back(d2[(size_t)i], 2);  // NaN: too large
    }
    if (!deep.empty()) {
        esim_status a3 = ensure_a3ws(g);
        if (a3 != ESIM_OK) return a3;
        // Each node's Lemma 5 computation waits on the host between its levels (the next
        // level's probe count); workers on their own streams take nodes from a shared
        // counter, so one node's waits leave the GPU to the others.  A node's result does
        // not depend on the worker that computes it.
        const int want = std::max(1, std::min<int>(g.alg3_workers, (int)deep.size()));
        const int nw = 1 + (want > 1 ? ensure_a3workers(g, want - 1) : 0);
        std::vector<double> zs(deep.size());
        std::atomic<size_t> next{0};
        std::vector<cudaError_t> errs((size_t)nw, cudaSuccess);
        std::vector<int> counts((size_t)nw, 0);
        auto run = [&](int wi) {
            Graph view = g;
            void* ws = g.a3ws;
            int* clean = &g.a3ws_clean;
            if (wi > 0) {
                Graph::A3Worker& wk = g.a3workers[(size_t)wi - 1];
                if ((errs[(size_t)wi] = cudaSetDevice(g.device)) != cudaSuccess) return;
                view.stream = wk.stream;
                view.partial = wk.partial;
                view.scan_part = wk.scan_part;
                view.norm_part = wk.norm_part;
                ws = wk.ws;
                clean = &wk.clean;
            }
            for (;;) {
                const size_t i = next.fetch_add(1);
                if (i >= deep.size()) return;
                const int d = deep[i].second;
                double z[kAlg3MaxDepth] = {};
                const cudaError_t e = alg3_first_meeting(view, deep[i].first, d, c, ws, clean, z,
                                                         &counts[(size_t)wi]);
                if (e != cudaSuccess) {
                    errs[(size_t)wi] = e;
                    next.store(deep.size());  // the others stop after their current node
                    return;
                }
                double sum = 0.0;
                for (int j = 0; j < d; ++j) sum += z[j];
                zs[i] = sum;
            }
        };
        std::vector<std::thread> threads;
        for (int wi = 1; wi < nw; ++wi) threads.emplace_back(run, wi);
        run(0);
        for (auto& t : threads) t.join();
        for (int wi = 0; wi < nw; ++wi) {
            ESIM_CUDA_TRY(errs[(size_t)wi], "Algorithm 3 first meetings");
            *launches += counts[(size_t)wi];
        }
        for (size_t i = 0; i < deep.size(); ++i)
            ESIM_CUDA_TRY(cudaMemcpyAsync(zsum + deep[i].first, &zs[i], sizeof(double), cudaMemcpyHostToDevice,
                                          g.stream),
                          "set zsum");
        ESIM_CUDA_TRY(cudaStreamSynchronize(g.stream), "Algorithm 3 plan");  // zs is a local
    }
    return ESIM_OK;
}

// The same from a device depth array alone (every node): the host reads it back and
// lists the nodes.  Returns the number of nodes with depth >= 1 in *used.
esim_status alg3_zsums(Graph& g, const uint8_t* depth_dev, double c, double* zsum, int* launches, int* used_out) {
    std::vector<uint8_t> depth((size_t)g.n);
    ESIM_CUDA_TRY(cudaMemcpyAsync(depth.data(), depth_dev, (size_t)g.n, cudaMemcpyDeviceToHost, g.stream), "copy depth");
    ESIM_CUDA_TRY(cudaStreamSynchronize(g.stream), "Algorithm 3 depths");
    std::vector<int32_t> d2;
    std::vector<std::pair<int32_t, int>> deep;
    int used = 0;
    for (int64_t k = 0; k < g.n; ++k) {
        const int d = depth[(size_t)k];
        if (d == 0) continue;
        ++used;
        if (d == 2) d2.push_back((int32_t)k);
        else if (d > 2) deep.emplace_back((int32_t)k, d);
    }
    *used_out = used;
    return alg3_zsums_of(g, depth_dev, d2, std::move(deep), c, zsum, launches);
}

// Algorithm 3 with the paper's adaptive depth: every node with R(k) > 0 (din >= 2; the
// allocation gave the others none) explores until its explored edges reach
// 2 R(k)/sqrt(c), at most alg3_max_depth levels (alg3_paper.cu); it keeps its R(k)
// pairs, which move without the continuation draw for depth(k) steps; then the sums of
// its exact Z (alg3_zsums).
esim_status plan_alg3_paper(Graph& g, const Ws& w, double c, int* launches, uint64_t seed, bool* side) {
    esim_status a3 = ensure_a3pws(g);
    if (a3 != ESIM_OK) return a3;
    ESIM_CUDA_TRY(alg3_paper_depths(g, w.R, c, g.alg3_max_depth, g.a3pws, g.a3pws_bytes, w.depth, launches),
                  "Algorithm 3 depths (explored edges)");
    // Every node's walks are final now (the allocation's R(k) and offsets, the depths):
    // with a side stream they all run there while the first-meeting sums are computed,
    // and the main stream's candidate launch is empty (cand = 0 everywhere).
    if (g.side_stream && g.alg3_overlap > 0) {
        ESIM_CUDA_TRY(cudaMemsetAsync(w.cand, 0, (size_t)g.n, g.stream), "reset candidates");
        esim_status st = launch_side_walks(g, w, w.off, c, seed, w.depth);
        if (st != ESIM_OK) return st;
        g.side_candidates = 0;
        *side = true;
        *launches += 1;
    }
    int used = 0;
    a3 = alg3_zsums(g, w.depth, c, w.zsum, launches, &used);
    if (a3 != ESIM_OK) return a3;
    g.last_alg3_nodes = used;
    return ESIM_OK;
}

esim_status plan_alg3(Graph& g, const Ws& w, double c, double R_b, int* launches, uint64_t seed, bool* side) {
    if (g.has_duplicates) return fail(ESIM_ENOTSUP, "Algorithm 3 needs a graph without repeated in-edges");
    *side = false;
    if (g.alg3_rule == 0) return plan_alg3_paper(g, w, c, launches, seed, side);
    esim_status a3 = ensure_a3ws(g);
    if (a3 != ESIM_OK) return a3;
    ESIM_CUDA_TRY(cudaMemsetAsync(w.depth, 0, (size_t)g.n, g.stream), "reset depth");
    const int K = (int)std::min<int64_t>(g.alg3_max_nodes, g.n);
    char* stage = (char*)g.topk_ws + topk_stage_offset(g.n);
    double* vals_d = (double*)stage;
    int32_t* ids_d = (int32_t*)(stage + sizeof(double) * kTopkMax);
    ESIM_CUDA_TRY(launch_topk(g, w.pi, -1, K, ids_d, vals_d, g.topk_ws), "Algorithm 3 node selection");
    *launches += 2;
    std::vector<int32_t> ids((size_t)K);
    std::vector<double> pis((size_t)K);
    ESIM_CUDA_TRY(cudaMemcpyAsync(ids.data(), ids_d, sizeof(int32_t) * K, cudaMemcpyDeviceToHost, g.stream), "copy ids");
    ESIM_CUDA_TRY(cudaMemcpyAsync(pis.data(), vals_d, sizeof(double) * K, cudaMemcpyDeviceToHost, g.stream), "copy pi");
    ESIM_CUDA_TRY(cudaStreamSynchronize(g.stream), "Algorithm 3 node selection");
    const std::vector<uint32_t>& din = *g.din_host;
    // candidates: the heaviest nodes with din >= 2 and enough Algorithm 2 pairs
    std::vector<int32_t> cand;
    std::vector<double> cand_v;
    for (int i = 0; i < K; ++i) {
        const int32_t kk = ids[i];
        const double p = pis[i];
        if (kk < 0 || !(p > 0.0)) break;
        if (din[kk] < 2) continue;
        const double v = g.alloc_mode == 0 ? R_b * (p * p) : R_b * p;
        double r0 = ceil(v);
        if (r0 < 1.0) r0 = 1.0;
        if (r0 < g.alg3_min_pairs) continue;
        cand.push_back(kk);
        cand_v.push_back(v);
    }
    // The budget applies to the pairs actually drawn: drop the verdict on the
    // Algorithm 2 counts (no other error can be raised before the walks); the side
    // sampler judges the other nodes' pairs and the rescan below all of them.
    ESIM_CUDA_TRY(cudaMemsetAsync((char*)g.status + offsetof(Status, err), 0, sizeof(int), g.stream), "reset budget");
    g.side_candidates = 0;
    *side = !cand.empty() && g.side_stream && g.alg3_overlap > 0;
    if (*side) {  // cand = 1 for the candidates (2 for the early ones below)
        ESIM_CUDA_TRY(cudaMemsetAsync(w.cand, 0, (size_t)g.n, g.stream), "reset candidates");
        ESIM_CUDA_TRY(cudaMemcpyAsync(w.cand_ids, cand.data(), sizeof(int32_t) * cand.size(), cudaMemcpyHostToDevice,
                                      g.stream),
                      "upload candidates");
        ESIM_CUDA_TRY(launch_mark(g, w.cand_ids, (int)cand.size(), w.cand), "mark candidates");
        *launches += 1;
    }
    const int levels = std::max(0, g.alg3_max_depth - 2);
    std::vector<uint64_t> supps(cand.size() * (kAlg3MaxDepth + 1), 0);
    if (!cand.empty())
        ESIM_CUDA_TRY(alg3_supports(g, cand.data(), (int)cand.size(), levels, g.a3ws, supps.data(), launches),
                      "Algorithm 3 supports");
    // The cost model picks each depth from the supports alone, so every plan is final
    // before any first-meeting term is computed: R(k) and depth(k) go to the device at
    // once, and the walks of the other nodes and of the candidates with at least
    // alg3_early_pairs pairs start on the side stream while the terms are computed.
    std::vector<PlanEntry> plan;
    std::vector<int32_t> d2;
    std::vector<std::pair<int32_t, int>> deep;
    int used = 0, n_early = 0;
    for (size_t ci = 0; ci < cand.size(); ++ci) {
        const int32_t kk = cand[ci];
        const double v = cand_v[ci];
        const uint64_t* supp = supps.data() + ci * (kAlg3MaxDepth + 1);
        const int d = alg3_depth(v, c, supp, g.alg3_max_depth, g.n, g.m, g.alg3_w_sweep, g.alg3_w_probe,
                                 g.alg3_w_launch, g.alg3_w_last);
        double r = d >= 1 ? ceil(v * pow(c, (double)(2 * d))) : ceil(v);
        if (r < 1.0) r = 1.0;
        if (r >= 1.8e19) r = 1.8e19;  // the rescan's budget check reports it
        PlanEntry e{};
        e.k = kk;
        e.depth = (uint8_t)std::max(0, d);
        e.early = (uint8_t)(*side && r >= g.alg3_early_pairs ? 1 : 0);
        e.R = (uint64_t)r;
        if (!e.depth && !e.early) continue;
        plan.push_back(e);
        n_early += e.early;
        if (d >= 1) ++used;
        if (d == 2) d2.push_back(kk);
        else if (d > 2) deep.emplace_back(kk, d);
    }
    if (!plan.empty()) {
        ESIM_CUDA_TRY(cudaMemcpyAsync(w.plan, plan.data(), sizeof(PlanEntry) * plan.size(), cudaMemcpyHostToDevice,
                                      g.stream),
                      "upload the plan");
        ESIM_CUDA_TRY(launch_plan_scatter(g, w.plan, (int)plan.size(), w.R, w.depth, w.cand), "scatter the plan");
        *launches += 1;
    }
    g.side_candidates = n_early;
    if (*side) {
        esim_status ss = start_side_walks(g, w, c, seed, launches);
        if (ss != ESIM_OK) return ss;
    }
    ESIM_CUDA_TRY(cudaStreamSynchronize(g.stream), "Algorithm 3 plan");  // plan is a local
    esim_status zs = alg3_zsums_of(g, w.depth, d2, std::move(deep), c, w.zsum, launches);
    if (zs != ESIM_OK) return zs;
    g.last_alg3_nodes = used;
    const int64_t nb = allocate_blocks(g.n);
    ESIM_CUDA_TRY(launch_scan_R(g, g.n, w.R, w.off, g.scan_part, g.norm_part + nb, scan_ticket(g)), "Algorithm 3 rescan");
    *launches += 2;
    return ESIM_OK;
}

// The sampler of a step call, with a chunk counter that no other launch in flight uses.  A
// captured one has none: the graph may be launched on several streams at once.
esim_status sample_step(Graph& g, const uint64_t* off, double c, uint64_t seed, uint64_t* counts, uint64_t* pair_steps,
                        const uint8_t* depth) {
    cudaStreamCaptureStatus capture;
    ESIM_CUDA_TRY(cudaStreamIsCapturing(g.stream, &capture), "stream capture status");
    if (capture != cudaStreamCaptureStatusNone) {
        ESIM_CUDA_TRY(launch_sample(g, off, c, seed, counts, pair_steps, depth, nullptr), "walk pairs");
        return ESIM_OK;
    }
    const unsigned slot = g.sample_slot++ % kSampleSlots;
    cudaEvent_t& done = g.sample_ev[slot];
    if (!done) ESIM_CUDA_TRY(cudaEventCreateWithFlags(&done, cudaEventDisableTiming), "cudaEventCreate");
    ESIM_CUDA_TRY(cudaStreamWaitEvent(g.stream, done, 0), "wait for a chunk counter");
    ESIM_CUDA_TRY(cudaMemsetAsync(g.sample_taken + slot, 0, sizeof(*g.sample_taken), g.stream), "reset chunk counter");
    ESIM_CUDA_TRY(launch_sample(g, off, c, seed, counts, pair_steps, depth, g.sample_taken + slot), "walk pairs");
    ESIM_CUDA_TRY(cudaEventRecord(done, g.stream), "record");
    return ESIM_OK;
}

// Runs the whole query; s_dev may be NULL (the workspace holds s); k > 0 adds top-k.
esim_status run_query(Graph& g, int64_t u, double c, double eps, uint64_t seed, double* s_dev, int32_t k,
                      int32_t* ids_dev, double* vals_dev, double* s_host, int32_t* ids_host, double* vals_host) {
    if (u < 0 || u >= g.n) return fail(ESIM_EINVAL, "source node out of range");
    if (!valid_c_eps(c, eps)) return fail(ESIM_EINVAL, "need 0 < c < 1 and 0 < eps < 1");
    if (k > kTopkMax) return fail(ESIM_ENOTSUP, "k above 4096");
    ESIM_CUDA_TRY(cudaSetDevice(g.device), "cudaSetDevice");
    // sparse linearization (Section 3.2): the query runs at eps/2 and drops the
    // history entries pi^l(k) <= (1 - sqrt c)^2 eps/2, which adds at most eps/2
    const bool sparse = g.sparse_hist && g.precision == 0;
    const double eps_q = sparse ? 0.5 * eps : eps;
    const int32_t L = esim_levels(c, eps_q);
    const double kappa = kappa_of(g, c);
    const double R_b = kappa * log((double)g.n) / (eps_q * eps_q);
    const double a_c = 1.0 - sqrt(c);
    const double theta = a_c * a_c * eps_q;
    Ws w;
    uint64_t cap = 0;
    int count_launches = 0;
    // The pigeonhole bound itself where it is small beside the four n-vectors (half of them): the
    // counting pass below would be a third of the query (n = 1e6, m = 1.75e7: 5.4 against 3.7 ms)
    const uint64_t bound = sparse ? sparse_capacity(g.n, L, theta) : 0;
    if (sparse && bound <= (uint64_t)g.n * 16 / 12) {
        cap = bound;
    } else if (sparse) {
        // counting pass: the forward sweeps once without storing, then a workspace
        // sized to the kept entries (never above the pigeonhole bound)
        esim_status st0 = ensure_ws(g, L, 0, w, 1);
        if (st0 != ESIM_OK) return st0;
        ESIM_CUDA_TRY(cudaMemsetAsync(g.status, 0, sizeof(Status), g.stream), "reset status");
        const SparseHist none{nullptr, nullptr, nullptr, 0};
        ESIM_CUDA_TRY(launch_forward_sparse(g, u, c, L, theta, none, w.lev, w.pirun, w.xa, w.xb),
                      "forward sweeps (counting pass)");
        ESIM_CUDA_TRY(cudaMemcpyAsync(g.status_host, g.status, sizeof(Status), cudaMemcpyDeviceToHost, g.stream),
                      "copy status");
        ESIM_CUDA_TRY(cudaStreamSynchronize(g.stream), "forward sweeps (counting pass)");
        const uint64_t kept = g.status_host->hist_count;
        cap = std::max<uint64_t>(1, std::min<uint64_t>(kept, bound));
        count_launches = 2 + L * 2;
    }
    esim_status st = ensure_ws(g, L, g.precision, w, cap);
    if (st != ESIM_OK) return st;
    double* s = s_dev ? s_dev : w.s;
    if (g.timing)
        for (auto& ev : g.ev)
            if (!ev) ESIM_CUDA_TRY(cudaEventCreate(&ev), "cudaEventCreate");
    ESIM_CUDA_TRY(cudaMemsetAsync(g.status, 0, sizeof(Status), g.stream), "reset status");
    if (g.timing) cudaEventRecord(g.ev[0], g.stream);
    if (sparse)
        ESIM_CUDA_TRY(launch_forward_sparse(g, u, c, L, theta, w.sh, w.lev, w.pirun, w.xa, w.xb),
                      "forward sweeps (sparse history)");
    else if (g.precision == 0) ESIM_CUDA_TRY(launch_forward(g, u, c, L, w.hist, w.xa, w.xb), "forward sweeps");
    else ESIM_CUDA_TRY(launch_forward32(g, u, c, L, w.hist32, w.xa32, w.xb32), "forward sweeps (FP32c)");
    if (g.timing) cudaEventRecord(g.ev[1], g.stream);
    // kernels of the allocation, sampling and D^ phases (the default counts 2 + 1 + 1)
    int extra_launches = 0;
    bool side_used = false;
    g.last_alg3_nodes = 0;
    if (g.diag_mode == 1) {
        // ParSim's approximation D = (1-c) I: no allocation and no walk pairs
        if (g.timing) {
            cudaEventRecord(g.ev[2], g.stream);
            cudaEventRecord(g.ev[6], g.stream);
            cudaEventRecord(g.ev[7], g.stream);
            cudaEventRecord(g.ev[3], g.stream);
        }
        ESIM_CUDA_TRY(launch_fill(g, g.n, 1.0 - c, w.dhat), "dhat (ParSim)");
        extra_launches -= 3;
    } else {
        if (sparse)  // pi was summed level by level during the forward sweeps
            ESIM_CUDA_TRY(launch_allocate(g, w.pirun, 0, R_b, g.alloc_mode, w.pi, w.R, w.off), "allocation");
        else if (g.precision == 0)
            ESIM_CUDA_TRY(launch_allocate(g, w.hist, L, R_b, g.alloc_mode, w.pi, w.R, w.off), "allocation");
        else
            ESIM_CUDA_TRY(launch_allocate32(g, w.hist32, L, R_b, g.alloc_mode, w.pi, w.R, w.off),
                          "allocation (FP32c)");
        bool side = false;
        if (g.alg3) {
            esim_status a3 = plan_alg3(g, w, c, R_b, &extra_launches, seed, &side);
            if (a3 != ESIM_OK) {
                if (side) cudaStreamSynchronize(g.side_stream);  // no walks left running into the next query
                return a3;
            }
        }
        if (g.timing) cudaEventRecord(g.ev[2], g.stream);
        if (side) {
            // the remaining candidates' walks here; the side stream's counts for the rest
            ESIM_CUDA_TRY(launch_mask_R(g, w.R, w.cand, 1u << 1, w.R2), "candidates' R");
            ESIM_CUDA_TRY(launch_scan_R(g, g.n, w.R2, w.offc, g.scan_part, g.norm_part + allocate_blocks(g.n),
                                        scan_ticket(g), false),
                          "candidates' scan");
            if (g.timing) cudaEventRecord(g.ev[6], g.stream);
            ESIM_CUDA_TRY(launch_sample(g, w.offc, c, seed, w.nonmeet, nullptr, w.depth, &g.status->taken[0]),
                          "candidates' walk pairs");
            if (g.timing) cudaEventRecord(g.ev[7], g.stream);
            ESIM_CUDA_TRY(cudaStreamWaitEvent(g.stream, g.side_ev[1], 0), "wait for the side walks");
            ESIM_CUDA_TRY(launch_merge_counts(g, w.cand, w.nm2, w.nonmeet), "merge counts");
            extra_launches += 4;
        } else {
            if (g.timing) cudaEventRecord(g.ev[6], g.stream);
            ESIM_CUDA_TRY(launch_sample(g, w.off, c, seed, w.nonmeet, nullptr, g.alg3 ? w.depth : nullptr,
                                        &g.status->taken[0]),
                          "walk pairs");
            if (g.timing) cudaEventRecord(g.ev[7], g.stream);
        }
        side_used = side;
        if (g.timing) cudaEventRecord(g.ev[3], g.stream);
        if (g.alg3)
            ESIM_CUDA_TRY(launch_dhat_alg3(g, w.nonmeet, w.off, w.depth, w.zsum, c, w.dhat), "dhat (Algorithm 3)");
        else ESIM_CUDA_TRY(launch_dhat(g, w.nonmeet, w.off, w.dhat), "dhat");
    }
    if (sparse)
        ESIM_CUDA_TRY(launch_reverse_sparse(g, w.sh, L, c, w.dhat, s, w.xa), "reverse sweeps (sparse history)");
    else if (g.precision == 0)
        ESIM_CUDA_TRY(launch_reverse(g, w.hist, L, c, w.dhat, s, w.xa, w.xb), "reverse sweeps");
    else
        ESIM_CUDA_TRY(launch_reverse32(g, w.hist32, L, c, w.dhat, s, w.w2, w.sa2, w.sb2), "reverse sweeps (FP32c)");
    if (g.timing) cudaEventRecord(g.ev[4], g.stream);
    if (k > 0) {
        int32_t* ids = ids_dev;
        double* vals = vals_dev;
        if (!ids) {  // host outputs: stage behind the top-k workspace
            char* stage = (char*)g.topk_ws + topk_stage_offset(g.n);
            vals = (double*)stage;
            ids = (int32_t*)(stage + sizeof(double) * kTopkMax);
        }
        ESIM_CUDA_TRY(launch_topk(g, s, g.exclude_source ? u : -1, k, ids, vals, g.topk_ws), "top-k");
        if (ids_host) {
            ESIM_CUDA_TRY(cudaMemcpyAsync(ids_host, ids, sizeof(int32_t) * (size_t)k, cudaMemcpyDeviceToHost, g.stream),
                          "copy ids");
            ESIM_CUDA_TRY(cudaMemcpyAsync(vals_host, vals, sizeof(double) * (size_t)k, cudaMemcpyDeviceToHost, g.stream),
                          "copy scores");
        }
    }
    if (g.timing) cudaEventRecord(g.ev[5], g.stream);
    if (s_host)
        ESIM_CUDA_TRY(cudaMemcpyAsync(s_host, s, sizeof(double) * (size_t)g.n, cudaMemcpyDeviceToHost, g.stream),
                      "copy scores");
    ESIM_CUDA_TRY(cudaMemcpyAsync(g.status_host, g.status, sizeof(Status), cudaMemcpyDeviceToHost, g.stream),
                  "copy status");
    ESIM_CUDA_TRY(cudaStreamSynchronize(g.stream), "query");
    const Status hs = *g.status_host;
    g.last_L = L;
    // kernels launched: forward init + per level, 2 allocation
    // kernels, the sampler, D^, reverse init + per level, and 2 for top-k
    g.last_launches = (1 + L) + 2 + 1 + 1 + (1 + L) + (k > 0 ? 2 : 0) + extra_launches;
    if (sparse) g.last_launches += 2 * (L + 1) + count_launches;  // compactions, scatters, counting pass
    g.last_hist_entries = sparse ? std::min<uint64_t>(hs.hist_count, cap) : (uint64_t)(L + 1) * (uint64_t)g.n;
    g.last_R_b = R_b;
    g.last_kappa = kappa;
    g.last_norm2 = hs.pi_norm2;
    g.last_sum_R = hs.sum_R;
    g.last_steps = hs.pair_steps + (side_used ? hs.pair_steps_side : 0ull);
    g.last_steps_side = side_used ? hs.pair_steps_side : 0ull;
    for (float& x : g.last_ms) x = 0.f;
    g.last_ms_kernel = g.last_ms_side = 0.f;
    g.last_side_candidates = side_used ? g.side_candidates : 0;
    if (g.timing) {
        for (int i = 0; i < 5; ++i) cudaEventElapsedTime(&g.last_ms[i], g.ev[i], g.ev[i + 1]);
        cudaEventElapsedTime(&g.last_ms[5], g.ev[0], g.ev[5]);
        cudaEventElapsedTime(&g.last_ms_kernel, g.ev[6], g.ev[7]);
        if (side_used) cudaEventElapsedTime(&g.last_ms_side, g.side_tev[0], g.side_tev[1]);
    }
    if (hs.err & kErrBudget)
        return fail(ESIM_EBUDGET, "sum of R(k) = " + std::to_string((double)hs.sum_R) + " exceeds the pair budget");
    if (hs.err & kErrTimeout) return fail(ESIM_ETIMEOUT, "device wait timed out");
    if (hs.err & kErrCapacity) return fail(ESIM_ENOMEM, "sparse history above its capacity");
    return ESIM_OK;
}


// ---------------------------------------------------------------- batches

// Batch workspace (its own arena).
struct BWs {
    float* hist;      // (Lmax+1) n W
    float* xa;        // n W
    float* xb;        // n W
    float2* w;        // n W
    float2* sa;       // n W
    float2* sb;       // n W
    void* partial;    // nseg_max W two-floats
    uint64_t* R;      // B n
    uint64_t* off;    // B n + 1
    uint64_t* nonmeet;// B n
    uint64_t* rbase;  // B n  shared walks: first pair of each (node, interval) segment
    uint64_t* scount; // B n  shared walks: interval lengths, then interval counts
    double* dhat;     // B n
    double* s;        // B n
    int64_t* u;       // W
    int32_t* L;       // W
    double* Rb;       // W
    unsigned long long* part_R;  // tiles of B n
    unsigned* ticket;            // of their scan
    double* part_Rd;
    void* topk;       // batched top-k state
    int32_t* ids;     // B k (staging)
    double* vals;     // B k
};

size_t bws_layout(int64_t n_, int W, int B, int32_t Lmax, int64_t nseg_max, int k, char* base, BWs* out) {
    const size_t n = (size_t)n_, nw = n * (size_t)W, bn = n * (size_t)B;
    size_t o = 0;
    auto take = [&](size_t bytes) -> char* {
        char* p = base ? base + o : nullptr;
        o += round256(bytes);
        return p;
    };
    BWs t{};
    t.hist = (float*)take(4 * nw * (size_t)(Lmax + 1));
    t.xa = (float*)take(4 * nw);
    t.xb = (float*)take(4 * nw);
    t.w = (float2*)take(8 * nw);
    t.sa = (float2*)take(8 * nw);
    t.sb = (float2*)take(8 * nw);
    t.partial = take(8 * (size_t)std::max<int64_t>(1, nseg_max) * (size_t)W);
    t.R = (uint64_t*)take(8 * bn);
    t.off = (uint64_t*)take(8 * (bn + 1));
    t.nonmeet = (uint64_t*)take(8 * bn);
    t.rbase = (uint64_t*)take(8 * bn);
    t.scount = (uint64_t*)take(8 * bn);
    t.dhat = (double*)take(8 * bn);
    t.s = (double*)take(8 * bn);
    t.u = (int64_t*)take(8 * W);
    t.L = (int32_t*)take(4 * W);
    t.Rb = (double*)take(8 * W);
    const size_t nb = (size_t)allocate_blocks((int64_t)bn);
    t.part_R = (unsigned long long*)take(8 * nb);
    t.ticket = (unsigned*)take(sizeof(unsigned));
    t.part_Rd = (double*)take(8 * nb);
    t.topk = take(topk_batch_workspace_bytes(B));
    t.ids = (int32_t*)take(4 * (size_t)B * (size_t)std::max(k, 1));
    t.vals = (double*)take(8 * (size_t)B * (size_t)std::max(k, 1));
    if (out) *out = t;
    return o;
}

// Autotune: time each tile shape on one forward and one reverse level of the live
// batch (the results are identical for every tile, so the timing runs are harmless).
esim_status tune_batch_tiles(Graph& g, const Graph& view, int W, int B, double c, const BWs& w) {
    const int wi = batch_wi(W);
    if (g.batch_tile_force >= 0) {
        g.batch_tile_fwd[wi] = g.batch_tile_rev[wi] = g.batch_tile_force;
        return ESIM_OK;
    }
    if (g.batch_tile_fwd[wi] >= 0) return ESIM_OK;
    cudaEvent_t e0, e1;
    ESIM_CUDA_TRY(cudaEventCreate(&e0), "cudaEventCreate");
    ESIM_CUDA_TRY(cudaEventCreate(&e1), "cudaEventCreate");
    const size_t nw = (size_t)g.n * W;
    float best_f = 1e30f, best_r = 1e30f;
    for (int t = 0; t < batch_tile_count(); ++t) {
        for (int rep = 0; rep < 2; ++rep) {  // first run warms up
            cudaEventRecord(e0, view.stream);
            ESIM_CUDA_TRY(launch_batch_forward_level(view, W, t, 1, c, w.L, w.xa, w.hist + nw, w.xb, w.partial),
                          "batch tune forward");
            cudaEventRecord(e1, view.stream);
            ESIM_CUDA_TRY(cudaEventSynchronize(e1), "batch tune");
            float ms = 0.f;
            cudaEventElapsedTime(&ms, e0, e1);
            if (rep == 1) {
                g.batch_tune_ms[wi][0][t] = ms;
                if (ms < best_f) { best_f = ms; g.batch_tile_fwd[wi] = t; }
            }
            cudaEventRecord(e0, view.stream);
            ESIM_CUDA_TRY(launch_batch_reverse_level(view, W, B, t, false, c, w.w, w.hist, w.sa, w.sb, nullptr,
                                                     w.partial),
                          "batch tune reverse");
            cudaEventRecord(e1, view.stream);
            ESIM_CUDA_TRY(cudaEventSynchronize(e1), "batch tune");
            cudaEventElapsedTime(&ms, e0, e1);
            if (rep == 1) {
                g.batch_tune_ms[wi][1][t] = ms;
                if (ms < best_r) { best_r = ms; g.batch_tile_rev[wi] = t; }
            }
        }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    return ESIM_OK;
}

esim_status run_batch(Graph& g, int32_t B, const int64_t* u, const double* eps, uint64_t seed, double c,
                      double* s_dev, double* s_host, int32_t k, int32_t* ids_dev, double* vals_dev, int32_t* ids_host,
                      double* vals_host) {
    BatchPlan plan;
    esim_status st = (esim_status)batch_plan(g, B, u, eps, c, k, &plan);
    if (st != ESIM_OK) return st;
    ESIM_CUDA_TRY(cudaSetDevice(g.device), "cudaSetDevice");
    const size_t need = batch_ws_bytes(g, plan);
    if (need > g.bws_bytes) {
        cudaStreamSynchronize(g.stream);
        cudaFree(g.bws);
        g.bws = nullptr;
        g.bws_bytes = 0;
        if (cudaMalloc(&g.bws, need) != cudaSuccess) {
            cudaGetLastError();
            return fail(ESIM_ENOMEM, "cudaMalloc(batch workspace of " + std::to_string(need) + " bytes)");
        }
        g.bws_bytes = need;
    }
    if (g.timing)
        for (auto& ev : g.ev)
            if (!ev) ESIM_CUDA_TRY(cudaEventCreate(&ev), "cudaEventCreate");
    st = (esim_status)batch_enqueue(g, g, plan, g.bws, seed, c, s_dev, s_host, ids_dev, vals_dev, ids_host, vals_host,
                                   true);
    if (st != ESIM_OK) return st;
    ESIM_CUDA_TRY(cudaStreamSynchronize(g.stream), "batch query");
    const Status hs = *g.status_host;
    g.last_L = plan.Lmax;
    g.last_launches = 1 + plan.Lmax * (1 + (g.out.bnlong > 0 ? 1 : 0)) + 1 + 2 + 1 + 1 + 1 +
                      plan.Lmax * (1 + (g.in.bnlong > 0 ? 1 : 0)) + (k > 0 ? 2 : 0) + (g.shared_walks ? 2 : 0);
    g.last_R_b = plan.Rb[0];
    g.last_kappa = kappa_of(g, c);
    g.last_norm2 = 0.0;
    g.last_sum_R = hs.sum_R;
    g.last_steps = hs.pair_steps;
    for (float& x : g.last_ms) x = 0.f;
    g.last_ms_kernel = g.last_ms_side = 0.f;
    g.last_side_candidates = 0;
    g.last_steps_side = 0;
    if (g.timing) {
        for (int i = 0; i < 5; ++i) cudaEventElapsedTime(&g.last_ms[i], g.ev[i], g.ev[i + 1]);
        cudaEventElapsedTime(&g.last_ms[5], g.ev[0], g.ev[5]);
        g.last_ms_kernel = g.last_ms[2];
    }
    if (hs.err & kErrBudget)
        return fail(ESIM_EBUDGET, "sum of R(k) = " + std::to_string((double)hs.sum_R) + " exceeds the pair budget");
    return ESIM_OK;
}

}  // namespace

int esim::set_error(int status, const std::string& message) {
    t_err = message;
    return status;
}

namespace esim {

Graph* graph_of(::esim_graph* h) { return &h->g; }

int batch_width(int B) { return B <= 16 ? 16 : (B <= 32 ? 32 : 64); }
int batch_wi(int W) { return W == 16 ? 0 : (W == 32 ? 1 : 2); }

int batch_plan(const Graph& g, int32_t B, const int64_t* u, const double* eps, double c, int32_t k, BatchPlan* plan) {
    if (B < 1) return fail(ESIM_EINVAL, "need B >= 1");
    if (B > kBatchMax) return fail(ESIM_ENOTSUP, "B above 64: split the batch");
    if (!u || !eps) return fail(ESIM_EINVAL, "NULL u or eps");
    if (!(c > 0.0 && c < 1.0)) return fail(ESIM_EINVAL, "need 0 < c < 1");
    if (k > kTopkMax) return fail(ESIM_ENOTSUP, "k above 4096");
    BatchPlan p{};
    p.B = B;
    p.W = batch_width(B);
    p.k = k;
    p.Lmax = 0;
    for (int q = 0; q < kBatchMax; ++q) {
        p.Lq[q] = -1;
        p.Rb[q] = 0.0;
        p.u[q] = -1;
    }
    for (int q = 0; q < B; ++q) {
        if (u[q] < 0 || u[q] >= g.n) return fail(ESIM_EINVAL, "source node out of range");
        if (!valid_c_eps(c, eps[q])) return fail(ESIM_EINVAL, "need 0 < eps < 1");
        p.Lq[q] = esim_levels(c, eps[q]);
        p.Rb[q] = kappa_of(g, c) * log((double)g.n) / (eps[q] * eps[q]);
        p.u[q] = u[q];
        p.Lmax = std::max(p.Lmax, p.Lq[q]);
    }
    *plan = p;
    return ESIM_OK;
}

size_t batch_ws_bytes(const Graph& g, const BatchPlan& p) {
    return bws_layout(g.n, p.W, p.B, p.Lmax, std::max(g.in.bnseg, g.out.bnseg), p.k, nullptr, nullptr);
}

// Enqueue the whole batch on view.stream using the arena `ws`; results go to the
// given device or host buffers (host copies are asynchronous).  The status block
// view.status is reset first and copied to view.status_host last.
int batch_enqueue(Graph& tuner, const Graph& view, const BatchPlan& p, void* ws, uint64_t seed, double c,
                  double* s_dev, double* s_host, int32_t* ids_dev, double* vals_dev, int32_t* ids_host,
                  double* vals_host, bool allow_tune) {
    BWs w;
    bws_layout(view.n, p.W, p.B, p.Lmax, std::max(view.in.bnseg, view.out.bnseg), p.k, (char*)ws, &w);
    const int W = p.W, B = p.B, k = p.k;
    const int32_t Lmax = p.Lmax;
    const size_t nw = (size_t)view.n * W;
    const int64_t N = view.n * (int64_t)B;
    const cudaStream_t stream = view.stream;
    const bool timing = view.timing && view.ev[0];
    ESIM_CUDA_TRY(cudaMemsetAsync(view.status, 0, sizeof(Status), stream), "reset status");
    ESIM_CUDA_TRY(cudaMemcpyAsync(w.u, p.u, sizeof(int64_t) * W, cudaMemcpyHostToDevice, stream), "upload sources");
    ESIM_CUDA_TRY(cudaMemcpyAsync(w.L, p.Lq, sizeof(int32_t) * W, cudaMemcpyHostToDevice, stream), "upload depths");
    ESIM_CUDA_TRY(cudaMemcpyAsync(w.Rb, p.Rb, sizeof(double) * W, cudaMemcpyHostToDevice, stream), "upload R_b");
    ESIM_CUDA_TRY(cudaMemsetAsync(w.ticket, 0, sizeof(*w.ticket), stream), "reset scan ticket");
    if (timing) cudaEventRecord(view.ev[0], stream);
    ESIM_CUDA_TRY(launch_batch_forward_init(view, W, B, w.u, c, w.hist, w.xa), "batch forward init");
    const int wi = batch_wi(W);
    if (Lmax >= 1 && allow_tune) {
        esim_status ts = (esim_status)tune_batch_tiles(tuner, view, W, B, c, w);
        if (ts != ESIM_OK) return ts;
    }
    const int tf = tuner.batch_tile_fwd[wi] < 0 ? 0 : tuner.batch_tile_fwd[wi];
    const int tr = tuner.batch_tile_rev[wi] < 0 ? 0 : tuner.batch_tile_rev[wi];
    float* x[2] = {w.xa, w.xb};
    for (int32_t l = 1; l <= Lmax; ++l)
        ESIM_CUDA_TRY(launch_batch_forward_level(view, W, tf, l, c, w.L, x[(l - 1) & 1], w.hist + (size_t)l * nw,
                                                 x[l & 1], w.partial),
                      "batch forward level");
    if (timing) cudaEventRecord(view.ev[1], stream);
    ESIM_CUDA_TRY(launch_batch_alloc(view, W, B, w.hist, Lmax, w.Rb, view.alloc_mode, w.R), "batch allocation");
    if (view.shared_walks) {
        // one walk set per node: intervals between the distinct R_q(k), sampled once
        ESIM_CUDA_TRY(launch_shared_plan(view, B, w.R, w.scount, w.rbase), "shared walk plan");
        ESIM_CUDA_TRY(launch_scan_R(view, N, w.scount, w.off, w.part_R, w.part_Rd, w.ticket), "shared walk scan");
        if (timing) cudaEventRecord(view.ev[2], stream);
        ESIM_CUDA_TRY(launch_sample_segments(view, N, w.off, c, seed, w.scount, &view.status->taken[0], nullptr, nullptr,
                                             B, w.rbase),
                      "batch walk pairs (shared)");
        if (timing) cudaEventRecord(view.ev[3], stream);
        ESIM_CUDA_TRY(launch_shared_columns(view, B, w.R, w.rbase, w.off, w.scount, w.nonmeet), "shared walk counts");
        ESIM_CUDA_TRY(launch_dhat_from_R(view, N, w.nonmeet, w.R, w.dhat), "batch dhat");
    } else {
        ESIM_CUDA_TRY(launch_scan_R(view, N, w.R, w.off, w.part_R, w.part_Rd, w.ticket), "batch scan");
        if (timing) cudaEventRecord(view.ev[2], stream);
        ESIM_CUDA_TRY(launch_sample_segments(view, N, w.off, c, seed, w.nonmeet, &view.status->taken[0], nullptr),
                      "batch walk pairs");
        if (timing) cudaEventRecord(view.ev[3], stream);
        ESIM_CUDA_TRY(launch_dhat_segments(view, N, w.nonmeet, w.off, w.dhat), "batch dhat");
    }
    double* s = s_dev ? s_dev : w.s;
    ESIM_CUDA_TRY(launch_batch_reverse_init(view, W, B, w.dhat, c, w.hist + (size_t)Lmax * nw, w.w, w.sa,
                                            Lmax == 0 ? s : nullptr),
                  "batch reverse init");
    float2* sb[2] = {w.sa, w.sb};
    for (int32_t l = 1; l <= Lmax; ++l)
        ESIM_CUDA_TRY(launch_batch_reverse_level(view, W, B, tr, l == Lmax, c, w.w, w.hist + (size_t)(Lmax - l) * nw,
                                                 sb[(l - 1) & 1], sb[l & 1], s, w.partial),
                      "batch reverse level");
    if (timing) cudaEventRecord(view.ev[4], stream);
    if (k > 0) {
        int32_t* ids = ids_dev ? ids_dev : w.ids;
        double* vals = vals_dev ? vals_dev : w.vals;
        ESIM_CUDA_TRY(launch_topk_batch(view, B, s, view.exclude_source ? w.u : nullptr, k, ids, vals, w.topk),
                      "batch top-k");
        if (ids_host) {
            ESIM_CUDA_TRY(cudaMemcpyAsync(ids_host, ids, sizeof(int32_t) * (size_t)B * k, cudaMemcpyDeviceToHost,
                                          stream), "copy ids");
            ESIM_CUDA_TRY(cudaMemcpyAsync(vals_host, vals, sizeof(double) * (size_t)B * k, cudaMemcpyDeviceToHost,
                                          stream), "copy scores");
        }
    }
    if (timing) cudaEventRecord(view.ev[5], stream);
    if (s_host)
        ESIM_CUDA_TRY(cudaMemcpyAsync(s_host, s, sizeof(double) * (size_t)N, cudaMemcpyDeviceToHost, stream),
                      "copy scores");
    ESIM_CUDA_TRY(cudaMemcpyAsync(view.status_host, view.status, sizeof(Status), cudaMemcpyDeviceToHost, stream),
                  "copy status");
    return ESIM_OK;
}

}  // namespace esim

extern "C" {

const char* esim_version(void) { return "exactsim-gb300 0.1 (sm_103a)"; }

const char* esim_last_error(void) { return t_err.c_str(); }

int32_t esim_levels(double c, double eps) {
    if (!valid_c_eps(c, eps)) return -1;
    return (int32_t)ceil(log(2.0 / eps) / log(1.0 / c));
}

double esim_sample_base(int64_t n, double c, double eps, double kappa) {
    if (n < 1 || !valid_c_eps(c, eps)) return -1.0;
    if (kappa <= 0.0) {
        const double a = 1.0 - sqrt(c);
        kappa = 6.0 / (a * a * a * a);
    }
    return kappa * log((double)n) / (eps * eps);
}

uint32_t esim_walk_threshold(double c) { return walk_threshold(c); }

esim_status esim_load_graph(int64_t n, const int64_t* in_rowptr, const int32_t* in_col, esim_graph** out) {
    if (!out) return fail(ESIM_EINVAL, "out is NULL");
    *out = nullptr;
    if (n < 1 || n >= (int64_t)1 << 31) return fail(ESIM_EINVAL, "need 1 <= n < 2^31");
    if (!in_rowptr) return fail(ESIM_EINVAL, "in_rowptr is NULL");
    if (in_rowptr[0] != 0) return fail(ESIM_EINVAL, "in_rowptr[0] must be 0");
    for (int64_t j = 0; j < n; ++j)
        if (in_rowptr[j + 1] < in_rowptr[j]) return fail(ESIM_EINVAL, "in_rowptr is not non-decreasing");
    const int64_t m = in_rowptr[n];
    if (m >= ((int64_t)1 << 32) - 4096) return fail(ESIM_EINVAL, "need m < 2^32 - 4096");
    if (m > 0 && !in_col) return fail(ESIM_EINVAL, "in_col is NULL");
    for (int64_t p = 0; p < m; ++p)
        if (in_col[p] < 0 || (int64_t)in_col[p] >= n) return fail(ESIM_EINVAL, "in_col entry out of range");

    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return cuda_fail(e, "cudaGetDevice (no usable CUDA device)");
    cudaDeviceProp prop;
    ESIM_CUDA_TRY(cudaGetDeviceProperties(&prop, dev), "cudaGetDeviceProperties");

    esim_graph* h = new (std::nothrow) esim_graph();
    if (!h) return fail(ESIM_ENOMEM, "host allocation");
    Graph& g = h->g;
    g.device = dev;
    g.sm_count = prop.multiProcessorCount;
    g.n = n;
    g.m = m;

    // host: 32-bit in-CSR, and the out-CSR by a stable counting sort (rows of the
    // out-CSR list targets j in increasing order)
    std::vector<uint32_t> in_rp((size_t)n + 1), out_rp((size_t)n + 1, 0);
    for (int64_t j = 0; j <= n; ++j) in_rp[j] = (uint32_t)in_rowptr[j];
    std::vector<int32_t> out_c((size_t)m);
    for (int64_t p = 0; p < m; ++p) out_rp[(size_t)in_col[p] + 1]++;
    for (int64_t i = 0; i < n; ++i) out_rp[i + 1] += out_rp[i];
    {
        std::vector<uint32_t> cur(out_rp.begin(), out_rp.end() - 1);
        for (int64_t j = 0; j < n; ++j)
            for (int64_t p = in_rowptr[j]; p < in_rowptr[j + 1]; ++p) out_c[cur[in_col[p]]++] = (int32_t)j;
    }
    // repeated in-edges (Algorithm 3 needs a simple graph): a row of the out-CSR is ascending, so they
    // are neighbours there; equal neighbours of two rows are taken off again
    int64_t repeated = 0;
    for (int64_t p = 1; p < m; ++p) repeated += out_c[(size_t)p] == out_c[(size_t)p - 1];
    for (int64_t i = 0; i < n && repeated > 0; ++i) {
        const uint32_t p = out_rp[(size_t)i];
        if (p > 0 && p < out_rp[(size_t)i + 1]) repeated -= out_c[p] == out_c[p - 1];
    }
    g.has_duplicates = repeated > 0;
    auto din = std::make_shared<std::vector<uint32_t>>((size_t)n);
    for (int64_t j = 0; j < n; ++j) (*din)[j] = in_rp[j + 1] - in_rp[j];
    g.din_host = din;
    g.stream = cudaStreamPerThread;
    const esim_status st = upload_graph(g, in_rp, in_col, out_rp, out_c.data());
    if (st != ESIM_OK) {
        release(g);
        delete h;
        return st;
    }
    const bool ok = cudaMallocHost((void**)&g.status_host, sizeof(Status)) == cudaSuccess &&
                    cudaStreamCreateWithFlags(&g.own_stream, cudaStreamNonBlocking) == cudaSuccess &&
                    cudaStreamCreateWithFlags(&g.side_stream, cudaStreamNonBlocking) == cudaSuccess &&
                    cudaEventCreateWithFlags(&g.side_ev[0], cudaEventDisableTiming) == cudaSuccess &&
                    cudaEventCreateWithFlags(&g.side_ev[1], cudaEventDisableTiming) == cudaSuccess;
    if (!ok) {
        cudaGetLastError();
        release(g);
        delete h;
        return fail(ESIM_ENOMEM, "device allocation for graph workspace");
    }
    g.stream = g.own_stream;
    *out = h;
    return ESIM_OK;
}

void esim_free_graph(esim_graph* h) {
    if (!h) return;
    release(h->g);
    delete h;
}

int64_t esim_num_nodes(const esim_graph* h) { return h ? h->g.n : -1; }
int64_t esim_num_edges(const esim_graph* h) { return h ? h->g.m : -1; }

esim_status esim_set_stream(esim_graph* h, void* stream) {
    if (check_graph(h)) return ESIM_EINVAL;
    h->g.stream = stream ? (cudaStream_t)stream : h->g.own_stream;
    return ESIM_OK;
}

esim_status esim_set_option(esim_graph* h, const char* key, double value) {
    if (check_graph(h)) return ESIM_EINVAL;
    if (!key) return fail(ESIM_EINVAL, "option key is NULL");
    Graph& g = h->g;
    const std::string k(key);
    if (k == "kappa") {
        if (!(value == value)) return fail(ESIM_EINVAL, "kappa is NaN");
        g.kappa = value;
    } else if (k == "alloc") {
        if (value != 0.0 && value != 1.0) return fail(ESIM_EINVAL, "alloc must be 0 (pi^2) or 1 (basic)");
        g.alloc_mode = (int)value;
    } else if (k == "exclude_source") {
        if (value != 0.0 && value != 1.0) return fail(ESIM_EINVAL, "exclude_source must be 0 or 1");
        g.exclude_source = (int)value;
    } else if (k == "pair_budget") {
        if (!(value >= 0.0)) return fail(ESIM_EINVAL, "pair_budget must be >= 0");
        g.pair_budget = value;
    } else if (k == "timing") {
        if (value != 0.0 && value != 1.0) return fail(ESIM_EINVAL, "timing must be 0 or 1");
        g.timing = (int)value;
    } else if (k == "batch_tile") {
        if (value != -1.0 && value != 0.0 && value != 1.0 && value != 2.0)
            return fail(ESIM_EINVAL, "batch_tile must be -1 (autotune), 0, 1 or 2");
        g.batch_tile_force = (int)value;
        for (int i = 0; i < 3; ++i) g.batch_tile_fwd[i] = g.batch_tile_rev[i] = -1;
    } else if (k == "precision") {
        if (value != 0.0 && value != 1.0) return fail(ESIM_EINVAL, "precision must be 0 (FP64) or 1 (FP32c)");
        if (value == 1.0 && g.sparse_hist) return fail(ESIM_ENOTSUP, "sparse_hist needs precision 0 (FP64)");
        g.precision = (int)value;
    } else if (k == "shared_walks") {
        if (value != 0.0 && value != 1.0) return fail(ESIM_EINVAL, "shared_walks must be 0 or 1");
        g.shared_walks = (int)value;
    } else if (k == "sparse_hist") {
        if (value != 0.0 && value != 1.0) return fail(ESIM_EINVAL, "sparse_hist must be 0 or 1");
        if (value == 1.0 && g.precision != 0) return fail(ESIM_ENOTSUP, "sparse_hist needs precision 0 (FP64)");
        g.sparse_hist = (int)value;
    } else if (k == "diag") {
        if (value != 0.0 && value != 1.0) return fail(ESIM_EINVAL, "diag must be 0 (estimated) or 1 (ParSim (1-c) I)");
        g.diag_mode = (int)value;
    } else if (k == "alg3") {
        if (value != 0.0 && value != 1.0) return fail(ESIM_EINVAL, "alg3 must be 0 or 1");
        if (value == 1.0 && g.has_duplicates)
            return fail(ESIM_ENOTSUP, "Algorithm 3 needs a graph without repeated in-edges");
        g.alg3 = (int)value;
    } else if (k == "alg3_rule") {
        if (value != 0.0 && value != 1.0)
            return fail(ESIM_EINVAL, "alg3_rule must be 0 (the paper's explored-edge rule) or 1 (cost model)");
        g.alg3_rule = (int)value;
    } else if (k == "alg3_max_depth") {
        if (!(value >= 1.0 && value <= (double)kAlg3MaxDepth) || value != floor(value))
            return fail(ESIM_EINVAL, "alg3_max_depth must be an integer in [1, 16]");
        g.alg3_max_depth = (int)value;
    } else if (k == "alg3_min_pairs") {
        if (!(value >= 0.0)) return fail(ESIM_EINVAL, "alg3_min_pairs must be >= 0");
        g.alg3_min_pairs = value;
    } else if (k == "alg3_w_last") {
        if (!(value >= 0.0)) return fail(ESIM_EINVAL, "alg3_w_last must be >= 0");
        g.alg3_w_last = value;
    } else if (k == "alg3_w_sweep" || k == "alg3_w_probe" || k == "alg3_w_launch") {
        if (!(value >= 0.0)) return fail(ESIM_EINVAL, k + " must be >= 0");
        (k == "alg3_w_sweep" ? g.alg3_w_sweep : k == "alg3_w_probe" ? g.alg3_w_probe : g.alg3_w_launch) = value;
    } else if (k == "alg3_early_pairs") {
        if (!(value >= 1.0)) return fail(ESIM_EINVAL, "alg3_early_pairs must be >= 1");
        g.alg3_early_pairs = value;
    } else if (k == "alg3_push_div") {
        if (!(value >= 1.0 && value <= 1e6) || value != floor(value))
            return fail(ESIM_EINVAL, "alg3_push_div must be an integer in [1, 1e6]");
        g.alg3_push_div = (int)value;
    } else if (k == "alg3_overlap") {
        if (!(value >= 0.0 && value <= 64.0) || value != floor(value))
            return fail(ESIM_EINVAL, "alg3_overlap must be an integer in [0, 64]");
        g.alg3_overlap = (int)value;
    } else if (k == "alg3_workers") {
        if (!(value >= 1.0 && value <= 16.0) || value != floor(value))
            return fail(ESIM_EINVAL, "alg3_workers must be an integer in [1, 16]");
        g.alg3_workers = (int)value;
    } else if (k == "alg3_max_nodes") {
        if (!(value >= 1.0 && value <= 4096.0)) return fail(ESIM_EINVAL, "alg3_max_nodes must be in [1, 4096]");
        g.alg3_max_nodes = (int)value;
    } else {
        return fail(ESIM_EINVAL, "unknown option '" + k + "'");
    }
    return ESIM_OK;
}

esim_status esim_get_option(const esim_graph* h, const char* key, double* value) {
    if (check_graph(h)) return ESIM_EINVAL;
    if (!key || !value) return fail(ESIM_EINVAL, "NULL argument");
    const Graph& g = h->g;
    const std::string k(key);
    if (k == "kappa") *value = g.kappa;
    else if (k == "alloc") *value = g.alloc_mode;
    else if (k == "exclude_source") *value = g.exclude_source;
    else if (k == "pair_budget") *value = g.pair_budget;
    else if (k == "timing") *value = g.timing;
    else if (k == "precision") *value = g.precision;
    else if (k == "diag") *value = g.diag_mode;
    else if (k == "sparse_hist") *value = g.sparse_hist;
    else if (k == "shared_walks") *value = g.shared_walks;
    else if (k == "alg3") *value = g.alg3;
    else if (k == "alg3_rule") *value = g.alg3_rule;
    else if (k == "alg3_max_depth") *value = g.alg3_max_depth;
    else if (k == "alg3_min_pairs") *value = g.alg3_min_pairs;
    else if (k == "alg3_max_nodes") *value = g.alg3_max_nodes;
    else if (k == "alg3_overlap") *value = g.alg3_overlap;
    else if (k == "alg3_push_div") *value = g.alg3_push_div;
    else if (k == "alg3_early_pairs") *value = g.alg3_early_pairs;
    else if (k == "alg3_w_sweep") *value = g.alg3_w_sweep;
    else if (k == "alg3_w_probe") *value = g.alg3_w_probe;
    else if (k == "alg3_w_last") *value = g.alg3_w_last;
    else if (k == "alg3_workers") *value = g.alg3_workers;
    else if (k == "alg3_w_launch") *value = g.alg3_w_launch;
    else if (k == "batch_tile") *value = g.batch_tile_force;
    else if (k == "batch_tile_fwd16") *value = g.batch_tile_fwd[0];
    else if (k == "batch_tile_fwd32") *value = g.batch_tile_fwd[1];
    else if (k == "batch_tile_fwd64") *value = g.batch_tile_fwd[2];
    else if (k == "batch_tile_rev16") *value = g.batch_tile_rev[0];
    else if (k == "batch_tile_rev32") *value = g.batch_tile_rev[1];
    else if (k == "batch_tile_rev64") *value = g.batch_tile_rev[2];
    else return fail(ESIM_EINVAL, "unknown option '" + k + "'");
    return ESIM_OK;
}

esim_status esim_query(esim_graph* h, int64_t u, double c, double eps, uint64_t seed, double* s_out) {
    if (check_graph(h)) return ESIM_EINVAL;
    if (!s_out) return fail(ESIM_EINVAL, "s_out is NULL");
    return run_query(h->g, u, c, eps, seed, nullptr, 0, nullptr, nullptr, s_out, nullptr, nullptr);
}

esim_status esim_query_device(esim_graph* h, int64_t u, double c, double eps, uint64_t seed, double* s_dev) {
    if (check_graph(h)) return ESIM_EINVAL;
    if (!s_dev) return fail(ESIM_EINVAL, "s_dev is NULL");
    return run_query(h->g, u, c, eps, seed, s_dev, 0, nullptr, nullptr, nullptr, nullptr, nullptr);
}

esim_status esim_topk(esim_graph* h, int64_t u, double c, double eps, uint64_t seed, int32_t k, int32_t* ids_out,
                      double* scores_out) {
    if (check_graph(h)) return ESIM_EINVAL;
    if (k < 1) return fail(ESIM_EINVAL, "k must be >= 1");
    if (!ids_out || !scores_out) return fail(ESIM_EINVAL, "NULL output");
    return run_query(h->g, u, c, eps, seed, nullptr, k, nullptr, nullptr, nullptr, ids_out, scores_out);
}

esim_status esim_topk_device(esim_graph* h, int64_t u, double c, double eps, uint64_t seed, int32_t k,
                             int32_t* ids_dev, double* scores_dev) {
    if (check_graph(h)) return ESIM_EINVAL;
    if (k < 1) return fail(ESIM_EINVAL, "k must be >= 1");
    if (!ids_dev || !scores_dev) return fail(ESIM_EINVAL, "NULL output");
    return run_query(h->g, u, c, eps, seed, nullptr, k, ids_dev, scores_dev, nullptr, nullptr, nullptr);
}

esim_status esim_last_stats(const esim_graph* h, esim_query_stats* out) {
    if (check_graph(h)) return ESIM_EINVAL;
    if (!out) return fail(ESIM_EINVAL, "out is NULL");
    const Graph& g = h->g;
    memset(out, 0, sizeof(*out));
    out->L = g.last_L;
    out->launches = g.last_launches;
    out->R_b = g.last_R_b;
    out->kappa = g.last_kappa;
    out->pi_norm2 = g.last_norm2;
    out->sum_R = g.last_sum_R;
    out->pair_steps = g.last_steps;
    out->ms_forward = g.last_ms[0];
    out->ms_allocate = g.last_ms[1];
    out->ms_sample = g.last_ms[2];
    out->ms_reverse = g.last_ms[3];
    out->ms_topk = g.last_ms[4];
    out->ms_total = g.last_ms[5];
    out->ms_sample_kernel = g.last_ms_kernel;
    out->ms_sample_side = g.last_ms_side;
    out->pair_steps_side = g.last_steps_side;
    out->side_candidates = g.last_side_candidates;
    out->alg3_nodes = g.last_alg3_nodes;
    out->hist_entries = g.last_hist_entries;
    out->workspace_bytes = g.last_ws_bytes;
    return ESIM_OK;
}

esim_status esim_forward(esim_graph* h, int64_t u, double c, int32_t L, double* hist) {
    if (check_graph(h)) return ESIM_EINVAL;
    Graph& g = h->g;
    if (u < 0 || u >= g.n) return fail(ESIM_EINVAL, "source node out of range");
    if (!(c > 0.0 && c < 1.0)) return fail(ESIM_EINVAL, "need 0 < c < 1");
    if (L < 0 || L > 4096) return fail(ESIM_EINVAL, "need 0 <= L <= 4096");
    if (!hist) return fail(ESIM_EINVAL, "hist is NULL");
    ESIM_CUDA_TRY(cudaSetDevice(g.device), "cudaSetDevice");
    Ws w;
    esim_status st = ensure_ws(g, 0, 0, w);
    if (st != ESIM_OK) return st;
    ESIM_CUDA_TRY(launch_forward(g, u, c, L, hist, w.xa, w.xb), "forward sweeps");
    return ESIM_OK;
}

esim_status esim_allocate(esim_graph* h, const double* hist, int32_t L, double R_b, int32_t mode, double* pi_out,
                          uint64_t* R_out, uint64_t* off) {
    if (check_graph(h)) return ESIM_EINVAL;
    Graph& g = h->g;
    if (!hist || !R_out || !off) return fail(ESIM_EINVAL, "NULL argument");
    if (L < 0 || L > 4096) return fail(ESIM_EINVAL, "need 0 <= L <= 4096");
    if (mode != 0 && mode != 1) return fail(ESIM_EINVAL, "mode must be 0 or 1");
    if (!(R_b >= 0.0)) return fail(ESIM_EINVAL, "need R_b >= 0");
    ESIM_CUDA_TRY(cudaSetDevice(g.device), "cudaSetDevice");
    ESIM_CUDA_TRY(cudaMemsetAsync(scan_ticket(g), 0, sizeof(unsigned), g.stream), "reset ticket");
    ESIM_CUDA_TRY(launch_allocate(g, hist, L, R_b, mode, pi_out, R_out, off), "allocation");
    return ESIM_OK;
}

esim_status esim_sample(esim_graph* h, const uint64_t* off, double c, uint64_t seed, uint64_t* nonmeet,
                        uint64_t* pair_steps) {
    if (check_graph(h)) return ESIM_EINVAL;
    Graph& g = h->g;
    if (!off || !nonmeet) return fail(ESIM_EINVAL, "NULL argument");
    if (!(c > 0.0 && c < 1.0)) return fail(ESIM_EINVAL, "need 0 < c < 1");
    ESIM_CUDA_TRY(cudaSetDevice(g.device), "cudaSetDevice");
    return sample_step(g, off, c, seed, nonmeet, pair_steps, nullptr);
}

esim_status esim_dhat(esim_graph* h, const uint64_t* nonmeet, const uint64_t* off, double* dhat) {
    if (check_graph(h)) return ESIM_EINVAL;
    Graph& g = h->g;
    if (!nonmeet || !off || !dhat) return fail(ESIM_EINVAL, "NULL argument");
    ESIM_CUDA_TRY(cudaSetDevice(g.device), "cudaSetDevice");
    ESIM_CUDA_TRY(launch_dhat(g, nonmeet, off, dhat), "dhat");
    return ESIM_OK;
}

esim_status esim_reverse(esim_graph* h, const double* hist, int32_t L, double c, const double* dhat, double* s_out) {
    if (check_graph(h)) return ESIM_EINVAL;
    Graph& g = h->g;
    if (!hist || !dhat || !s_out) return fail(ESIM_EINVAL, "NULL argument");
    if (L < 0 || L > 4096) return fail(ESIM_EINVAL, "need 0 <= L <= 4096");
    if (!(c > 0.0 && c < 1.0)) return fail(ESIM_EINVAL, "need 0 < c < 1");
    ESIM_CUDA_TRY(cudaSetDevice(g.device), "cudaSetDevice");
    Ws w;
    esim_status st = ensure_ws(g, 0, 0, w);
    if (st != ESIM_OK) return st;
    ESIM_CUDA_TRY(launch_reverse(g, hist, L, c, dhat, s_out, w.xa, w.xb), "reverse sweeps");
    return ESIM_OK;
}

esim_status esim_select_topk(esim_graph* h, const double* scores, int64_t exclude, int32_t k, int32_t* ids_out,
                             double* vals_out) {
    if (check_graph(h)) return ESIM_EINVAL;
    Graph& g = h->g;
    if (!scores || !ids_out || !vals_out) return fail(ESIM_EINVAL, "NULL argument");
    if (k < 1) return fail(ESIM_EINVAL, "k must be >= 1");
    if (k > kTopkMax) return fail(ESIM_ENOTSUP, "k above 4096");
    if (exclude < -1 || exclude >= g.n) return fail(ESIM_EINVAL, "exclude out of range");
    ESIM_CUDA_TRY(cudaSetDevice(g.device), "cudaSetDevice");
    ESIM_CUDA_TRY(cudaMemsetAsync(topk_tickets(g), 0, 2 * sizeof(unsigned), g.stream), "reset tickets");
    ESIM_CUDA_TRY(launch_topk(g, scores, exclude, k, ids_out, vals_out, g.topk_ws), "top-k");
    return ESIM_OK;
}

esim_status esim_forward_f32(esim_graph* h, int64_t u, double c, int32_t L, float* hist) {
    if (check_graph(h)) return ESIM_EINVAL;
    Graph& g = h->g;
    if (u < 0 || u >= g.n) return fail(ESIM_EINVAL, "source node out of range");
    if (!(c > 0.0 && c < 1.0)) return fail(ESIM_EINVAL, "need 0 < c < 1");
    if (L < 0 || L > 4096) return fail(ESIM_EINVAL, "need 0 <= L <= 4096");
    if (!hist) return fail(ESIM_EINVAL, "hist is NULL");
    ESIM_CUDA_TRY(cudaSetDevice(g.device), "cudaSetDevice");
    Ws w;
    esim_status st = ensure_ws(g, 0, 1, w);
    if (st != ESIM_OK) return st;
    ESIM_CUDA_TRY(launch_forward32(g, u, c, L, hist, w.xa32, w.xb32), "forward sweeps (FP32c)");
    return ESIM_OK;
}

esim_status esim_allocate_f32(esim_graph* h, const float* hist, int32_t L, double R_b, int32_t mode, double* pi_out,
                              uint64_t* R_out, uint64_t* off) {
    if (check_graph(h)) return ESIM_EINVAL;
    Graph& g = h->g;
    if (!hist || !R_out || !off) return fail(ESIM_EINVAL, "NULL argument");
    if (L < 0 || L > 4096) return fail(ESIM_EINVAL, "need 0 <= L <= 4096");
    if (mode != 0 && mode != 1) return fail(ESIM_EINVAL, "mode must be 0 or 1");
    if (!(R_b >= 0.0)) return fail(ESIM_EINVAL, "need R_b >= 0");
    ESIM_CUDA_TRY(cudaSetDevice(g.device), "cudaSetDevice");
    ESIM_CUDA_TRY(cudaMemsetAsync(scan_ticket(g), 0, sizeof(unsigned), g.stream), "reset ticket");
    ESIM_CUDA_TRY(launch_allocate32(g, hist, L, R_b, mode, pi_out, R_out, off), "allocation (FP32c)");
    return ESIM_OK;
}

esim_status esim_reverse_f32(esim_graph* h, const float* hist, int32_t L, double c, const double* dhat,
                             double* s_out) {
    if (check_graph(h)) return ESIM_EINVAL;
    Graph& g = h->g;
    if (!hist || !dhat || !s_out) return fail(ESIM_EINVAL, "NULL argument");
    if (L < 0 || L > 4096) return fail(ESIM_EINVAL, "need 0 <= L <= 4096");
    if (!(c > 0.0 && c < 1.0)) return fail(ESIM_EINVAL, "need 0 < c < 1");
    ESIM_CUDA_TRY(cudaSetDevice(g.device), "cudaSetDevice");
    Ws w;
    esim_status st = ensure_ws(g, 0, 1, w);
    if (st != ESIM_OK) return st;
    ESIM_CUDA_TRY(launch_reverse32(g, hist, L, c, dhat, s_out, w.w2, w.sa2, w.sb2), "reverse sweeps (FP32c)");
    return ESIM_OK;
}

esim_status esim_query_batch(esim_graph* h, int32_t B, const int64_t* u, const double* eps, uint64_t seed, double c,
                             double* s_out) {
    if (check_graph(h)) return ESIM_EINVAL;
    if (!s_out) return fail(ESIM_EINVAL, "s_out is NULL");
    return run_batch(h->g, B, u, eps, seed, c, nullptr, s_out, 0, nullptr, nullptr, nullptr, nullptr);
}

esim_status esim_query_batch_device(esim_graph* h, int32_t B, const int64_t* u, const double* eps, uint64_t seed,
                                    double c, double* s_dev) {
    if (check_graph(h)) return ESIM_EINVAL;
    if (!s_dev) return fail(ESIM_EINVAL, "s_dev is NULL");
    return run_batch(h->g, B, u, eps, seed, c, s_dev, nullptr, 0, nullptr, nullptr, nullptr, nullptr);
}

esim_status esim_topk_batch(esim_graph* h, int32_t B, const int64_t* u, const double* eps, uint64_t seed, double c,
                            int32_t k, int32_t* ids_out, double* scores_out) {
    if (check_graph(h)) return ESIM_EINVAL;
    if (k < 1) return fail(ESIM_EINVAL, "k must be >= 1");
    if (!ids_out || !scores_out) return fail(ESIM_EINVAL, "NULL output");
    return run_batch(h->g, B, u, eps, seed, c, nullptr, nullptr, k, nullptr, nullptr, ids_out, scores_out);
}

esim_status esim_topk_batch_device(esim_graph* h, int32_t B, const int64_t* u, const double* eps, uint64_t seed,
                                   double c, int32_t k, int32_t* ids_dev, double* scores_dev) {
    if (check_graph(h)) return ESIM_EINVAL;
    if (k < 1) return fail(ESIM_EINVAL, "k must be >= 1");
    if (!ids_dev || !scores_dev) return fail(ESIM_EINVAL, "NULL output");
    return run_batch(h->g, B, u, eps, seed, c, nullptr, nullptr, k, ids_dev, scores_dev, nullptr, nullptr);
}

esim_status esim_alg3_first_meeting(esim_graph* h, int64_t k, int32_t depth, double c, double* z_out) {
    if (check_graph(h)) return ESIM_EINVAL;
    Graph& g = h->g;
    if (k < 0 || k >= g.n) return fail(ESIM_EINVAL, "node out of range");
    if (depth < 1 || depth > kAlg3MaxDepth) return fail(ESIM_EINVAL, "need 1 <= depth <= 16");
    if (!(c > 0.0 && c < 1.0)) return fail(ESIM_EINVAL, "need 0 < c < 1");
    if (!z_out) return fail(ESIM_EINVAL, "z_out is NULL");
    if (g.has_duplicates) return fail(ESIM_ENOTSUP, "Algorithm 3 needs a graph without repeated in-edges");
    ESIM_CUDA_TRY(cudaSetDevice(g.device), "cudaSetDevice");
    esim_status a3 = ensure_a3ws(g);
    if (a3 != ESIM_OK) return a3;
    ESIM_CUDA_TRY(alg3_first_meeting(g, k, depth, c, g.a3ws, &g.a3ws_clean, z_out, nullptr), "Algorithm 3 first meetings");
    return ESIM_OK;
}

esim_status esim_alg3_paper_depth(esim_graph* h, const uint64_t* R, double c, int32_t max_depth, uint8_t* depth) {
    if (check_graph(h)) return ESIM_EINVAL;
    Graph& g = h->g;
    if (!R || !depth) return fail(ESIM_EINVAL, "NULL argument");
    if (!(c > 0.0 && c < 1.0)) return fail(ESIM_EINVAL, "need 0 < c < 1");
    if (max_depth < 0 || max_depth > kAlg3MaxDepth) return fail(ESIM_EINVAL, "need 0 <= max_depth <= 16");
    ESIM_CUDA_TRY(cudaSetDevice(g.device), "cudaSetDevice");
    esim_status a3 = ensure_a3pws(g);
    if (a3 != ESIM_OK) return a3;
    ESIM_CUDA_TRY(alg3_paper_depths(g, R, c, max_depth, g.a3pws, g.a3pws_bytes, depth, nullptr), "Algorithm 3 depths (explored edges)");
    return ESIM_OK;
}

esim_status esim_alg3_zsum(esim_graph* h, const uint8_t* depth, double c, double* zsum) {
    if (check_graph(h)) return ESIM_EINVAL;
    Graph& g = h->g;
    if (!depth || !zsum) return fail(ESIM_EINVAL, "NULL argument");
    if (!(c > 0.0 && c < 1.0)) return fail(ESIM_EINVAL, "need 0 < c < 1");
    if (g.has_duplicates) return fail(ESIM_ENOTSUP, "Algorithm 3 needs a graph without repeated in-edges");
    ESIM_CUDA_TRY(cudaSetDevice(g.device), "cudaSetDevice");
    int launches = 0, used = 0;
    return alg3_zsums(g, depth, c, zsum, &launches, &used);
}

int32_t esim_alg3_depth(double v, double c, const uint64_t* supp, int32_t max_depth, int64_t n, int64_t m,
                        double w_sweep, double w_probe, double w_launch, double w_last) {
    if (!supp || !(c > 0.0 && c < 1.0) || max_depth < 0 || max_depth > kAlg3MaxDepth || n < 1 || m < 0 ||
        !(v >= 0.0) || !(w_sweep >= 0.0) || !(w_probe >= 0.0) || !(w_launch >= 0.0) || !(w_last >= 0.0))
        return -1;
    return alg3_depth(v, c, supp, max_depth, n, m, w_sweep, w_probe, w_launch, w_last);
}

esim_status esim_sample_depth(esim_graph* h, const uint64_t* off, const uint8_t* depth, double c, uint64_t seed,
                              uint64_t* counts, uint64_t* pair_steps) {
    if (check_graph(h)) return ESIM_EINVAL;
    Graph& g = h->g;
    if (!off || !counts) return fail(ESIM_EINVAL, "NULL argument");
    if (!(c > 0.0 && c < 1.0)) return fail(ESIM_EINVAL, "need 0 < c < 1");
    ESIM_CUDA_TRY(cudaSetDevice(g.device), "cudaSetDevice");
    return sample_step(g, off, c, seed, counts, pair_steps, depth);
}

esim_status esim_dhat_alg3(esim_graph* h, const uint64_t* counts, const uint64_t* off, const uint8_t* depth,
                           const double* zsum, double c, double* dhat) {
    if (check_graph(h)) return ESIM_EINVAL;
    Graph& g = h->g;
    if (!counts || !off || !depth || !zsum || !dhat) return fail(ESIM_EINVAL, "NULL argument");
    if (!(c > 0.0 && c < 1.0)) return fail(ESIM_EINVAL, "need 0 < c < 1");
    ESIM_CUDA_TRY(cudaSetDevice(g.device), "cudaSetDevice");
    ESIM_CUDA_TRY(launch_dhat_alg3(g, counts, off, depth, zsum, c, dhat), "dhat (Algorithm 3)");
    return ESIM_OK;
}

esim_status esim_sync(esim_graph* h) {
    if (check_graph(h)) return ESIM_EINVAL;
    Graph& g = h->g;
    ESIM_CUDA_TRY(cudaSetDevice(g.device), "cudaSetDevice");
    ESIM_CUDA_TRY(cudaMemcpyAsync(g.status_host, g.status, sizeof(Status), cudaMemcpyDeviceToHost, g.stream),
                  "copy status");
    ESIM_CUDA_TRY(cudaStreamSynchronize(g.stream), "stream synchronize");
    const int err = g.status_host->err;
    ESIM_CUDA_TRY(cudaMemsetAsync(g.status, 0, sizeof(Status), g.stream), "reset status");
    ESIM_CUDA_TRY(cudaStreamSynchronize(g.stream), "stream synchronize");
    if (err & kErrBudget) return fail(ESIM_EBUDGET, "pair budget exceeded or R(k) overflow");
    if (err & kErrTimeout) return fail(ESIM_ETIMEOUT, "device wait timed out");
    return ESIM_OK;
}

}  // extern "C"
