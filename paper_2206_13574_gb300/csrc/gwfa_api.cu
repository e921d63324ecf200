// gwfa_api.cu -- host side of the C ABI declared in include/gwfa.h.
//
// Graph upload (packing, arc merging, CSR), the plain one-query path, the
// engine (per-CTA slabs in tiers, retry lists) and the batch entry points.
// Every step of the alignment itself runs in the kernels of gwfa_kernels.cu.
#include <cuda_runtime.h>
#include <stdint.h>
#include <string.h>

#include <algorithm>
#include <cmath>
#include <mutex>
#include <new>
#include <utility>
#include <vector>

#include "gwfa_internal.cuh"

using gwfa::TierArgs;

namespace {

int host_code(char c) {
    switch (c) {
    case 'A': case 'a': return 0;
    case 'C': case 'c': return 1;
    case 'G': case 'g': return 2;
    case 'T': case 't': return 3;
    default: return -1;
    }
}

template <class T>
int dmalloc(T **p, uint64_t bytes) {
    if (bytes == 0) bytes = 16;
    if (cudaMalloc((void **)p, bytes) != cudaSuccess) {
        cudaGetLastError();
        *p = nullptr;
        return GWFA_ERR_OOM;
    }
    return GWFA_OK;
}

int cuda_status(cudaError_t e) {
    if (e == cudaSuccess) return GWFA_OK;
    if (e == cudaErrorMemoryAllocation) return GWFA_ERR_OOM;
    return GWFA_ERR_CUDA;
}

// Grow-only device buffer.
int ensure(uint8_t **buf, uint64_t *have, uint64_t need) {
    if (*have >= need) return GWFA_OK;
    if (*buf) cudaFree(*buf);
    *buf = nullptr;
    *have = 0;
    uint64_t want = std::max<uint64_t>(need, 1 << 20);
    if (dmalloc(buf, want)) return GWFA_ERR_OOM;
    *have = want;
    return GWFA_OK;
}

// Host reachability v_s -> v_e (Def. 2 assumes it; the paper's loop never ends otherwise).
// Breadth first: v_e is about as many vertices away as the query has, while depth first runs
// to the far end of the graph before it looks beside its way.  `seen` holds the number of
// the call that reached a vertex last, so nothing is cleared (both guarded by g->mu).
bool reachable(const gwfa_graph *g, uint32_t vs, uint32_t ve) {
    if (vs == ve) return true;
    if (g->seen.size() != g->nv || ++g->seen_call == 0) {
        g->seen.assign(g->nv, 0);
        g->seen_call = 1;
    }
    std::vector<uint32_t> &q = g->bfs;
    q.clear();
    q.push_back(vs);
    g->seen[vs] = g->seen_call;
    for (size_t head = 0; head < q.size(); ++head) {
        const uint32_t v = q[head];
        for (uint32_t a = g->h_arc_off[v]; a < g->h_arc_off[v + 1]; ++a) {
            const uint32_t u = g->h_arc_dst[a];
            if (u == ve) return true;
            if (g->seen[u] != g->seen_call) {
                g->seen[u] = g->seen_call;
                q.push_back(u);
            }
        }
    }
    return false;
}

// 2-bit packing of a query on the host, as pack_kernel does it; false for a base other
// than A/C/G/T.  (n + 15) / 16 words.
bool pack_host(const char *q, uint32_t n, uint32_t *w) {
    static const struct Lut {
        uint8_t c[256];
        Lut() {
            for (int i = 0; i < 256; ++i) c[i] = 4;
            for (int i = 0; i < 4; ++i) c[(uint8_t)"ACGT"[i]] = c[(uint8_t)"acgt"[i]] = (uint8_t)i;
        }
    } lut;
    uint32_t bad = 0;
    for (uint32_t p = 0; p < n; p += 16) {
        uint32_t x = 0;
        const uint32_t e = std::min(n - p, 16u);
        for (uint32_t i = 0; i < e; ++i) {
            const uint32_t c = lut.c[(uint8_t)q[p + i]];
            bad |= c;
            x |= (c & 3u) << (2 * i);
        }
        w[p >> 4] = x;
    }
    return (bad & 4u) == 0;
}

// Grow-only pinned host buffer, mapped into the device's address space.
int ensure_pinned(uint8_t **buf, uint64_t *have, uint64_t need) {
    if (*have >= need) return GWFA_OK;
    if (*buf) cudaFreeHost(*buf);
    *buf = nullptr;
    *have = 0;
    const uint64_t want = std::max<uint64_t>(need, 64 << 10);
    if (cudaHostAlloc((void **)buf, want, cudaHostAllocMapped | cudaHostAllocPortable) != cudaSuccess) {
        cudaGetLastError();
        *buf = nullptr;
        return GWFA_ERR_OOM;
    }
    *have = want;
    return GWFA_OK;
}

struct Carve {
    uint8_t *base;
    uint64_t off = 0;
    template <class T> T *take(uint64_t bytes) {
        T *p = (T *)(base + off);
        off = gwfa::align256(off + bytes);
        return p;
    }
};

// Host-buffer batches up to this many bytes of inputs go over in one copy.
constexpr uint64_t kStagedBatch = 256 << 10;

// Mean lengths from which n queries get 1024 and 512 threads each, see auto_threads.
uint64_t wide_from(uint64_t n, int sms) { return 600 * n / (uint64_t)sms; }
uint64_t mid_from(uint64_t n, int sms) { return 180 * n / (uint64_t)sms; }

// Width of tier 0's CTAs for n queries of `len` bases on average, where the configuration
// leaves it to the engine.  A wide CTA shortens a query, a
// narrow one wastes fewer warps on small frontiers and at barriers: few queries are bound
// by their longest, many by throughput, and a frontier grows with the length.  Measured
// crossings, 1024 -> 512 -> 256 threads (ms at 1024 / 512 / 256): 1-20 kb reads, 6.4 kb on
// average, n = 1000: 8.4 / 10.4 / 17.6, 1500: 12.1 / 12.3 / 21.0, 2500: 19.6 / 12.5 / 21.2,
// 5000: 38.7 / 23.8 / 25.3, 7000: 54 / 33.5 / 28.2; 0.5-5 kb, 2.0 kb on average, n = 600:
// 1.27 / 1.33 / 1.57, 1000: 1.84 / 1.40 / 1.64, 2500: 4.5 / 2.40 / 2.12; 1 kb, n = 1000:
// 0.58 / 0.33 / 0.20.
// Lag pruning keeps the frontier near 0.03 tiles per unit of lag, whatever the length
// (lag 1000, 1024 / 256 / 128 threads, n = 150: 9.0 / 9.1 / 9.8, 400: 24.4 / 9.4 / 10.5,
// 1000: 56 / 17.4 / 11.1; lag 4000: 15.3 / 20.1 / 25.7, 40.6 / 20.3 / 28.1, 93 / 38 / 32).
uint32_t auto_threads(uint64_t n, uint64_t len, int sms, int max_lag) {
    const uint64_t m = (uint64_t)sms;
    if (max_lag > 0) return n <= m && max_lag > 2000 ? 1024u : n <= 4 * m ? 256u : 128u;
    return len >= wide_from(n, sms) ? 1024u : len >= mid_from(n, sms) ? 512u : gwfa::kNarrow;
}

uint64_t words_for(uint32_t nq, uint64_t nbases) { return (nbases >> 4) + nq + 2; }

}  // namespace

extern "C" {

const char *gwfa_strerror(int s) {
    switch (s) {
    case GWFA_OK: return "ok";
    case GWFA_PENDING: return "pending";
    case GWFA_ERR_INVALID: return "invalid argument";
    case GWFA_ERR_OOM: return "out of memory";
    case GWFA_ERR_CUDA: return "CUDA error";
    case GWFA_ERR_UNREACHABLE: return "end vertex not reachable from start vertex";
    case GWFA_ERR_EMPTY_FRONTIER: return "pruning emptied the wavefront";
    case GWFA_ERR_CAPACITY: return "workspace capacity exceeded";
    case GWFA_ERR_TIMEOUT: return "device wait timed out";
    case GWFA_ERR_SCORE_LIMIT: return "edit distance above max_score";
    case GWFA_ERR_NOT_RUN: return "query not run";
    default: return "unknown status";
    }
}

int gwfa_graph_create(uint32_t nv, const char *h_seq, const uint64_t *h_seq_off, uint64_t na,
                      const uint32_t *h_arc_src, const uint32_t *h_arc_dst, int device,
                      gwfa_graph **out) {
    gwfa::Range range_("gwfa_graph_create");
    if (!out || !h_seq_off || (nv > 0 && !h_seq) || (na > 0 && (!h_arc_src || !h_arc_dst)))
        return GWFA_ERR_INVALID;
    *out = nullptr;
    if (nv == 0 || nv >= 0x7FFFFFFFu) return GWFA_ERR_INVALID;
    // labels: non-empty, ACGT, 2-bit packed, each vertex on a word boundary
    std::vector<uint32_t> vstart(nv), vlen(nv);
    uint64_t nwords = 0, total = 0;
    for (uint32_t v = 0; v < nv; ++v) {
        if (h_seq_off[v + 1] <= h_seq_off[v]) return GWFA_ERR_INVALID;
        uint64_t L = h_seq_off[v + 1] - h_seq_off[v];
        if (L >= (1ull << 30)) return GWFA_ERR_INVALID;
        vlen[v] = (uint32_t)L;
        vstart[v] = (uint32_t)nwords;
        nwords += (L + 15) >> 4;
        total += L;
        if (nwords >= 0xFFFFFFF0ull) return GWFA_ERR_INVALID;
    }
    std::vector<uint32_t> words(nwords + 2, 0);
    for (uint32_t v = 0; v < nv; ++v) {
        const char *s = h_seq + h_seq_off[v];
        uint32_t *w = words.data() + vstart[v];
        for (uint32_t p = 0; p < vlen[v]; ++p) {
            int c = host_code(s[p]);
            if (c < 0) return GWFA_ERR_INVALID;
            w[p >> 4] |= (uint32_t)c << (2 * (p & 15));
        }
    }
    // arcs: validate, merge duplicates, CSR by source
    std::vector<std::pair<uint32_t, uint32_t>> arcs(na);
    int has_cycles = 0;
    for (uint64_t a = 0; a < na; ++a) {
        if (h_arc_src[a] >= nv || h_arc_dst[a] >= nv) return GWFA_ERR_INVALID;
        arcs[a] = {h_arc_src[a], h_arc_dst[a]};
        if (h_arc_dst[a] <= h_arc_src[a]) has_cycles = 1;
    }
    std::sort(arcs.begin(), arcs.end());
    arcs.erase(std::unique(arcs.begin(), arcs.end()), arcs.end());
    gwfa_graph *g = new (std::nothrow) gwfa_graph();
    if (!g) return GWFA_ERR_OOM;
    g->device = device;
    g->nv = nv;
    g->na = arcs.size();
    g->total = total;
    g->n_words = nwords + 2;
    g->has_cycles = has_cycles;
    g->h_arc_off.assign(nv + 1, 0);
    g->h_arc_dst.resize(arcs.size());
    for (auto &a : arcs) g->h_arc_off[a.first + 1]++;
    for (uint32_t v = 0; v < nv; ++v) {
        g->max_outdeg = std::max(g->max_outdeg, g->h_arc_off[v + 1]);
        g->h_arc_off[v + 1] += g->h_arc_off[v];
    }
    for (size_t a = 0; a < arcs.size(); ++a) g->h_arc_dst[a] = arcs[a].second;
    g->h_vlen = vlen;

    int st = cuda_status(cudaSetDevice(device));
    if (st) { delete g; return st; }
    std::vector<uint4> vinfo(nv);
    for (uint32_t v = 0; v < nv; ++v)
        vinfo[v] = make_uint4(vstart[v], vlen[v], g->h_arc_off[v], g->h_arc_off[v + 1]);
    std::vector<uint4> vx(2 * (uint64_t)nv);
    for (uint32_t v = 0; v < nv; ++v) {
        uint32_t dst[4] = {0, 0, 0, 0};
        for (uint32_t a = 0; a < 4 && g->h_arc_off[v] + a < g->h_arc_off[v + 1]; ++a)
            dst[a] = g->h_arc_dst[g->h_arc_off[v] + a];
        vx[2 * (uint64_t)v] = vinfo[v];
        vx[2 * (uint64_t)v + 1] = make_uint4(dst[0], dst[1], dst[2], dst[3]);
    }
    st = dmalloc(&g->d_words, g->n_words * 4);
    if (!st) st = dmalloc(&g->d_vx, vx.size() * sizeof(uint4));
    if (!st) st = cuda_status(cudaMemcpy(g->d_vx, vx.data(), vx.size() * sizeof(uint4), cudaMemcpyHostToDevice));
    if (!st) st = dmalloc(&g->d_vinfo, (uint64_t)nv * sizeof(uint4));
    if (!st) st = dmalloc(&g->d_arc_dst, std::max<uint64_t>(g->na, 1) * 4);
    if (!st) st = cuda_status(cudaMemcpy(g->d_words, words.data(), g->n_words * 4, cudaMemcpyHostToDevice));
    if (!st) st = cuda_status(cudaMemcpy(g->d_vinfo, vinfo.data(), (uint64_t)nv * sizeof(uint4), cudaMemcpyHostToDevice));
    if (!st && g->na) st = cuda_status(cudaMemcpy(g->d_arc_dst, g->h_arc_dst.data(), g->na * 4, cudaMemcpyHostToDevice));
    if (!st) st = cuda_status(cudaStreamCreateWithFlags(&g->stream, cudaStreamNonBlocking));
    g->device_bytes = g->n_words * 4 + 3 * (uint64_t)nv * sizeof(uint4) + g->na * 4;
    if (st) { gwfa_graph_destroy(g); return st; }
    *out = g;
    return GWFA_OK;
}

int gwfa_graph_destroy(gwfa_graph *g) {
    if (!g) return GWFA_ERR_INVALID;
    cudaSetDevice(g->device);
    cudaFree(g->d_words);
    cudaFree(g->d_vinfo);
    cudaFree(g->d_vx);
    cudaFree(g->d_arc_dst);
    cudaFree(g->plain_slab);
    cudaFree(g->plain_stage);
    if (g->plain_host) cudaFreeHost(g->plain_host);
    if (g->stream) cudaStreamDestroy(g->stream);
    delete g;
    return GWFA_OK;
}

int gwfa_graph_get_info(const gwfa_graph *g, gwfa_graph_info *o) {
    if (!g || !o) return GWFA_ERR_INVALID;
    o->n_vertices = g->nv;
    o->max_out_degree = g->max_outdeg;
    o->n_arcs = g->na;
    o->total_bases = g->total;
    o->device_bytes = g->device_bytes;
    o->device = g->device;
    o->has_cycles = g->has_cycles;
    return GWFA_OK;
}

// ---------------------------------------------------------------- plain path

static int align_plain(const gwfa_graph *g, const char *h_q, uint32_t n, uint32_t vs, uint32_t ve,
                       const gwfa_opts &o, gwfa_result *out, uint32_t *h_path, uint32_t path_cap,
                       uint32_t *path_len);

// formulation variant flags: known bits only, and not combined with pruning; the
// memory bound on H~ needs pruning and the walk base in the payload (no traceback)
static bool ends_ok(const gwfa_opts &o) {
    return (o.ends & ~(GWFA_FREE_START | GWFA_FREE_END | GWFA_EXTEND)) == 0 && (o.ends == 0 || o.max_lag == 0) &&
           o.evict_lag >= 0 && o.evict_every >= 0 && (o.evict_lag == 0 || (o.max_lag > 0 && !o.traceback));
}

int gwfa_align(const gwfa_graph *g, const char *h_q, uint32_t n, uint32_t vs, uint32_t ve,
               const gwfa_opts *opts, gwfa_result *out) {
    gwfa_opts o = opts ? *opts : gwfa_opts{0, 0, -1, 0};
    if (o.traceback != 0) return GWFA_ERR_INVALID;   // the walk needs gwfa_align_path
    return align_plain(g, h_q, n, vs, ve, o, out, nullptr, 0, nullptr);
}

int gwfa_align_path(const gwfa_graph *g, const char *h_q, uint32_t n, uint32_t vs, uint32_t ve,
                    const gwfa_opts *opts, gwfa_result *out, uint32_t *h_path, uint32_t path_cap,
                    uint32_t *path_len) {
    gwfa_opts o = opts ? *opts : gwfa_opts{0, 0, -1, 0};
    if (!path_len || (path_cap && !h_path)) return GWFA_ERR_INVALID;
    o.traceback = 1;
    return align_plain(g, h_q, n, vs, ve, o, out, h_path, path_cap, path_len);
}

static int align_plain(const gwfa_graph *g, const char *h_q, uint32_t n, uint32_t vs, uint32_t ve,
                       const gwfa_opts &o, gwfa_result *out, uint32_t *h_path, uint32_t path_cap,
                       uint32_t *path_len) {
    gwfa::Range range_(o.traceback ? "gwfa_align_path" : "gwfa_align");
    if (!g || !out || (n > 0 && !h_q)) return GWFA_ERR_INVALID;
    memset(out, 0, sizeof(*out));
    out->edit_distance = -1;
    if (path_len) *path_len = 0;
    if (o.ends & GWFA_EXTEND) ve = vs;   // no end vertex
    if (vs >= g->nv || ve >= g->nv || o.max_lag < 0 || n >= 0x7FFFFFFFu || !ends_ok(o)) {
        out->status = GWFA_ERR_INVALID;
        return GWFA_ERR_INVALID;
    }
    std::lock_guard<std::mutex> lk(g->mu);
    if (!reachable(g, vs, ve)) {
        out->status = GWFA_ERR_UNREACHABLE;
        return GWFA_OK;
    }
    int st = cuda_status(cudaSetDevice(g->device));
    if (st) return st;
    const bool prune = o.max_lag > 0 || o.traceback;   // 64-bit values (walk base) and trace words
    // A short call is bound by its launches and copies (one 1 kb read took 118 us with four copies
    // in, a clear, a packing kernel and a copy out, of which the alignment is about 70), so the
    // inputs go over in one copy from pinned memory, packed here, and the result comes back in
    // pinned memory that the kernel writes itself: 97 us.
    //   staged: q_off[2] | v_s | v_e | work counter | words;  pinned only: result, path_len
    const uint64_t in_bytes = 64 + words_for(1, n) * 4;
    const uint64_t res_off = gwfa::align256(in_bytes);
    st = ensure_pinned(&g->plain_host, &g->plain_host_bytes, res_off + 256);
    if (st) return st;
    struct In {
        uint64_t off[2];
        uint32_t vs, ve, head, pad;
    };
    static_assert(sizeof(In) <= 64, "words start at byte 64");
    In *in = (In *)g->plain_host;
    uint32_t *h_words = (uint32_t *)(g->plain_host + 64);
    *in = In{{0, n}, vs, ve, 0u, 0u};
    if (!pack_host(h_q, n, h_words)) {
        out->status = GWFA_ERR_INVALID;
        return GWFA_OK;
    }
    for (uint64_t w = ((uint64_t)n + 15) >> 4; w < words_for(1, n); ++w) h_words[w] = 0;
    st = ensure(&g->plain_stage, &g->plain_stage_bytes, gwfa::align256(in_bytes) + (uint64_t)path_cap * 4);
    if (st) return st;
    In *d_in = (In *)g->plain_stage;
    uint32_t *d_path = (uint32_t *)(g->plain_stage + gwfa::align256(in_bytes));
    gwfa_result *h_res = (gwfa_result *)(g->plain_host + res_off);
    uint32_t *h_plen = (uint32_t *)(h_res + 1);
    void *d_res = nullptr, *d_plen = nullptr;
    st = cuda_status(cudaHostGetDevicePointer(&d_res, h_res, 0));
    if (!st) st = cuda_status(cudaHostGetDevicePointer(&d_plen, h_plen, 0));
    if (st) return st;
    cudaStream_t s = g->stream;
    uint32_t log2 = g->plain_log2 && g->plain_prune == prune ? g->plain_log2 : (prune ? 15u : 16u);
    for (;;) {
        if (!g->plain_slab || g->plain_log2 != log2 || g->plain_prune != prune) {
            cudaFree(g->plain_slab);
            g->plain_slab = nullptr;
            const uint64_t bytes = gwfa::slab_layout(log2, prune).total;
            st = dmalloc(&g->plain_slab, bytes);
            if (st) return st;
            st = cuda_status(gwfa::launch_slab_init(g->plain_slab, bytes, 1, log2, prune, s));
            if (st) return st;
            g->plain_log2 = log2;
            g->plain_prune = prune;
        }
        st = cuda_status(cudaMemcpyAsync(g->plain_stage, g->plain_host, in_bytes, cudaMemcpyHostToDevice, s));
        if (st) return st;
        *h_plen = 0;
        TierArgs a{};
        a.g = g->dev();
        a.qwords = (const uint32_t *)(g->plain_stage + 64);
        a.q_off = d_in->off;
        a.v_s = &d_in->vs;
        a.v_e = &d_in->ve;
        a.out = (gwfa_result *)d_res;
        a.count_val = 1;
        a.head = &d_in->head;
        a.slabs = g->plain_slab;
        a.slab_bytes = gwfa::slab_layout(log2, prune).total;
        a.log2cap = log2;
        a.max_lag = o.max_lag;
        a.max_score = o.max_score;
        a.traceback = o.traceback ? 1 : 0;
        a.ends = o.ends;
        a.evict_lag = o.evict_lag;
        a.evict_every = o.evict_every ? o.evict_every : 64;
        a.paths = o.traceback ? d_path : nullptr;
        a.path_len = o.traceback ? (uint32_t *)d_plen : nullptr;
        a.path_cap = path_cap;
        st = cuda_status(gwfa::launch_align(a, prune, 1, o.max_lag > 0 ? 256 : n < 3000 ? 512 : 1024, s));
        if (!st) st = cuda_status(cudaStreamSynchronize(s));
        if (st) return st;
        *out = *h_res;
        if (o.traceback) {
            *path_len = *h_plen;
            if (path_cap && *path_len)
                st = cuda_status(cudaMemcpy(h_path, d_path, (uint64_t)std::min(path_cap, *path_len) * 4,
                                            cudaMemcpyDeviceToHost));
            if (st) return st;
        }
        if (out->status == GWFA_ERR_CAPACITY && log2 + 3 <= gwfa::kMaxLog2Tiles) {
            log2 += 3;   // grow the workspace and run again
            continue;
        }
        return GWFA_OK;
    }
}

// ---------------------------------------------------------------- engine

int gwfa_engine_default_config(const gwfa_graph *g, int prune, gwfa_engine_config *cfg) {
    if (!g || !cfg) return GWFA_ERR_INVALID;
    memset(cfg, 0, sizeof(*cfg));
    int st = cuda_status(cudaSetDevice(g->device));
    if (st) return st;
    int sms = 0, bps = 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, g->device) != cudaSuccess)
        return GWFA_ERR_CUDA;
    // width chosen for each batch (auto_threads); as many narrow CTAs as fit on an SM
    cfg->threads = GWFA_THREADS_AUTO;
    if (gwfa::align_occupancy(prune != 0, prune ? gwfa::kNarrow / 2 : gwfa::kNarrow, &bps) || bps < 1) bps = 1;
    cfg->wide = {0u, prune ? 18u : 19u, 512u, 0u};   // no concurrent classes by default
    cfg->huge = {0u, 22u, 512u, 0u};
    cfg->n_tiers = 3;
    cfg->tiers[0] = {(uint32_t)(sms * bps), prune ? 15u : 16u, 0u, 0u};
    cfg->tiers[1] = {(uint32_t)sms, 19u, 0u, 0u};
    cfg->tiers[2] = {(uint32_t)std::max(sms / 8, 1), 22u, 0u, 0u};
    cfg->prune_slabs = prune ? 1 : 0;
    cfg->max_queries = 1 << 16;
    cfg->max_bases = 1ull << 28;
    return GWFA_OK;
}

int gwfa_engine_destroy(gwfa_engine *e) {
    if (!e) return GWFA_ERR_INVALID;
    cudaSetDevice(e->g->device);
    for (int t = 0; t < GWFA_MAX_TIERS; ++t) cudaFree(e->slabs[t]);
    cudaFree(e->wide_slabs);
    cudaFree(e->huge_slabs);
    if (e->side) cudaStreamDestroy(e->side);
    if (e->side2) cudaStreamDestroy(e->side2);
    if (e->ev_join2) cudaEventDestroy(e->ev_join2);
    if (e->ev_fork) cudaEventDestroy(e->ev_fork);
    if (e->ev_join) cudaEventDestroy(e->ev_join);
    cudaFree(e->counters);
    cudaFree(e->retry_lists);
    cudaFree(e->stage);
    if (e->host) cudaFreeHost(e->host);
    if (e->stream) cudaStreamDestroy(e->stream);
    delete e;
    return GWFA_OK;
}

static int engine_retry_capacity(gwfa_engine *e, uint64_t n) {
    if (e->retry_cap >= n) return GWFA_OK;
    cudaFree(e->retry_lists);
    e->retry_lists = nullptr;
    e->retry_cap = 0;
    uint64_t want = std::max<uint64_t>(n, 1024);
    if (dmalloc(&e->retry_lists, want * 4 * (GWFA_MAX_TIERS + 1))) return GWFA_ERR_OOM;
    e->retry_cap = want;
    return GWFA_OK;
}

int gwfa_engine_create(const gwfa_graph *g, const gwfa_engine_config *cfg, gwfa_engine **out) {
    gwfa::Range range_("gwfa_engine_create");
    if (!g || !cfg || !out) return GWFA_ERR_INVALID;
    *out = nullptr;
    if (cfg->n_tiers < 1 || cfg->n_tiers > GWFA_MAX_TIERS) return GWFA_ERR_INVALID;
    const uint32_t threads = cfg->threads ? cfg->threads : 128;
    if (threads != GWFA_THREADS_AUTO && (threads % 32 || threads < 32 || threads > 1024)) return GWFA_ERR_INVALID;
    for (uint32_t t = 0; t < cfg->n_tiers + 2; ++t) {
        const gwfa_tier &tt = t < cfg->n_tiers ? cfg->tiers[t] : (t == cfg->n_tiers ? cfg->wide : cfg->huge);
        if (t >= cfg->n_tiers && tt.ctas == 0) continue;   // class not used
        const uint32_t th = tt.threads;
        if (tt.ctas == 0 || tt.log2_tiles < 8 || tt.log2_tiles > gwfa::kMaxLog2Tiles ||
            (th && (th % 32 || th < 32 || th > 1024)))
            return GWFA_ERR_INVALID;
    }
    int st = cuda_status(cudaSetDevice(g->device));
    if (!st) st = cuda_status(gwfa::preload_kernels());
    if (st) return st;
    gwfa_engine *e = new (std::nothrow) gwfa_engine();
    if (!e) return GWFA_ERR_OOM;
    e->g = g;
    e->cfg = *cfg;
    e->cfg.threads = threads;
    if (cudaDeviceGetAttribute(&e->sms, cudaDevAttrMultiProcessorCount, g->device) != cudaSuccess) e->sms = 1;
    st = cuda_status(cudaStreamCreateWithFlags(&e->stream, cudaStreamNonBlocking));
    for (uint32_t t = 0; !st && t < cfg->n_tiers; ++t) {
        e->slab_bytes[t] = gwfa::slab_layout(cfg->tiers[t].log2_tiles, cfg->prune_slabs != 0).total;
        const uint64_t bytes = e->slab_bytes[t] * cfg->tiers[t].ctas;
        st = dmalloc(&e->slabs[t], bytes);
        if (!st)
            st = cuda_status(gwfa::launch_slab_init(e->slabs[t], e->slab_bytes[t], cfg->tiers[t].ctas,
                                                    cfg->tiers[t].log2_tiles, cfg->prune_slabs != 0,
                                                    e->stream));
        e->device_bytes += bytes;
    }
    if (!st && cfg->huge.ctas) {
        e->huge_slab_bytes = gwfa::slab_layout(cfg->huge.log2_tiles, cfg->prune_slabs != 0).total;
        const uint64_t bytes = e->huge_slab_bytes * cfg->huge.ctas;
        st = dmalloc(&e->huge_slabs, bytes);
        if (!st)
            st = cuda_status(gwfa::launch_slab_init(e->huge_slabs, e->huge_slab_bytes, cfg->huge.ctas,
                                                    cfg->huge.log2_tiles, cfg->prune_slabs != 0,
                                                    e->stream));
        e->device_bytes += bytes;
    }
    if (!st) st = cuda_status(cudaStreamCreateWithFlags(&e->side2, cudaStreamNonBlocking));
    if (!st) st = cuda_status(cudaEventCreateWithFlags(&e->ev_join2, cudaEventDisableTiming));
    if (!st && cfg->wide.ctas) {
        e->wide_slab_bytes = gwfa::slab_layout(cfg->wide.log2_tiles, cfg->prune_slabs != 0).total;
        const uint64_t bytes = e->wide_slab_bytes * cfg->wide.ctas;
        st = dmalloc(&e->wide_slabs, bytes);
        if (!st)
            st = cuda_status(gwfa::launch_slab_init(e->wide_slabs, e->wide_slab_bytes, cfg->wide.ctas,
                                                    cfg->wide.log2_tiles, cfg->prune_slabs != 0,
                                                    e->stream));
        e->device_bytes += bytes;
    }
    if (!st) st = cuda_status(cudaStreamCreateWithFlags(&e->side, cudaStreamNonBlocking));
    if (!st) st = cuda_status(cudaEventCreateWithFlags(&e->ev_fork, cudaEventDisableTiming));
    if (!st) st = cuda_status(cudaEventCreateWithFlags(&e->ev_join, cudaEventDisableTiming));
    if (!st) st = dmalloc(&e->counters, 256);
    if (!st) st = ensure_pinned(&e->host, &e->host_bytes, kStagedBatch);
    if (!st) st = engine_retry_capacity(e, cfg->max_queries);
    if (!st) st = cuda_status(cudaStreamSynchronize(e->stream));
    if (st) { gwfa_engine_destroy(e); return st; }
    *out = e;
    return GWFA_OK;
}

uint64_t gwfa_engine_device_bytes(const gwfa_engine *e) {
    return e ? e->device_bytes + e->retry_cap * 4 * (GWFA_MAX_TIERS + 1) + e->stage_bytes : 0;
}

uint32_t gwfa_engine_last_launches(const gwfa_engine *e) { return e ? e->last_launches : 0; }

int gwfa_engine_last_retries(gwfa_engine *e, uint32_t *out) {
    if (!e || !out) return GWFA_ERR_INVALID;
    std::lock_guard<std::mutex> lk(e->mu);
    int st = cuda_status(cudaSetDevice(e->g->device));
    if (!st) st = cuda_status(cudaDeviceSynchronize());
    if (!st)
        st = cuda_status(cudaMemcpy(out, e->counters + GWFA_MAX_TIERS, GWFA_MAX_TIERS * 4,
                                    cudaMemcpyDeviceToHost));
    return st;
}

int gwfa_plan_schedule(uint32_t n, const float *h_pred, uint64_t tier0_tiles, uint64_t wide_tiles,
                       uint32_t *h_order, gwfa_schedule *out) {
    if ((n && (!h_pred || !h_order)) || !out) return GWFA_ERR_INVALID;
    std::vector<uint32_t> huge, big, small;
    // diagonals -> hash tiles: on the benchmark graphs a claimed 8-diagonal tile
    // holds about 6 visited diagonals; 0.25 tiles per diagonal leaves a margin of 1.5
    const double tile_per_diag = 0.25;
    for (uint32_t i = 0; i < n; ++i) {
        const double tiles = std::expm1((double)h_pred[(uint64_t)i * 4 + 2]) * tile_per_diag;
        if (wide_tiles && tiles > (double)wide_tiles) huge.push_back(i);
        else if (tiles > (double)tier0_tiles) big.push_back(i);
        else small.push_back(i);
    }
    auto by_cells = [&](uint32_t a, uint32_t b) {
        const float ca = h_pred[(uint64_t)a * 4 + 3], cb = h_pred[(uint64_t)b * 4 + 3];
        return ca != cb ? ca > cb : a < b;
    };
    std::sort(huge.begin(), huge.end(), by_cells);
    std::sort(big.begin(), big.end(), by_cells);
    std::sort(small.begin(), small.end(), by_cells);
    uint32_t k = 0;
    for (uint32_t i : huge) h_order[k++] = i;
    for (uint32_t i : big) h_order[k++] = i;
    for (uint32_t i : small) h_order[k++] = i;
    out->n_huge = (uint32_t)huge.size();
    out->n_wide = (uint32_t)big.size();
    return GWFA_OK;
}

int gwfa_engine_set_paths(gwfa_engine *e, uint32_t *d_paths, uint32_t path_cap, uint32_t *d_path_len) {
    if (!e || (path_cap && !d_paths)) return GWFA_ERR_INVALID;
    std::lock_guard<std::mutex> lk(e->mu);
    e->paths = d_paths;
    e->path_cap = path_cap;
    e->path_len = d_path_len;
    return GWFA_OK;
}

int gwfa_engine_set_stats(gwfa_engine *e, uint64_t *d_stats) {
    if (!e) return GWFA_ERR_INVALID;
    std::lock_guard<std::mutex> lk(e->mu);
    e->stats = (unsigned long long *)d_stats;
    return GWFA_OK;
}

int gwfa_pack_queries_device(uint32_t n_queries, const char *d_q, const uint64_t *d_q_off,
                             uint32_t *d_words, int32_t *d_status, void *stream) {
    if (!d_q_off || !d_words || (n_queries && !d_q)) return GWFA_ERR_INVALID;
    return cuda_status(gwfa::launch_pack(n_queries, d_q, d_q_off, d_words, d_status,
                                         (cudaStream_t)stream));
}

// Arguments of one alignment launch over queue positions [offset, offset + count)
// of `list` (or of the retry list given by list_count).
static TierArgs tier_args(gwfa_engine *e, const uint32_t *d_words, const uint64_t *d_q_off,
                          const uint32_t *d_vs, const uint32_t *d_ve, const int32_t *d_status,
                          const gwfa_opts &o, gwfa_result *d_out) {
    TierArgs a{};
    a.g = e->g->dev();
    a.qwords = d_words;
    a.q_off = d_q_off;
    a.v_s = d_vs;
    a.v_e = d_ve;
    a.qstatus = d_status;
    a.out = d_out;
    a.max_lag = o.max_lag;
    a.max_score = o.max_score;
    a.stats = e->stats;
    a.traceback = o.traceback ? 1 : 0;
    a.ends = o.ends;
    a.evict_lag = o.evict_lag;
    a.evict_every = o.evict_every ? o.evict_every : 64;
    a.paths = e->paths;
    a.path_len = e->path_len;
    a.path_cap = e->path_cap;
    return a;
}

static int run_tiers(gwfa_engine *e, uint32_t n, const uint32_t *d_words, const uint64_t *d_q_off,
                     const uint32_t *d_vs, const uint32_t *d_ve, const uint32_t *d_order,
                     const gwfa_schedule *sched, const int32_t *d_status, const gwfa_opts &o,
                     gwfa_result *d_out, uint64_t len, cudaStream_t s) {
    int st = engine_retry_capacity(e, n);
    if (st) return st;
    const uint32_t T = e->cfg.n_tiers;
    uint32_t *heads = e->counters, *rcount = e->counters + GWFA_MAX_TIERS;
    st = cuda_status(cudaMemsetAsync(e->counters, 0, 256, s));
    if (st) return st;
    const bool prune = o.max_lag > 0 || o.traceback;   // 64-bit values
    e->last_launches = 0;
    // queue order: [huge | wide | tier 0]; the two first classes run on their own
    // CTAs, concurrently with tier 0, and hand their overflows to the retry tiers
    uint32_t n_huge = sched && e->huge_slabs ? std::min(sched->n_huge, n) : 0;
    uint32_t n_wide = sched && e->wide_slabs ? std::min(sched->n_wide, n - n_huge) : 0;
    // a batch without an order, and with more queries than the widest CTAs take at once
    // (997 reads of 1-20 kb: 14.3 ms in input order, 9.4 longest first; the sort takes a few us)
    if (!d_order && n_huge + n_wide == 0 && n > (uint32_t)e->sms) {
        uint32_t *order = e->retry_lists + (uint64_t)GWFA_MAX_TIERS * e->retry_cap;
        st = cuda_status(gwfa::launch_order(n, d_q_off, order, s));
        if (st) return st;
        e->last_launches++;
        d_order = order;
    }
    struct Cls {
        const gwfa_tier *tier;
        uint8_t *slabs;
        uint64_t slab_bytes;
        uint32_t count, offset, *head, *retry, *retry_count;
    } cls[2] = {
        {&e->cfg.huge, e->huge_slabs, e->huge_slab_bytes, n_huge, 0,
         e->counters + 2 * GWFA_MAX_TIERS + 1, T > 1 ? e->retry_lists + (uint64_t)(T - 2) * e->retry_cap : nullptr,
         rcount + (T > 1 ? T - 2 : 0)},
        {&e->cfg.wide, e->wide_slabs, e->wide_slab_bytes, n_wide, n_huge,
         e->counters + 2 * GWFA_MAX_TIERS, T > 1 ? e->retry_lists : nullptr, rcount},
    };
    auto tier_threads = [&](const gwfa_tier &t, uint32_t count) {
        if (t.threads) return t.threads;
        return e->cfg.threads != GWFA_THREADS_AUTO ? e->cfg.threads
                                              : auto_threads(count, len ? len : 4000, e->sms, o.max_lag);
    };
    auto per_sm = [&](uint32_t threads) {
        int b = 1;
        return gwfa::align_occupancy(prune, threads, &b) || b < 1 ? 1u : (uint32_t)b;
    };
    const uint32_t t0_threads = tier_threads(e->cfg.tiers[0], n - n_huge - n_wide);
    // (an engine with classes has its own place for heavy queries)
    const bool few = T > 1 && n <= 4u * (uint32_t)e->sms && !e->wide_slabs && !e->huge_slabs &&
                     !e->cfg.tiers[0].threads && e->cfg.threads == GWFA_THREADS_AUTO &&
                     e->cfg.tiers[1].log2_tiles > e->cfg.tiers[0].log2_tiles &&
                     e->cfg.tiers[1].ctas >= std::min(n, (uint32_t)e->sms);
    // the classes' CTAs and tier 0's must be resident together (tier 0 would otherwise fill
    // every SM and the heaviest queries would start only after it, or the other way round):
    // the classes leave tier 0 half of the SMs, or what their part of tier 0's CTAs (the
    // measure by which plans size them) leaves it if that is less: a wide CTA takes up to
    // half an SM (5,000 reads of 1-100 kb, 489 of them on 443 CTAs of 512 threads, two an
    // SM: with one CTA left for tier 0 the batch takes 13 s, so 0.43)
    double taken = 0;   // SMs
    const double part = (double)(std::min(e->cfg.huge.ctas, n_huge) + std::min(e->cfg.wide.ctas, n_wide)) / e->cfg.tiers[0].ctas;
    const double room = e->sms * std::min(std::max(0.5, part), 0.9);
    uint32_t cctas[2] = {0, 0};
    for (int c = 0; c < 2; ++c) {
        if (!cls[c].count) continue;
        cctas[c] = std::min(cls[c].tier->ctas, cls[c].count);
        const double fit = per_sm(tier_threads(*cls[c].tier, cctas[c]));
        cctas[c] = std::max(std::min(cctas[c], (uint32_t)(std::max(room - taken, 0.0) * fit)), 1u);
        taken += cctas[c] / fit;
    }
    auto t0_ctas = [&](uint32_t threads) {
        return std::min(e->cfg.tiers[0].ctas, (uint32_t)e->sms * per_sm(threads));
    };
    // A class is dispatched before tier 0, which would else leave no SM with room for a wide
    // CTA until it ends: the first one in the caller's stream itself, the second one event
    // later, tier 0 another event later.  Tier 0 has all its CTAs: those that
    // find no room beside the classes start when a class CTA ends (10,000 reads of 1-20 kb,
    // the longest 25 or 100 in a class of 512-thread CTAs: 44.5 / 50.3 ms with the classes on
    // side streams and fewer CTAs for tier 0, 33.1 / 34.5 so, 32.7 without a class; a
    // replayed graph with both classes may still take tier 0 first, 43.2).
    cudaStream_t ts = s;   // tier 0's
    const bool two = n_huge && n_wide;
    if (n_huge || n_wide) {
        ts = e->side;
        st = cuda_status(cudaEventRecord(e->ev_fork, s));
        if (two) {
            if (!st) st = cuda_status(cudaStreamWaitEvent(e->side2, e->ev_fork, 0));
            if (!st) st = cuda_status(cudaEventRecord(e->ev_join2, e->side2));
        }
        if (!st) st = cuda_status(cudaStreamWaitEvent(ts, two ? e->ev_join2 : e->ev_fork, 0));
        if (st) return st;
    }
    for (int c = 0; c < 2; ++c) {
        if (!cls[c].count) continue;
        TierArgs a = tier_args(e, d_words, d_q_off, d_vs, d_ve, d_status, o, d_out);
        a.list = d_order;
        a.count_val = cls[c].count;
        a.list_offset = cls[c].offset;
        a.retry = cls[c].retry;
        a.retry_count = cls[c].retry_count;
        a.head = cls[c].head;
        a.slabs = cls[c].slabs;
        a.slab_bytes = cls[c].slab_bytes;
        a.log2cap = cls[c].tier->log2_tiles;
        const uint32_t th = tier_threads(*cls[c].tier, cctas[c]);
        st = cuda_status(gwfa::launch_align(a, prune, cctas[c], th, c == 1 && two ? e->side2 : s));
        if (st) return st;
        e->last_launches++;
    }
    auto join = [&]() -> int {
        if (ts == s) return GWFA_OK;
        int r = cuda_status(cudaEventRecord(e->ev_join, ts));
        if (!r) r = cuda_status(cudaStreamWaitEvent(s, e->ev_join, 0));
        if (!r && two) r = cuda_status(cudaEventRecord(e->ev_join2, e->side2));
        if (!r && two) r = cuda_status(cudaStreamWaitEvent(s, e->ev_join2, 0));
        return r;
    };
    for (uint32_t t = 0; t < T; ++t) {
        if (t == 1) {
            st = join();   // the retry tiers also take the classes' overflows
            if (st) return st;
        }
        TierArgs a = tier_args(e, d_words, d_q_off, d_vs, d_ve, d_status, o, d_out);
        a.list = t == 0 ? d_order : e->retry_lists + (uint64_t)(t - 1) * e->retry_cap;
        a.list_count = t == 0 ? nullptr : rcount + (t - 1);
        a.count_val = t == 0 ? n - n_huge - n_wide : n;
        a.list_offset = t == 0 ? n_huge + n_wide : 0;
        a.retry = t + 1 < T ? e->retry_lists + (uint64_t)t * e->retry_cap : nullptr;
        a.retry_count = rcount + t;
        a.head = heads + t;
        a.slabs = e->slabs[t];
        a.slab_bytes = e->slab_bytes[t];
        a.log2cap = e->cfg.tiers[t].log2_tiles;
        const uint32_t most = t == 0 ? a.count_val : n;   // no more CTAs than queries there can be
        auto launch = [&](uint32_t th, uint32_t ctas) {
            TierArgs b = a;
            if (t == 0 && th == 1024 && few) {
                // a few queries, one wide CTA an SM: they start on tier 1's slabs, so that the
                // heaviest do not run a second time after the others (300 reads with a heavy
                // tail, 15 to 20 of which overflow tier 0: 67 ms, 46 so)
                b.slabs = e->slabs[1];
                b.slab_bytes = e->slab_bytes[1];
                b.log2cap = e->cfg.tiers[1].log2_tiles;
                b.retry = T > 2 ? e->retry_lists + e->retry_cap : nullptr;
                b.retry_count = rcount + 1;
                ctas = std::min(ctas, e->cfg.tiers[1].ctas);   // (one slab a CTA)
            }
            const int r = cuda_status(gwfa::launch_align(b, prune, std::max(std::min(ctas, most), 1u), th, t == 0 ? ts : s));
            if (!r) e->last_launches++;
            return r;
        };
        if (t > 0) {
            st = launch(tier_threads(e->cfg.tiers[t], e->cfg.tiers[t].ctas), e->cfg.tiers[t].ctas);
        } else if (len || e->cfg.tiers[0].threads || e->cfg.threads != GWFA_THREADS_AUTO || o.max_lag > 0) {
            st = launch(t0_threads, t0_ctas(t0_threads));
        } else {
            // lengths in device memory only: one launch per width, two of which leave at once
            // (about 3 us each; the wrong width costs up to 3x, see auto_threads)
            const uint64_t from[4] = {1ull << 32, wide_from(most, e->sms), mid_from(most, e->sms), 0};
            const uint32_t width[3] = {1024u, 512u, gwfa::kNarrow};
            a.n_all = n;
            for (int w = 0; w < 3 && !st; ++w) {
                a.len_lo = (uint32_t)std::min<uint64_t>(from[w + 1], 0xFFFFFFFFull);
                a.len_hi = (uint32_t)std::min<uint64_t>(from[w], 0xFFFFFFFFull);
                if (a.len_lo < a.len_hi) st = launch(width[w], t0_ctas(width[w]));
            }
        }
        if (st) return st;
    }
    if (T == 1) return join();
    return GWFA_OK;
}

int gwfa_align_batch_device(gwfa_engine *e, uint32_t n, const uint32_t *d_words,
                            const uint64_t *d_q_off, const uint32_t *d_vs, const uint32_t *d_ve,
                            const uint32_t *d_order, const gwfa_schedule *sched, const int32_t *d_status,
                            const gwfa_opts *opts, gwfa_result *d_out, void *stream) {
    gwfa::Range range_("gwfa_align_batch_device");
    if (!e || !d_words || !d_q_off || !d_vs || !d_ve || !d_out) return GWFA_ERR_INVALID;
    gwfa_opts o = opts ? *opts : gwfa_opts{0, 0, -1, 0};
    if (o.max_lag < 0 || !ends_ok(o)) return GWFA_ERR_INVALID;
    if ((o.max_lag > 0 || o.traceback) && !e->cfg.prune_slabs) return GWFA_ERR_INVALID;
    if (n == 0) return GWFA_OK;
    std::lock_guard<std::mutex> lk(e->mu);
    int st = cuda_status(cudaSetDevice(e->g->device));
    if (st) return st;
    // exactly the caller's stream (NULL = the legacy default stream), so the batch is
    // ordered after whatever produced its inputs on that stream
    return run_tiers(e, n, d_words, d_q_off, d_vs, d_ve, d_order, sched, d_status, o, d_out, 0,
                     (cudaStream_t)stream);
}

int gwfa_align_batch(gwfa_engine *e, uint32_t n, const char *h_q, const uint64_t *h_q_off,
                     const uint32_t *h_vs, const uint32_t *h_ve, const uint32_t *h_order,
                     const gwfa_schedule *sched, const gwfa_opts *opts, gwfa_result *h_out, void *stream) {
    if (!e || !h_q_off || !h_vs || !h_ve || !h_out) return GWFA_ERR_INVALID;
    gwfa::Range range_("gwfa_align_batch");
    gwfa_opts o = opts ? *opts : gwfa_opts{0, 0, -1, 0};
    if (o.max_lag < 0 || !ends_ok(o)) return GWFA_ERR_INVALID;
    if ((o.max_lag > 0 || o.traceback) && !e->cfg.prune_slabs) return GWFA_ERR_INVALID;
    if (n == 0) return GWFA_OK;
    if (h_q_off[0] != 0) return GWFA_ERR_INVALID;
    const uint64_t nb = h_q_off[n];
    if (nb > 0 && !h_q) return GWFA_ERR_INVALID;
    std::lock_guard<std::mutex> lk(e->mu);
    int st = cuda_status(cudaSetDevice(e->g->device));
    if (st) return st;
    cudaStream_t s = stream ? (cudaStream_t)stream : e->stream;
    const uint64_t need = gwfa::align256(nb + 16) + gwfa::align256((uint64_t)(n + 1) * 8) +
                          3 * gwfa::align256((uint64_t)n * 4) + gwfa::align256((uint64_t)n * 4) +
                          gwfa::align256(words_for(n, nb) * 4) +
                          gwfa::align256((uint64_t)n * sizeof(gwfa_result)) + 4096;
    st = ensure(&e->stage, &e->stage_bytes, need);
    if (st) return st;
    Carve c{e->stage};
    char *d_q = c.take<char>(nb + 16);
    uint64_t *d_off = c.take<uint64_t>((uint64_t)(n + 1) * 8);
    uint32_t *d_vs = c.take<uint32_t>((uint64_t)n * 4);
    uint32_t *d_ve = c.take<uint32_t>((uint64_t)n * 4);
    uint32_t *d_order = c.take<uint32_t>((uint64_t)n * 4);
    const uint64_t in_bytes = c.off;   // the inputs come first
    int32_t *d_status = c.take<int32_t>((uint64_t)n * 4);
    uint32_t *d_words = c.take<uint32_t>(words_for(n, nb) * 4);
    gwfa_result *d_out = c.take<gwfa_result>((uint64_t)n * sizeof(gwfa_result));
    nvtxRangePushA("copy in + pack");
    if (in_bytes <= kStagedBatch) {
        // a small batch is bound by its copies and launches: its arrays are gathered in pinned
        // memory (the call waits for the batch, so the buffer is free again when it returns)
        auto put = [&](void *d, const void *h, uint64_t bytes) {
            if (bytes) memcpy(e->host + ((uint8_t *)d - e->stage), h, bytes);
        };
        put(d_q, h_q, nb);
        put(d_off, h_q_off, (uint64_t)(n + 1) * 8);
        put(d_vs, h_vs, (uint64_t)n * 4);
        put(d_ve, h_ve, (uint64_t)n * 4);
        if (h_order) put(d_order, h_order, (uint64_t)n * 4);
        st = cuda_status(cudaMemcpyAsync(e->stage, e->host, in_bytes, cudaMemcpyHostToDevice, s));
    } else {
        st = cuda_status(cudaMemcpyAsync(d_q, h_q, nb, cudaMemcpyHostToDevice, s));
        if (!st) st = cuda_status(cudaMemcpyAsync(d_off, h_q_off, (uint64_t)(n + 1) * 8, cudaMemcpyHostToDevice, s));
        if (!st) st = cuda_status(cudaMemcpyAsync(d_vs, h_vs, (uint64_t)n * 4, cudaMemcpyHostToDevice, s));
        if (!st) st = cuda_status(cudaMemcpyAsync(d_ve, h_ve, (uint64_t)n * 4, cudaMemcpyHostToDevice, s));
        if (!st && h_order) st = cuda_status(cudaMemcpyAsync(d_order, h_order, (uint64_t)n * 4, cudaMemcpyHostToDevice, s));
    }
    if (!st) st = cuda_status(gwfa::launch_pack(n, d_q, d_off, d_words, d_status, s));
    nvtxRangePop();
    nvtxRangePushA("alignment tiers");
    if (!st)
        st = run_tiers(e, n, d_words, d_off, d_vs, d_ve, h_order ? d_order : nullptr, sched, d_status, o,
                       d_out, nb / n, s);
    nvtxRangePop();
    if (!st) e->last_launches += 1;
    nvtxRangePushA("copy out + wait");
    if (!st) st = cuda_status(cudaMemcpyAsync(h_out, d_out, (uint64_t)n * sizeof(gwfa_result), cudaMemcpyDeviceToHost, s));
    if (!st) st = cuda_status(cudaStreamSynchronize(s));
    nvtxRangePop();
    return st;
}

}  // extern "C"
