// C ABI of libwd: contexts, gauge upload, pack/unpack and the plain operators.
#include <algorithm>
#include <cstring>
#include <cmath>
#include "dslash.cuh"
#include "blas.cuh"
#include "wd_host.h"

using namespace wd;

namespace wd {

wd_status fail(wd_ctx *c, wd_status s, const std::string &msg) {
    if (c) c->last_error = msg;
    return s;
}

wd_status cuda_fail(wd_ctx *c, cudaError_t e, const char *where) {
    std::string m = std::string(where) + ": " + cudaGetErrorName(e) + " (" + cudaGetErrorString(e) + ")";
    return fail(c, e == cudaErrorMemoryAllocation ? WD_ERR_OOM : WD_ERR_CUDA, m);
}

// A copy of the links is not made inside a stream capture: it would only be filled when the graph
// runs, while this context took it as filled for every call from now on.
static wd_status not_capturing(wd_ctx *c) {
    cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
    const cudaError_t e = cudaStreamIsCapturing(c->stream, &st);
    if (e == cudaSuccess && st == cudaStreamCaptureStatusNone) return WD_OK;
    if (e != cudaSuccess && e != cudaErrorStreamCaptureImplicit) return cuda_fail(c, e, "cudaStreamIsCapturing");
    cudaGetLastError();
    return fail(c, WD_ERR_STATE, "the links have no copy for this call yet, and none is made inside a stream capture: "
                                 "one such call outside it first");
}

// Frees the link copies that new links or another compression left to be refilled (wd_ctx.h) and that
// have not been, with the graphs that hold their addresses: called before device memory is allocated,
// so that a context never holds more than its present use and what it last held for refilling.
static void free_stale_copies(wd_ctx *c) {
    bool any = false;
    for (int p = 0; p < kNumPrec; ++p)
        any |= (c->gauge[p] && !c->gauge_ok[p]) || (c->gauge_eo[p] && !c->gauge_eo_ok[p]);
    if (!any || not_capturing(c) != WD_OK) return;
    cudaStreamSynchronize(c->stream);
    for (int p = 0; p < kNumPrec; ++p) {
        if (c->gauge[p] && !c->gauge_ok[p]) {
            cudaFree(c->gauge[p]);
            c->gauge[p] = nullptr;
        }
        if (c->gauge_eo[p] && !c->gauge_eo_ok[p]) {
            cudaFree(c->gauge_eo[p]);
            c->gauge_eo[p] = nullptr;
        }
    }
    graph_clear(c);
}

wd_status ws_get(wd_ctx *c, const std::string &name, size_t bytes, void **out) {
    auto it = c->ws.find(name);
    if (it != c->ws.end() && c->ws_size[name] >= bytes) {
        *out = it->second;
        return WD_OK;
    }
    if (it != c->ws.end()) {
        cudaStreamSynchronize(c->stream);
        cudaFree(it->second);
        c->ws.erase(it);
        // graphs may hold the old pointer
        graph_clear(c);
    }
    free_stale_copies(c);
    void *p = nullptr;
    cudaError_t e = cudaMalloc(&p, bytes);
    if (e != cudaSuccess) return cuda_fail(c, e, ("cudaMalloc(" + name + ")").c_str());
    c->ws[name] = p;
    c->ws_size[name] = bytes;
    *out = p;
    return WD_OK;
}

size_t gauge_dir_bytes(const wd_ctx *c, Prec p) { return round_up(link_dir_bytes(p, link_recon(c, p), c->g.Vs), 256); }

template <int P, int RECON>
static void gauge_pack(const double *canon, void *dst, const Geom &g, size_t dir, cudaStream_t st) {
    dim3 grid((g.V + 127) / 128, 4);
    k_gauge_pack<P, RECON><<<grid, 128, 0, st>>>(reinterpret_cast<const double2 *>(canon), dst, g.V, g.Vs, dir, g.links_fx);
}

// *buf: a device buffer for links of compression recon (its size depends on that alone); one of
// another compression, stale by then, is freed
static wd_status link_buffer(wd_ctx *c, void **buf, int *have, int recon, size_t bytes) {
    if (*buf && *have == recon) return WD_OK;
    free_stale_copies(c);
    WD_CUDA(c, cudaMalloc(buf, bytes));
    *have = recon;
    return WD_OK;
}

wd_status gauge_get(wd_ctx *c, Prec p, const void **out) {
    if (!c->has_gauge) return fail(c, WD_ERR_STATE, "no gauge field set (call wd_set_gauge first)");
    if (!c->gauge_ok[p]) {
        wd_status s = not_capturing(c);
        if (s != WD_OK) return s;
        s = link_buffer(c, &c->gauge[p], &c->gauge_recon[p], link_recon(c, p),
                        gauge_bytes(p, link_recon(c, p), c->g.Vs));
        if (s != WD_OK) return s;
        void *d = c->gauge[p];
        const size_t dir = gauge_dir_bytes(c, p);
        with_recon(link_recon(c, p), [&](auto rc) {
            constexpr int R = decltype(rc)::value;
            if (p == F64) gauge_pack<F64, R>(c->gauge_canon, d, c->g, dir, c->stream);
            else if (p == F32) gauge_pack<F32, R>(c->gauge_canon, d, c->g, dir, c->stream);
            else if (p == DF32) gauge_pack<DF32, R>(c->gauge_canon, d, c->g, dir, c->stream);
            else gauge_pack<F16, R>(c->gauge_canon, d, c->g, dir, c->stream);
        });
        WD_CUDA(c, cudaGetLastError());
        c->launches += 1;
        c->gauge_ok[p] = true;
    }
    *out = c->gauge[p];
    return WD_OK;
}

// The 8-real parametrisation divides by |u01|^2 + |u02|^2 (zero for the unit link):
// WD_ERR_ARG unless it is at least 1e-6 on every link of the canonical copy.
wd_status check_recon8(wd_ctx *c, const char *who) {
    void *w;
    wd_status s = ws_get(c, "gauge_check", sizeof(unsigned), &w);
    if (s != WD_OK) return s;
    WD_CUDA(c, cudaMemsetAsync(w, 0x7f, sizeof(unsigned), c->stream));
    const size_t nl = (size_t)4 * c->g.V;
    k_gauge_min_offdiag<<<(int)std::min<size_t>((nl + 255) / 256, 4096), 256, 0, c->stream>>>(
        reinterpret_cast<const double2 *>(c->gauge_canon), nl, static_cast<unsigned *>(w));
    WD_CUDA(c, cudaGetLastError());
    c->launches += 1;
    unsigned bits = 0;
    WD_CUDA(c, cudaMemcpyAsync(&bits, w, sizeof bits, cudaMemcpyDeviceToHost, c->stream));
    WD_CUDA(c, cudaStreamSynchronize(c->stream));
    float nmin;
    std::memcpy(&nmin, &bits, sizeof nmin);
    if (!(nmin >= 1e-6f))
        return fail(c, WD_ERR_ARG, std::string(who) + ": recon 8 needs |U01|^2 + |U02|^2 >= 1e-6 on every link "
                                   "(smallest: " + std::to_string(nmin) + "); use recon 12 or 18");
    return WD_OK;
}

// Geom::links_fx for the canonical copy: every link unitary
static wd_status check_unitary(wd_ctx *c) {
    void *w;
    wd_status s = ws_get(c, "gauge_check", sizeof(unsigned), &w);
    if (s != WD_OK) return s;
    WD_CUDA(c, cudaMemsetAsync(w, 0, sizeof(unsigned), c->stream));
    const size_t nl = (size_t)4 * c->g.V;
    k_gauge_not_unitary<<<(int)std::min<size_t>((nl + 255) / 256, 4096), 256, 0, c->stream>>>(
        reinterpret_cast<const double2 *>(c->gauge_canon), nl, static_cast<unsigned *>(w));
    WD_CUDA(c, cudaGetLastError());
    c->launches += 1;
    unsigned bad = 0;
    WD_CUDA(c, cudaMemcpyAsync(&bad, w, sizeof bad, cudaMemcpyDeviceToHost, c->stream));
    WD_CUDA(c, cudaStreamSynchronize(c->stream));
    const int fx = bad ? 0 : 1;
    if (fx != c->g.links_fx) graph_clear(c);  // graphs hold the geometry
    c->g.links_fx = fx;
    return WD_OK;
}

// whether the FP64 kernels multiply limbs (dslash_kernel's FX form)
static bool fx_links(const wd_ctx *c) { return c->g.links_fx && link_recon(c, F64) != 8; }

Geom eo_geom(const wd_ctx *c, int parity) {
    Geom g = c->g;
    g.V = c->g.V / 2;
    g.Vs = (int)round_up((size_t)g.V, kSiteAlign);
    g.eo_parity = parity;
    return g;
}

template <int P, int RECON>
static void gauge_pack_eo(const double *canon, void *dst, const Geom &g, int Vhs, size_t dir, cudaStream_t st) {
    dim3 grid((g.V + 127) / 128, 4);
    k_gauge_pack_eo<P, RECON><<<grid, 128, 0, st>>>(reinterpret_cast<const double2 *>(canon), dst, g, Vhs, dir);
}

wd_status gauge_get_eo(wd_ctx *c, Prec p, const void **out, size_t *dir_bytes) {
    if (!c->has_gauge) return fail(c, WD_ERR_STATE, "no gauge field set (call wd_set_gauge first)");
    const int Vhs = eo_geom(c, 0).Vs;
    const size_t dir = round_up(link_dir_bytes(p, link_recon(c, p), Vhs), 256);
    if (!c->gauge_eo_ok[p]) {
        wd_status s = not_capturing(c);
        if (s != WD_OK) return s;
        s = link_buffer(c, &c->gauge_eo[p], &c->gauge_eo_recon[p], link_recon(c, p), 8 * dir);
        if (s != WD_OK) return s;
        void *d = c->gauge_eo[p];
        with_recon(link_recon(c, p), [&](auto rc) {
            constexpr int R = decltype(rc)::value;
            if (p == F64) gauge_pack_eo<F64, R>(c->gauge_canon, d, c->g, Vhs, dir, c->stream);
            else if (p == F32) gauge_pack_eo<F32, R>(c->gauge_canon, d, c->g, Vhs, dir, c->stream);
            else if (p == DF32) gauge_pack_eo<DF32, R>(c->gauge_canon, d, c->g, Vhs, dir, c->stream);
            else gauge_pack_eo<F16, R>(c->gauge_canon, d, c->g, Vhs, dir, c->stream);
        });
        WD_CUDA(c, cudaGetLastError());
        c->launches += 1;
        c->gauge_eo_ok[p] = true;
    }
    *out = c->gauge_eo[p];
    *dir_bytes = dir;
    return WD_OK;
}

void *graph_get(wd_ctx *c, const std::string &key) {
    auto it = c->graphs.find(key);
    if (it == c->graphs.end()) return nullptr;
    c->graph_used[key] = ++c->graph_tick;
    return it->second;
}

void graph_put(wd_ctx *c, const std::string &key, void *exec, const std::vector<long long> &info) {
    while (c->graphs.size() >= kMaxGraphs) {
        auto lru = c->graph_used.begin();
        for (auto it = c->graph_used.begin(); it != c->graph_used.end(); ++it)
            if (it->second < lru->second) lru = it;
        cudaGraphExecDestroy((cudaGraphExec_t)c->graphs[lru->first]);
        c->graphs.erase(lru->first);
        c->graph_info.erase(lru->first);
        c->graph_used.erase(lru);
    }
    c->graphs[key] = exec;
    c->graph_info[key] = info;
    c->graph_used[key] = ++c->graph_tick;
}

void graph_clear(wd_ctx *c) {
    for (auto &g : c->graphs) cudaGraphExecDestroy((cudaGraphExec_t)g.second);
    c->graphs.clear();
    c->graph_info.clear();
    c->graph_used.clear();
}

// Where no autotuner or wd_set_tiles chose a shape, the fused kernels take up to four right-hand
// sides per block (12 rows of FP32 at 24^3 x 48: 128.9 ms a solve against 129.8 with one and
// 130.8 with two per block; the plain operators differ, see tiles_for).  FP32 rows go in pairs on
// one thread from 2^17 site-rows on with four rows (24^3 x 48: 41.3 -> 39.6 ms) and, even-odd, with
// more (20^3 x 40, 12 rows 37.9 -> 36.3); two rows gain nothing (21.2 / 21.7 ms).  More rows on the
// whole lattice gain on small ones and lose on large ones, and stay single (single / pairs, ms a
// solve: 16^3 x 32 six rows 15.0 / 13.6, eight 17.3 / 16.3, sixteen 33.5 / 31.7; 24^3 x 48 six
// 64.6 / 66.2, eight 77.2 / 81.3, ten 102.9 / 109.3, twelve 116.9 / 125.6; recon-12 eight rows 15.8 /
// 16.0 and 75.5 / 79.3).  With recon-12 links the pairs of the rule still gain (four rows at
// 16^3 x 32 even-odd 6.13 -> 5.65 ms, at 24^4 19.6 -> 19.1), with recon-8 they lose (24^3 x 48 37.5 / 40.0).
// On a shape chosen for the plain operators they need its four rows: with two per block, four rows of
// 24^3 x 48 take 40.3 ms in pairs and 40.0 singly, of 16^3 x 32 9.51 and 9.21.
// FP64 takes one row per block, which shares links through L2 as well and wastes no lanes: blocks of
// 256 threads from 2^17 sites on (64 / 256, ms a solve: 16^3 x 32 24.8 / 23.0, 24^3 x 48 113.9 / 105.1,
// even-odd 39.5 / 38.3, 12 rows 1255 (64 x 4) / 1237), 128 below with several rows (64 x 4 / 128 x 1,
// four rows: 8^3 x 16 9.15 / 8.33, 16^3 x 32 even-odd 30.6 / 29.0; 256 x 1 at 12^3 x 24 30.9 against
// 29.0); single rows below keep 64 (128: -7 to +3 %, by how the last wave fills).
// With FP64 arithmetic (fx_links) 64 x 1 everywhere (64 x 1 / 64 x 4 / 256 x 1, four rows: 8^3 x 12 5.77 /
// 7.39 / 7.28, 16^3 x 32 82.1 / 84.3 / 81.5, even-odd 43.3 / 44.5 / 44.4).
static bool rows_in_pairs(wd_ctx *c, Prec p, int nrhs, bool eo) {
    return p == F32 && link_recon(c, p) != 8 && nrhs % 2 == 0 && (nrhs == 4 || (eo && nrhs > 4)) &&
           (long long)(c->g.V / (eo ? 2 : 1)) * nrhs >= (1 << 17);
}

DslashTiles cg_tiles_for(wd_ctx *c, Prec p, int nrhs, bool eo) {
    auto it = c->cg_tiles.find(p * 64 + nrhs + (eo ? kEoTileKey : 0));
    if (it != c->cg_tiles.end()) return it->second;
    it = c->tiles.find(p * 64 + nrhs);
    DslashTiles t;
    if (it != c->tiles.end()) {
        t = it->second;  // chosen for the plain operators, as are its right-hand sides per thread
    } else {
        t.site_tile = 64;
        t.rhs_tile = nrhs < 4 ? nrhs : 4;
        const long long sites = c->g.V / (eo ? 2 : 1);
        if (p == F64 && !fx_links(c)) {
            t.rhs_tile = 1;
        } else if (p == F64 && (nrhs > 1 || sites >= (1 << 17))) {
            t.site_tile = sites >= (1 << 17) ? 256 : 128;
            t.rhs_tile = 1;
        }
    }
    t.rhs_per_thread = rows_in_pairs(c, p, nrhs, eo) && t.rhs_tile >= 4 && pairs_fit(t) ? 2 : 1;
    return t;
}

void ws_release(wd_ctx *c, const std::string &name) {
    auto it = c->ws.find(name);
    if (it == c->ws.end()) return;
    cudaStreamSynchronize(c->stream);
    cudaFree(it->second);
    c->ws.erase(it);
    c->ws_size.erase(name);
}

// The launch shape where neither wd_set_tiles nor an autotuner chose one.  One right-hand side
// per block: the blocks of a site tile's right-hand sides start together and share its links
// through L2, and a block's rows leave no idle threads when nrhs is odd (24^3 x 48, 64 x 1
// against 64 x 4, us: FP32 12 rows 586 / 618, 7 rows 339 / 388; FP16 408 / 438, 241 / 277).
// FP32 rows with whole links go in pairs on one thread, each link loaded once for both, from 2^17
// site-rows on, two rows from 2^20 on (pairs / 64 x 1, us: 12 rows 569 / 608, 4 rows 190 / 206,
// 4 rows at 16^4 24.1 / 25.0; two rows 106 / 110, at 28^4 99 / 105, at 24^4 59.4 / 58.9, at 20^4
// 35.2 / 33.2).  Compressed links are few enough that the pairs' lower occupancy costs more
// (recon-12: 12 rows 571 / 539, two rows at 20^4 33.1 / 29.0).  Larger blocks for FP64 from 2^18 site-rows on (256 / 64
// threads: 12 rows 3144 / 3289, one row at 32^3 x 64 838 / 876, at 16^4 38.6 / 36.4) and DF32
// (128 / 64: 2810 / 2861).  With FP64 arithmetic (fx_links) 64 threads: more of them leave the FP64
// units of an SM's schedulers unevenly loaded (64 / 256 threads: 24^4 510 / 522, recon-12 797 / 839,
// recon-8 1886 / 1951).
DslashTiles tiles_for(wd_ctx *c, Prec p, int nrhs) {
    auto it = c->tiles.find(p * 64 + nrhs);
    if (it != c->tiles.end()) return it->second;
    const long long work = (long long)c->g.V * nrhs;
    DslashTiles t;
    t.site_tile = p == DF32 ? 128 : p == F64 && fx_links(c) && work >= (1 << 18) ? 256 : 64;
    t.rhs_tile = 1;
    if (p == F32 && link_recon(c, p) == 18 && nrhs % 2 == 0 && work >= (nrhs == 2 ? 1 << 20 : 1 << 17) && !c->split)
        t.rhs_tile = t.rhs_per_thread = 2;
    return t;
}

}  // namespace wd

wd_ctx::~wd_ctx() {
    for (auto &g : graphs) cudaGraphExecDestroy((cudaGraphExec_t)g.second);
    for (auto &w : ws) cudaFree(w.second);
    for (int p = 0; p < kNumPrec; ++p) {
        if (gauge[p]) cudaFree(gauge[p]);
        if (gauge_eo[p]) cudaFree(gauge_eo[p]);
    }
    if (gauge_canon) cudaFree(gauge_canon);
    if (g.dbg) cudaFree(g.dbg);
    if (staged_err) cudaFree(staged_err);
}

static bool bad_prec(int p) { return p < 0 || p >= kNumPrec; }

extern "C" {

const char *wd_status_string(wd_status s) {
    switch (s) {
    case WD_OK: return "ok";
    case WD_ERR_ARG: return "invalid argument";
    case WD_ERR_CUDA: return "CUDA error";
    case WD_ERR_OOM: return "out of device memory";
    case WD_ERR_NOT_CONVERGED: return "not converged";
    case WD_ERR_BREAKDOWN: return "CG breakdown";
    case WD_ERR_NONFINITE: return "non-finite value";
    case WD_ERR_TIMEOUT: return "device-side wait timed out";
    case WD_ERR_STATE: return "call out of order";
    }
    return "unknown status";
}

const char *wd_last_error(const wd_ctx *c) { return c ? c->last_error.c_str() : "null context"; }

long long wd_kernel_launches(const wd_ctx *c) { return c ? c->launches : 0; }

wd_status wd_create(wd_ctx **out, const int dims[4], int antiperiodic_t, void *stream) {
    if (!out || !dims) return WD_ERR_ARG;
    *out = nullptr;
    long long V = 1;
    for (int mu = 0; mu < 4; ++mu) {
        if (dims[mu] < 2) return WD_ERR_ARG;
        V *= dims[mu];
    }
    if (V > (1ll << 30)) return WD_ERR_ARG;
    wd_ctx *c = new wd_ctx();
    for (int mu = 0; mu < 4; ++mu) c->g.L[mu] = dims[mu];
    c->g.V = (int)V;
    c->g.Vs = (int)round_up((size_t)V, kSiteAlign);
    c->g.stride[0] = 1;
    c->g.stride[1] = dims[0];
    c->g.stride[2] = dims[0] * dims[1];
    c->g.stride[3] = dims[0] * dims[1] * dims[2];
    for (int mu = 0; mu < 3; ++mu) c->g.div[mu] = fast_div(dims[mu]);
    c->g.divh = fast_div(dims[0] / 2);
    c->g.antiperiodic = antiperiodic_t ? 1 : 0;
    c->g.eo_parity = -1;
    c->g.dbg = nullptr;
    c->g.split_t = 0;
    c->g.links_fx = 0;
    c->stream = (cudaStream_t)stream;
    if (cudaGetDevice(&c->device) != cudaSuccess) {
        delete c;
        return WD_ERR_CUDA;
    }
#ifdef WD_DEBUG
    if (cudaMalloc(&c->g.dbg, sizeof(unsigned)) != cudaSuccess || cudaMemset(c->g.dbg, 0, sizeof(unsigned)) != cudaSuccess) {
        delete c;
        return WD_ERR_CUDA;
    }
#endif
    *out = c;
    return WD_OK;
}

wd_status wd_destroy(wd_ctx *c) {
    if (!c) return WD_ERR_ARG;
    cudaStreamSynchronize(c->stream);
    delete c;
    return WD_OK;
}

wd_status wd_set_stream(wd_ctx *c, void *stream) {
    if (!c) return WD_ERR_ARG;
    c->stream = (cudaStream_t)stream;
    return WD_OK;
}

wd_status wd_set_gauge(wd_ctx *c, const double *U, int on_device, int recon) {
    wd::NvtxRange nvtx_("wd_set_gauge");
    if (!c) return WD_ERR_ARG;
    if (!U) return fail(c, WD_ERR_ARG, "wd_set_gauge: null gauge pointer");
    if (recon != 18 && recon != 12 && recon != 8) return fail(c, WD_ERR_ARG, "wd_set_gauge: recon must be 18, 12 or 8");
    const size_t bytes = (size_t)4 * c->g.V * 9 * 16;
    // The links are replaced in place, and operators or solves that read them may be under way on a
    // stream that this context (or a batch it took part in, or a captured graph) used before.
    WD_CUDA(c, c->gauge_canon ? cudaDeviceSynchronize() : cudaStreamSynchronize(c->stream));
    // the copies are written again when next needed, in place (16^3 x 32, new links and an FP32
    // solve from host buffers: 4.97 ms with them freed, allocated and the solver's graph rebuilt
    // each time, 4.57 ms without)
    for (int p = 0; p < kNumPrec; ++p) c->gauge_ok[p] = c->gauge_eo_ok[p] = false;
    if (!c->gauge_canon) WD_CUDA(c, cudaMalloc(&c->gauge_canon, bytes));
    WD_CUDA(c, cudaMemcpyAsync(c->gauge_canon, U, bytes, on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice,
                               c->stream));
    c->recon = recon;
    for (int p = 0; p < kNumPrec; ++p) c->recon_p[p] = 0;
    c->has_gauge = false;
    if (recon == 8) {
        wd_status s = check_recon8(c, "wd_set_gauge");
        if (s != WD_OK) return s;
    }
    wd_status s = check_unitary(c);
    if (s != WD_OK) return s;
    c->has_gauge = true;
    const void *d;
    s = gauge_get(c, F64, &d);
    if (s != WD_OK) return s;
    if (!on_device) WD_CUDA(c, cudaStreamSynchronize(c->stream));
    return WD_OK;
}

wd_status wd_debug_word(wd_ctx *c, unsigned *word, int *is_debug) {
    if (!c || !word) return WD_ERR_ARG;
    *word = 0;
#ifdef WD_DEBUG
    if (is_debug) *is_debug = 1;
    WD_CUDA(c, cudaStreamSynchronize(c->stream));
    WD_CUDA(c, cudaMemcpy(word, c->g.dbg, sizeof(unsigned), cudaMemcpyDeviceToHost));
    WD_CUDA(c, cudaMemset(c->g.dbg, 0, sizeof(unsigned)));
#else
    if (is_debug) *is_debug = 0;
#endif
    return WD_OK;
}

wd_status wd_set_link_compression(wd_ctx *c, wd_prec prec, int recon) {
    if (!c) return WD_ERR_ARG;
    if (bad_prec(prec)) return fail(c, WD_ERR_ARG, "wd_set_link_compression: bad precision");
    if (recon != 18 && recon != 12 && recon != 8)
        return fail(c, WD_ERR_ARG, "wd_set_link_compression: recon must be 18, 12 or 8");
    if (!c->has_gauge) return fail(c, WD_ERR_STATE, "no gauge field set (call wd_set_gauge first)");
    if (recon == link_recon(c, (Prec)prec)) return WD_OK;
    if (recon == 8) {
        wd_status s = check_recon8(c, "wd_set_link_compression");
        if (s != WD_OK) return s;
    }
    WD_CUDA(c, cudaDeviceSynchronize());  // as in wd_set_gauge: the copies are refilled in place
    c->gauge_ok[prec] = c->gauge_eo_ok[prec] = false;
    c->recon_p[prec] = recon;
    return WD_OK;
}

size_t wd_field_bytes(const wd_ctx *c, wd_prec prec, int nrhs) {
    if (!c || bad_prec(prec) || nrhs < 1) return 0;
    return spinor_bytes((Prec)prec, c->g.Vs) * (size_t)nrhs;
}

static wd_status canon_stage(wd_ctx *c, const double *canon, int nrhs, int on_device, const double **dev) {
    if (on_device) {
        *dev = canon;
        return WD_OK;
    }
    void *buf;
    const size_t bytes = (size_t)nrhs * c->g.V * 12 * 16;
    wd_status s = ws_get(c, "canon_stage", bytes, &buf);
    if (s != WD_OK) return s;
    WD_CUDA(c, cudaMemcpyAsync(buf, canon, bytes, cudaMemcpyHostToDevice, c->stream));
    *dev = (const double *)buf;
    return WD_OK;
}

wd_status wd_pack(wd_ctx *c, const double *canon, int on_device, void *field, wd_prec prec, int nrhs) {
    wd::NvtxRange nvtx_("wd_pack");
    if (!c) return WD_ERR_ARG;
    if (!canon || !field || bad_prec(prec) || nrhs < 1 || nrhs > WD_MAX_RHS)
        return fail(c, WD_ERR_ARG, "wd_pack: bad argument");
    const double *src = nullptr;
    wd_status s = canon_stage(c, canon, nrhs, on_device, &src);
    if (s != WD_OK) return s;
    VecArgs v{};
    v.V = c->g.V; v.Vs = c->g.Vs; v.nrhs = nrhs;
    v.a = src;
    v.b = field; v.b_stride = spinor_bytes((Prec)prec, c->g.Vs);
    dim3 grid((c->g.V + 127) / 128, nrhs);
    if (prec == WD_F64) k_pack<F64><<<grid, 128, 0, c->stream>>>(v);
    else if (prec == WD_F32) k_pack<F32><<<grid, 128, 0, c->stream>>>(v);
    else if (prec == WD_DF32) k_pack<DF32><<<grid, 128, 0, c->stream>>>(v);
    else k_pack<F16><<<grid, 128, 0, c->stream>>>(v);
    WD_CUDA(c, cudaGetLastError());
    c->launches += 1;
    if (!on_device) WD_CUDA(c, cudaStreamSynchronize(c->stream));
    return WD_OK;
}

wd_status wd_unpack(wd_ctx *c, const void *field, wd_prec prec, int nrhs, double *canon, int on_device) {
    wd::NvtxRange nvtx_("wd_unpack");
    if (!c) return WD_ERR_ARG;
    if (!canon || !field || bad_prec(prec) || nrhs < 1 || nrhs > WD_MAX_RHS)
        return fail(c, WD_ERR_ARG, "wd_unpack: bad argument");
    const size_t bytes = (size_t)nrhs * c->g.V * 12 * 16;
    void *dst = canon;
    if (!on_device) {
        wd_status s = ws_get(c, "canon_stage", bytes, &dst);
        if (s != WD_OK) return s;
    }
    VecArgs v{};
    v.V = c->g.V; v.Vs = c->g.Vs; v.nrhs = nrhs;
    v.a = field; v.a_stride = spinor_bytes((Prec)prec, c->g.Vs);
    v.b = dst;
    dim3 grid((c->g.V + 127) / 128, nrhs);
    if (prec == WD_F64) k_unpack<F64><<<grid, 128, 0, c->stream>>>(v);
    else if (prec == WD_F32) k_unpack<F32><<<grid, 128, 0, c->stream>>>(v);
    else if (prec == WD_DF32) k_unpack<DF32><<<grid, 128, 0, c->stream>>>(v);
    else k_unpack<F16><<<grid, 128, 0, c->stream>>>(v);
    WD_CUDA(c, cudaGetLastError());
    c->launches += 1;
    if (!on_device) {
        WD_CUDA(c, cudaMemcpyAsync(canon, dst, bytes, cudaMemcpyDeviceToHost, c->stream));
        WD_CUDA(c, cudaStreamSynchronize(c->stream));
    }
    return WD_OK;
}

static wd_status apply_common(wd_ctx *c, double kappa, const void *in, void *out, wd_prec prec, int nrhs,
                              bool dagger, const char *who) {
    if (!c) return WD_ERR_ARG;
    if (!in || !out || bad_prec(prec) || nrhs < 1 || nrhs > WD_MAX_RHS)
        return fail(c, WD_ERR_ARG, std::string(who) + ": bad argument");
    if (in == out) return fail(c, WD_ERR_ARG, std::string(who) + ": in and out must be distinct");
    if (!std::isfinite(kappa)) return fail(c, WD_ERR_ARG, std::string(who) + ": kappa not finite");
    if (c->split)
        return fail(c, WD_ERR_STATE, std::string(who) + ": a split sub-lattice needs its faces "
                                                      "(wd_apply_interior and wd_apply_faces)");
    const void *gauge;
    wd_status s = gauge_get(c, (Prec)prec, &gauge);
    if (s != WD_OK) return s;
    DslashArgs a{};
    a.g = c->g;
    a.in = in;
    a.in_stride = a.out_stride = spinor_bytes((Prec)prec, c->g.Vs);
    a.out = out;
    a.gauge = gauge;
    a.gauge_dir = gauge_dir_bytes(c, (Prec)prec);
    a.kappa = kappa;
    a.nrhs = nrhs;
    if (c->prefetch[prec] && prec == WD_F32) {
        DslashTiles t = tiles_for(c, F32, nrhs);
        t.rhs_per_thread = 1;
        WD_CUDA(c, launch_apply_prefetch(a, link_recon(c, F32), dagger, t, c->stream));
    } else if (c->staged_rows[prec]) {
        if ((s = staged_error_word(c)) != WD_OK) return s;
        WD_CUDA(c, launch_apply_staged(a, (Prec)prec, link_recon(c, (Prec)prec), dagger, c->staged_rows[prec],
                                       c->staged_stages[prec], c->staged_err, c->stream));
    } else {
        WD_CUDA(c, launch_apply(a, (Prec)prec, link_recon(c, (Prec)prec), dagger, tiles_for(c, (Prec)prec, nrhs),
                                c->stream));
    }
    c->launches += 1;
    return WD_OK;
}

wd_status wd_apply(wd_ctx *c, double kappa, const void *in, void *out, wd_prec prec, int nrhs) {
    wd::NvtxRange nvtx_("wd_apply");
    if (c) c->launches = 0;
    return apply_common(c, kappa, in, out, prec, nrhs, false, "wd_apply");
}

wd_status wd_apply_dagger(wd_ctx *c, double kappa, const void *in, void *out, wd_prec prec, int nrhs) {
    wd::NvtxRange nvtx_("wd_apply_dagger");
    if (c) c->launches = 0;
    return apply_common(c, kappa, in, out, prec, nrhs, true, "wd_apply_dagger");
}

wd_status wd_normal_apply(wd_ctx *c, double kappa, const void *in, void *out, wd_prec prec, int nrhs) {
    wd::NvtxRange nvtx_("wd_normal_apply");
    if (!c) return WD_ERR_ARG;
    c->launches = 0;
    if (bad_prec(prec) || nrhs < 1 || nrhs > WD_MAX_RHS) return fail(c, WD_ERR_ARG, "wd_normal_apply: bad argument");
    if (c->split) return fail(c, WD_ERR_STATE, "wd_normal_apply: not on a split sub-lattice");
    void *tmp;
    wd_status s = ws_get(c, "normal_tmp", spinor_bytes((Prec)prec, c->g.Vs) * nrhs, &tmp);
    if (s != WD_OK) return s;
    s = apply_common(c, kappa, in, tmp, prec, nrhs, false, "wd_normal_apply");
    if (s != WD_OK) return s;
    return apply_common(c, kappa, tmp, out, prec, nrhs, true, "wd_normal_apply");
}

}  // extern "C"
