// wl_api.cu -- host runtime and C ABI (include/wl.h) of the micromagnetic-
// ensemble Wang-Landau library (arXiv:1302.2320).
//
// A handle owns one lattice's walkers: the line table (l = 0..N/2 by up-down
// symmetry), ragged per-line ln g / histogram arrays over the even k, packed
// spins and up/down index lists, all resident on the device across calls.
// wl_run drives the walk in slices: each slice is one persistent launch over a
// device work queue of lines (queue_line), followed by a summary kernel whose
// result is read back; the slice is captured once as a CUDA graph and replayed.
// The alternative "plain" form issues one launch per line over a pool of streams.
#include <algorithm>
#include <chrono>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <map>
#include <mutex>
#include <string>
#include <tuple>
#include <vector>

#include "../../include/wl.h"
#include "wl_kernels.cuh"
#include "wl_runtime.cuh"

using namespace wl;
using namespace wl::rt;

namespace {

thread_local std::string g_err;

wl_status fail(wl_status s, const char* fmt, ...)
{
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof buf, fmt, ap);
    va_end(ap);
    g_err = buf;
    return s;
}

#define CU(call)                                                                          \
    do {                                                                                  \
        cudaError_t e_ = (call);                                                          \
        if (e_ != cudaSuccess)                                                            \
            return fail(WL_ECUDA, "%s failed: %s (%s:%d)", #call, cudaGetErrorString(e_), \
                        __FILE__, __LINE__);                                              \
    } while (0)

bool lattice_info(int type, int L, LatInfo* o)
{
    if (L < 3) return false;
    o->type = type;
    o->L = L;
    if (type == WL_SQUARE) {
        o->N = L * L;
        o->z = 4;
    } else if (type == WL_TRIANGULAR) {
        o->N = L * L;
        o->z = 6;
    } else if (type == WL_SIMPLE_CUBIC) {
        if (L > 101) return false;
        o->N = L * L * L;
        o->z = 6;
    } else if (type == WL_SQUARE_OPEN) {
        o->N = L * L;
        o->z = 4;
    } else {
        return false;
    }
    if (o->N > (1 << 20)) return false;
    o->NB = type == WL_SQUARE_OPEN ? 2 * L * (L - 1) : o->N * o->z / 2;
    o->kstep = type == WL_SQUARE_OPEN ? 1 : 2;
    return true;
}

// Bins of line l: k in [0, min(z*min(l, N-l), N_B)] (no more than z unhappy
// bonds per minority spin) with the lattice's spacing: every even k on the
// periodic lattices (even degrees), every k with open boundaries.
int line_nbins(const LatInfo& g, int ell)
{
    const int lm = std::min(ell, g.N - ell);
    const int64_t khi = std::min<int64_t>((int64_t)g.z * lm, g.NB);
    return (int)(khi / g.kstep + 1);
}

Layout make_layout(const LatInfo& g)
{
    Layout lo;
    lo.nlines = g.N / 2 + 1;
    lo.idx16 = g.N <= 65536;
    const size_t isz = lo.idx16 ? 2 : 4;
    lo.pstride = (int)(align16((size_t)g.N * isz) / isz);
    lo.W = (int)(align16((size_t)((g.N + 31) / 32) * 4) / 4);
    lo.desc.resize(lo.nlines);
    int64_t off = 0;
    for (int l = 0; l < lo.nlines; ++l) {
        lo.desc[l].bin_off = off;
        lo.desc[l].ell = l;
        lo.desc[l].nbins = line_nbins(g, l);
        off += lo.desc[l].nbins;
    }
    lo.nbins_total = off;
    return lo;
}

size_t required_bytes(const LatInfo& g, const Layout& lo)
{
    const size_t isz = lo.idx16 ? 2 : 4;
    size_t b = 0;
    b += (size_t)lo.nlines * sizeof(LineDesc) + (size_t)lo.nlines * sizeof(LineState);
    b += (size_t)lo.nlines * lo.pstride * isz;
    b += (size_t)lo.nlines * lo.W * 4;
    b += (size_t)lo.nbins_total * (8 + 8 + 8);   // lng, hist, assembled output
    b += (size_t)lo.nlines * 3 * 4;               // queue, per-line queue heads, identity
    b += kTableN * (4 + 8) + 4096;
    return b;
}

// Host-side exp threshold table, an independent evaluation in long double used
// to verify the device-built table bit for bit before a deterministic run.
int host_table_q(double u) { return wl::rt::table_shift(u); }

void host_table(double u, int q, std::vector<uint64_t>& t)
{
    t.resize(kTableN);
    for (int i = 0; i < kTableN; ++i) t[i] = wl::rt::table_entry(u, q, i);
}

constexpr size_t kThermoKept = (size_t)4 << 20;      // the largest workspace of wl_thermo that stays with a handle

struct TuneKey {
    int type, L, det;
    bool operator<(const TuneKey& o) const
    {
        return std::tie(type, L, det) < std::tie(o.type, o.L, o.det);
    }
};
// Autotuner record per (lattice, L, mode): the rate each candidate lane count
// reached on a slice of real work, at the acceptance rate seen then.
struct TuneRec {
    double rate[3] = {-1.0, -1.0, -1.0};   // for kTuneS[0..2]
    double accept = -1.0;                  // acceptance rate when the candidates were timed
    int best = 0;                          // 0 until every candidate has a rate
};
constexpr int kTuneS[3] = {32, 16, 8};
std::mutex g_tune_mu;
std::map<TuneKey, TuneRec> g_tune_cache;

}  // namespace

namespace wl {
// Lets other translation units of the library report through wl_last_error().
void set_last_error(const char* msg) { g_err = msg; }
}  // namespace wl

namespace {

void free_all(wl_ctx* h)
{
    if (h->graph) cudaGraphExecDestroy(h->graph);
    h->graph = nullptr;
    void* ptrs[] = {h->d_desc, h->d_st, h->d_perm, h->d_spins, h->d_lng, h->d_hist, h->d_out,
                    h->d_table, h->d_table64, h->d_order, h->d_ident, h->d_qheads, h->d_flags,
                    h->d_deadline, h->d_summary, h->d_thermo};
    for (void* p : ptrs)
        if (p) cudaFree(p);
    if (h->h_summary) cudaFreeHost(h->h_summary);
    if (h->h_abort) cudaFreeHost(h->h_abort);
    for (auto st : h->pool) cudaStreamDestroy(st);
    h->pool.clear();
    if (h->ev0) cudaEventDestroy(h->ev0);
    if (h->ev1) cudaEventDestroy(h->ev1);
    if (h->ev_join) cudaEventDestroy(h->ev_join);
    if (h->ev_t0) cudaEventDestroy(h->ev_t0);
    if (h->ev_i0) cudaEventDestroy(h->ev_i0);
    if (h->ev_i1) cudaEventDestroy(h->ev_i1);
    if (h->ev_t1) cudaEventDestroy(h->ev_t1);
    if (h->s) cudaStreamDestroy(h->s);
    h->allocated = false;
}

wl_status allocate(wl_ctx* h)
{
    if (h->allocated) return WL_OK;
    const size_t need = required_bytes(h->g, h->lo);
    if (h->hbm_budget > 0 && need > (size_t)h->hbm_budget)
        return fail(WL_ENOMEM, "lattice needs %zu device bytes, budget is %lld", need,
                    (long long)h->hbm_budget);
    CU(cudaGetDevice(&h->device));
    CU(cudaDeviceGetAttribute(&h->num_sms, cudaDevAttrMultiProcessorCount, h->device));
    CU(cudaStreamCreateWithFlags(&h->s, cudaStreamNonBlocking));
    CU(cudaEventCreate(&h->ev0));
    CU(cudaEventCreate(&h->ev1));
    CU(cudaEventCreateWithFlags(&h->ev_join, cudaEventDisableTiming));
    CU(cudaEventCreate(&h->ev_t0));
    CU(cudaEventCreate(&h->ev_i0));
    CU(cudaEventCreate(&h->ev_i1));
    CU(cudaEventCreate(&h->ev_t1));
    const Layout& lo = h->lo;
    const size_t isz = lo.idx16 ? 2 : 4;
    auto alloc = [&](void** p, size_t bytes) -> cudaError_t { return cudaMalloc(p, bytes ? bytes : 16); };
    cudaError_t e = cudaSuccess;
    if (!e) e = alloc((void**)&h->d_desc, lo.nlines * sizeof(LineDesc));
    if (!e) e = alloc((void**)&h->d_st, lo.nlines * sizeof(LineState));
    if (!e) e = alloc(&h->d_perm, (size_t)lo.nlines * lo.pstride * isz);
    if (!e) e = alloc((void**)&h->d_spins, (size_t)lo.nlines * lo.W * 4);
    if (!e) e = alloc((void**)&h->d_lng, (size_t)lo.nbins_total * 8);
    if (!e) e = alloc((void**)&h->d_hist, (size_t)lo.nbins_total * sizeof(hist_t));
    if (!e) e = alloc((void**)&h->d_out, (size_t)lo.nbins_total * 8);
    if (!e) e = alloc((void**)&h->d_table, kTableN * 4);
    if (!e) e = alloc((void**)&h->d_table64, kTableN * 8);
    if (!e) e = alloc((void**)&h->d_order, lo.nlines * 4);
    if (!e) e = alloc((void**)&h->d_ident, lo.nlines * 4);
    if (!e) e = alloc((void**)&h->d_qheads, (lo.nlines + 1) * 4);
    if (!e) e = alloc((void**)&h->d_flags, 16);
    if (!e) e = alloc((void**)&h->d_deadline, 32);
    if (!e) e = alloc((void**)&h->d_summary, sizeof(Summary));
    if (!e) e = cudaHostAlloc((void**)&h->h_summary, sizeof(Summary), cudaHostAllocDefault);
    if (!e) e = cudaHostAlloc((void**)&h->h_abort, 16, cudaHostAllocMapped);
    if (e) {
        const char* msg = cudaGetErrorString(e);
        free_all(h);
        cudaGetLastError();
        return fail(e == cudaErrorMemoryAllocation ? WL_ENOMEM : WL_ECUDA, "allocation failed: %s", msg);
    }
    CU(cudaHostGetDevicePointer((void**)&h->d_abort, h->h_abort, 0));
    *h->h_abort = 0;
    CU(cudaMemcpyAsync(h->d_desc, lo.desc.data(), lo.nlines * sizeof(LineDesc),
                       cudaMemcpyHostToDevice, h->s));
    std::vector<int32_t> ident(lo.nlines);
    for (int l = 0; l < lo.nlines; ++l) ident[l] = l;
    CU(cudaMemcpyAsync(h->d_ident, ident.data(), lo.nlines * 4, cudaMemcpyHostToDevice, h->s));
    CU(cudaMemsetAsync(h->d_deadline, 0, 32, h->s));
    CU(cudaStreamSynchronize(h->s));
    h->allocated = true;
    return WL_OK;
}

Geo make_geo(const wl_ctx* h) { return wl::make_geo(h->g.type, (LatticeShape)h->g.type, h->g.L, h->g.N, h->g.NB, h->lo.W); }

int32_t* queue_place(const wl_ctx* h) { return reinterpret_cast<int32_t*>(h->d_deadline + 2); }

// The work queue: selected lines by ascending l.  A slice that ends by moves takes every
// line equally far; batches take longest over a move where few up spins make neighbouring
// steps draw the same list slot, so these lines go first.  One that ends by time goes
// through the queue from its other end (queue_line).
wl_status upload_queue(wl_ctx* h)
{
    std::vector<int32_t> order;
    for (int l = h->ell_min; l <= h->ell_max; ++l)
        if (line_selected(h, l)) order.push_back(l);
    h->nqueue = (int)order.size();
    CU(cudaMemcpyAsync(h->d_order, order.data(), order.size() * 4, cudaMemcpyHostToDevice, h->s));
    CU(cudaMemsetAsync(queue_place(h), 0, 8, h->s));
    return WL_OK;
}

// The exp threshold table of ln f_min = u on the device, kept while u stays the same:
// the host's own build of it, in the long double that is software on the machines
// this GPU comes with, takes 2 ms, as long as a small walk.
wl_status exp_table(wl_ctx* h, double u)
{
    if (h->table_u != u) {
        const int q = host_table_q(u);
        if (q < 0) return fail(WL_EINVAL, "ln_f_min %g out of range", u);
        h->table_u = 0.0;
        h->table_checked = false;
        CU(launch_exp_table(u, q, h->d_table64, h->s));
        h->table64.assign(kTableN, 0);
        CU(cudaMemcpyAsync(h->table64.data(), h->d_table64, kTableN * 8, cudaMemcpyDeviceToHost, h->s));
        CU(cudaStreamSynchronize(h->s));
        std::vector<uint32_t> t32(kTableN);
        t32[0] = 0xFFFFFFFFu;   // entry 0 (2^32) is implicit in the kernel
        for (int i = 1; i < kTableN; ++i) t32[i] = (uint32_t)h->table64[i];
        CU(cudaMemcpyAsync(h->d_table, t32.data(), kTableN * 4, cudaMemcpyHostToDevice, h->s));
        h->table_u = u;
        h->q = q;
    }
    if (h->det && !h->table_checked) {
        std::vector<uint64_t> ref;
        host_table(u, h->q, ref);
        for (int i = 0; i < kTableN; ++i)
            if (ref[i] != h->table64[i])
                return fail(WL_EMISMATCH, "exp table entry %d: device %llu host %llu", i,
                            (unsigned long long)h->table64[i], (unsigned long long)ref[i]);
        h->table_checked = true;
    }
    return WL_OK;
}

InitArgs init_args(const wl_ctx* h, double u)
{
    InitArgs a;
    a.g = make_geo(h);
    a.desc = h->d_desc;
    a.st = h->d_st;
    a.perm = h->d_perm;
    a.spins = h->d_spins;
    a.lng = h->d_lng;
    a.hist = h->d_hist;
    a.pstride = h->lo.pstride;
    a.nlines = h->nqueue;
    a.seed = h->seed;
    a.F0 = std::llround(1.0 / u);
    a.order = h->d_order;
    return a;
}

int init_lattice(const wl_ctx* h) { return h->g.type == WL_SQUARE_OPEN ? (int)kSquareOpen : h->g.type; }

wl_status initialise(wl_ctx* h, double u, int flat_pm)
{
    wl_status st = exp_table(h, u);
    if (st) return st;
    st = upload_queue(h);
    if (st) return st;
    CU(cudaMemsetAsync(h->d_flags, 0, 16, h->s));
    // lines outside [ell_min, ell_max], or not in a selected set, are marked
    // converged with t = 0 so that no launch touches them
    CU(launch_blank_states(h->d_st, h->lo.nlines, h->s));
    const InitArgs a = init_args(h, u);
    CU(cudaEventRecord(h->ev_i0, h->s));
    CU(launch_init(init_lattice(h), h->lo.idx16, a, h->s));
    CU(cudaEventRecord(h->ev_i1, h->s));
    h->u = u;
    h->flat_pm = flat_pm;
    h->initialized = true;
    h->assembled = false;
    return WL_OK;
}

WalkArgs base_args(wl_ctx* h)
{
    WalkArgs a{};
    a.g = make_geo(h);
    a.desc = h->d_desc;
    a.st = h->d_st;
    a.perm = h->d_perm;
    a.spins = h->d_spins;
    a.lng = h->d_lng;
    a.hist = h->d_hist;
    a.table = h->d_table;
    a.order = h->d_order;
    a.qnext = h->d_qheads + h->lo.nlines;
    a.nqueue = h->nqueue;
    a.q = h->q;
    a.seg_per_log2 = (float)(std::log(2.0) / (std::ldexp(1.0, h->q) * h->u));
    a.inv_u = (float)(1.0 / h->u);
    a.seed = h->seed;
    a.flat_pm = h->flat_pm;
    a.pstride = h->lo.pstride;
    a.same_f_resets = h->same_f_resets;
    a.C = h->C;
    a.C_per_bin = h->C_per_bin;
    a.budget = h->budget;
    a.slice_moves = h->slice_moves;
    a.deadline_ns = h->d_deadline;
    a.slice_end_ns = h->slice_ms > 0 ? h->d_deadline + 1 : nullptr;
    a.abort_flag = h->d_abort;
    a.flags = h->d_flags;
    return a;
}

int kernel_lattice(const wl_ctx* h);

// Shape of the persistent form for the lines still running (`active` of them).
// The count is rounded up to whole walkers per SM, so the shape (and with it the
// captured graph) changes only when that number does.
wl_status persistent_shape(wl_ctx* h, int S, int active, Shape* sh)
{
    const int per_sm = h->num_sms * (32 / S);
    const int lines = std::min<int64_t>(h->nqueue, (int64_t)((active + per_sm - 1) / per_sm) * per_sm);
    const ShapeKey k{kernel_lattice(h), S, h->det != 0, h->lo.idx16, h->g.L, h->g.N, h->lo.pstride,
                     h->lo.desc.back().nbins, std::max(lines, 1), h->tail != 0 && S == 32};
    return plan_shape(k, sh);
}

static void set_turns(wl_ctx* h, const Shape& sh, WalkArgs* a)
{
    a->turns = line_turns(sh, h->running, std::min(h->slice_moves, h->budget));
    if (a->turns > 1) a->turn = h->d_qheads;
}

// The walker's arguments for a slice of the persistent form.
WalkArgs slice_args(wl_ctx* h, const Shape& sh)
{
    WalkArgs a = base_args(h);
    set_slot(sh.slot, &a);
    set_turns(h, sh, &a);
    if (h->slice_ms > 0) a.first = queue_place(h);
    return a;
}

// One slice of the persistent form on stream h->s (capturable).
wl_status enqueue_slice(wl_ctx* h, int S, const Shape& sh)
{
    const WalkArgs a = slice_args(h, sh);
    if (a.turns > 1)
        CU(cudaMemsetAsync(h->d_qheads, 0, (size_t)(h->lo.nlines + 1) * 4, h->s));     // with qnext
    else
        CU(cudaMemsetAsync(a.qnext, 0, 4, h->s));
    const int walkers = (int)(sh.grid * (sh.slot.lone ? 1u : sh.block / (unsigned)S));
    if (h->slice_ms > 0)
        CU(launch_begin_slice(h->d_deadline + 1, (uint64_t)h->slice_ms * 1000000ull, queue_place(h), walkers,
                              h->nqueue, h->s));
    CU(launch_walk(kernel_lattice(h), S, h->det != 0, h->lo.idx16, sh.grid, sh.block, sh.smem, h->s, a));
    CU(launch_summary(h->d_st, h->lo.nlines, h->budget, h->d_flags, h->d_summary, h->s));
    CU(cudaMemcpyAsync(h->h_summary, h->d_summary, sizeof(Summary), cudaMemcpyDeviceToHost, h->s));
    return WL_OK;
}

wl_status run_slice(wl_ctx* h, int S, const Shape& sh, bool use_graph)
{
    if (!use_graph) {
        wl_status st = enqueue_slice(h, S, sh);
        if (st) return st;
        h->launches += 2;
        return WL_OK;
    }
    const WalkArgs now = slice_args(h, sh);
    // everything baked into the graph: the kernel (S, the acceptance rule, fields of its
    // arguments), its launch, its arguments, and the time limit set before it
    const bool same = h->graph && h->graph_S == S && h->graph_det == h->det && h->graph_grid == sh.grid &&
                      h->graph_block == sh.block && h->graph_smem == sh.smem && h->graph_slice_ms == h->slice_ms &&
                      memcmp(&h->graph_args, &now, sizeof now) == 0;
    if (!same) {
        if (h->graph) cudaGraphExecDestroy(h->graph);
        h->graph = nullptr;
        cudaGraph_t g;
        CU(cudaStreamBeginCapture(h->s, cudaStreamCaptureModeThreadLocal));
        wl_status st = enqueue_slice(h, S, sh);
        cudaError_t e = cudaStreamEndCapture(h->s, &g);
        if (st) return st;
        if (e != cudaSuccess) return fail(WL_ECUDA, "graph capture failed: %s", cudaGetErrorString(e));
        e = cudaGraphInstantiate(&h->graph, g, 0);
        cudaGraphDestroy(g);
        if (e != cudaSuccess) return fail(WL_ECUDA, "graph instantiate failed: %s", cudaGetErrorString(e));
        h->graph_S = S;
        h->graph_det = h->det;
        h->graph_grid = sh.grid;
        h->graph_block = sh.block;
        h->graph_smem = sh.smem;
        h->graph_slice_ms = h->slice_ms;
        memcpy(&h->graph_args, &now, sizeof now);
    }
    CU(cudaGraphLaunch(h->graph, h->s));
    h->launches += 2;
    return WL_OK;
}

// What a slice's summary says: the lines that still run, and stop conditions on the device.
wl_status check_flags(wl_ctx* h, const Summary& sm)
{
    h->running = sm.active;
    if (sm.flags & 8) return fail(WL_ECUDA, "walker state invariant broken (k' outside its bins)");
    if (sm.overflow || (sm.flags & 4)) return fail(WL_EOVERFLOW, "a histogram bin exceeded 2^63-1 within one stage");
    if (sm.flags & 3) {
        CU(cudaMemsetAsync(h->d_flags, 0, 16, h->s));
        *h->h_abort = 0;
        if (sm.flags & 2) return fail(WL_EABORTED, "aborted");
        return fail(WL_ETIMEOUT, "device deadline reached");
    }
    return WL_OK;
}

// Walker specialisation: the square lattice with L a power of two takes the
// shift-and-mask geometry.
int kernel_lattice(const wl_ctx* h)
{
    if (h->g.type == WL_SQUARE && (h->g.L & (h->g.L - 1)) == 0) return kSquareP2;
    if (h->g.type == WL_SQUARE_OPEN) return kSquareOpen;
    return h->g.type;
}

// 32 lanes per walker: the fastest batches of every lattice measured (64x64: 3.7e9 moves/s
// with 32 lanes, 3.5e9 with 16, 2.6e9 with 8; 128x128: 1.24e10, 6.0e9, 5.2e9).
int pick_mapping_default(const wl_ctx*)
{
    return 32;
}

// Persistent form: slices until every selected line converged or hit the
// budget, or the run is stopped.
//
// Shape: a block per line where plan_shape finds that faster ("tail" = 1 and 32 lanes or
// none given).  Otherwise batches; their lane count is fixed by the "mapping" option, or
// (mapping = 0) tuned online over real slices: each candidate (32, 16, 8 lanes per walker)
// walks one slice, timed with CUDA events, then the fastest is used; the candidates are
// timed again when the acceptance rate has moved by more than 0.15 since (the best count
// depends on it).  Every shape and count walks the same chain, so the choice never
// changes results.
wl_status run_persistent(wl_ctx* h, std::chrono::steady_clock::time_point t_start)
{
    const TuneKey key{h->g.type, h->g.L, h->det};
    int64_t prev_moves = -1, prev_accepts = 0;
    double last_accept = -1.0;
    int tried = -1;                       // candidate timed by the current slice
    for (;;) {
        int curS = h->mapping;
        tried = -1;
        const int active = prev_moves < 0 ? h->nqueue : h->h_summary->active;
        // a block per line, where that is the faster shape, needs no tuning
        Shape sh;
        wl_status st = WL_OK;
        bool lone = false;
        if (h->tail && (h->mapping == 0 || h->mapping == 32)) {
            st = persistent_shape(h, 32, active, &sh);
            if (st) return st;
            lone = sh.slot.lone;
        }
        if (lone) {
            curS = 32;
        } else if (curS == 0) {
            std::lock_guard<std::mutex> lk(g_tune_mu);
            TuneRec& tr = g_tune_cache[key];
            if (tr.best && last_accept >= 0.0 && tr.accept >= 0.0 && std::fabs(last_accept - tr.accept) > 0.15)
                tr = TuneRec();           // the walk has changed character: time the candidates again
            for (int c = 0; c < 3 && tried < 0; ++c)
                if (tr.rate[c] < 0.0) tried = c;
            curS = tried >= 0 ? kTuneS[tried] : tr.best;
        }
        if (!lone) st = persistent_shape(h, curS, h->tail ? active : h->nqueue, &sh);
        if (st) return st;
        if (prev_moves < 0 && (lone || h->mapping != 0)) {
            prev_moves = 0;           // nothing is tuned
        } else if (prev_moves < 0) {
            // moves before this run, for the tuning rates
            CU(launch_summary(h->d_st, h->lo.nlines, h->budget, h->d_flags, h->d_summary, h->s));
            CU(cudaMemcpyAsync(h->h_summary, h->d_summary, sizeof(Summary), cudaMemcpyDeviceToHost, h->s));
            CU(cudaStreamSynchronize(h->s));
            prev_moves = h->h_summary->moves;
            prev_accepts = h->h_summary->accepts;
        }
        CU(cudaEventRecord(h->ev_t0, h->s));
        st = run_slice(h, curS, sh, true);
        if (st) return st;
        CU(cudaEventRecord(h->ev_t1, h->s));
        CU(cudaStreamSynchronize(h->s));
        const Summary sm = *h->h_summary;
        h->last_mapping = curS;
        h->last_lone = sh.slot.lone != 0;
        const int64_t dm = sm.moves - prev_moves;
        if (dm > 0) last_accept = (double)(sm.accepts - prev_accepts) / (double)dm;
        if (tried >= 0 && dm > 0) {
            float ms = 0;
            CU(cudaEventElapsedTime(&ms, h->ev_t0, h->ev_t1));
            std::lock_guard<std::mutex> lk(g_tune_mu);
            TuneRec& tr = g_tune_cache[key];
            tr.rate[tried] = (double)dm / std::max(1e-6, (double)ms);
            if (tr.accept < 0.0) tr.accept = last_accept;
            bool all = true;
            int bi = 0;
            for (int c = 0; c < 3; ++c) {
                all &= tr.rate[c] >= 0.0;
                if (tr.rate[c] > tr.rate[bi]) bi = c;
            }
            if (all) tr.best = kTuneS[bi];
        }
        prev_moves = sm.moves;
        prev_accepts = sm.accepts;
        st = check_flags(h, sm);
        if (st) return st;
        if (sm.active == 0) break;
        const double el = std::chrono::duration<double>(std::chrono::steady_clock::now() - t_start).count();
        if ((sm.flags & 1) || (h->timeout_ms > 0 && el * 1000.0 > (double)h->timeout_ms)) {
            CU(cudaMemsetAsync(h->d_flags, 0, 16, h->s));
            return fail(WL_ETIMEOUT, "timeout after %.1f ms", el * 1000.0);
        }
        if (*h->h_abort) {
            *h->h_abort = 0;
            return fail(WL_EABORTED, "aborted");
        }
    }
    return WL_OK;
}

// Plain form: one launch per line (one walker group per launch) issued
// round-robin over a pool of streams; each launch runs its line to the budget
// or to convergence.
wl_status run_plain(wl_ctx* h)
{
    int S = h->mapping ? h->mapping : pick_mapping_default(h);
    h->last_mapping = S;
    h->last_lone = false;
    const int npool = 128;      // the device runs at most 128 kernels at once
    while ((int)h->pool.size() < npool) {
        cudaStream_t st;
        CU(cudaStreamCreateWithFlags(&st, cudaStreamNonBlocking));
        h->pool.push_back(st);
    }
    // one group per launch; as many launches as lines may share the SMs
    Shape sh;
    const ShapeKey key{kernel_lattice(h), S, h->det != 0, h->lo.idx16, h->g.L, h->g.N, h->lo.pstride,
                       h->lo.desc.back().nbins, h->nqueue, false};
    wl_status ps = plan_shape(key, &sh);
    if (ps) return ps;
    const size_t smem = (size_t)sh.slot.bytes;
    CU(cudaMemsetAsync(h->d_qheads, 0, h->lo.nlines * 4, h->s));
    CU(cudaEventRecord(h->ev_join, h->s));
    for (auto st : h->pool) CU(cudaStreamWaitEvent(st, h->ev_join, 0));
    WalkArgs a = base_args(h);
    set_slot(sh.slot, &a);
    a.nqueue = 1;
    std::vector<LineState> st_host(h->lo.nlines);
    for (;;) {
        // one launch per unfinished line, each running one slice of that line
        CU(cudaMemcpyAsync(st_host.data(), h->d_st, st_host.size() * sizeof(LineState),
                           cudaMemcpyDeviceToHost, h->s));
        CU(cudaMemsetAsync(h->d_qheads, 0, h->lo.nlines * 4, h->s));
        CU(cudaStreamSynchronize(h->s));
        CU(cudaEventRecord(h->ev_join, h->s));
        for (auto st : h->pool) CU(cudaStreamWaitEvent(st, h->ev_join, 0));
        int issued = 0;
        for (int l = h->ell_min; l <= h->ell_max; ++l) {
            if (!line_selected(h, l) || st_host[l].status != 0 || st_host[l].t >= h->budget) continue;
            a.order = h->d_ident + l;
            a.qnext = h->d_qheads + l;
            cudaStream_t st = h->pool[issued % npool];
            CU(launch_walk(kernel_lattice(h), S, h->det != 0, h->lo.idx16, dim3(1), dim3(S), smem, st, a));
            ++issued;
        }
        for (auto st : h->pool) {
            CU(cudaEventRecord(h->ev_join, st));
            CU(cudaStreamWaitEvent(h->s, h->ev_join, 0));
        }
        h->launches += issued + 1;
        CU(launch_summary(h->d_st, h->lo.nlines, h->budget, h->d_flags, h->d_summary, h->s));
        CU(cudaMemcpyAsync(h->h_summary, h->d_summary, sizeof(Summary), cudaMemcpyDeviceToHost, h->s));
        CU(cudaStreamSynchronize(h->s));
        const Summary sm = *h->h_summary;
        wl_status fs = check_flags(h, sm);
        if (fs) return fs;
        if (sm.active == 0 || issued == 0) break;
    }
    return WL_OK;
}

bool valid_handle(wl_handle h) { return h != nullptr; }

}  // namespace

namespace wl {
namespace rt {

wl_status prepare(wl_ctx* h, double ln_f_min, double flatness, cudaStream_t after)
{
    if (!(ln_f_min >= 1e-10 && ln_f_min <= 0.5)) return fail(WL_EINVAL, "ln_f_min must be in [1e-10, 0.5]");
    if (!(flatness > 0.0 && flatness <= 1.0)) return fail(WL_EINVAL, "flatness must be in (0, 1]");
    if (h->ell_min > h->ell_max) return fail(WL_EINVAL, "ell_min > ell_max");
    const int flat_pm = (int)std::lround(flatness * 1000.0);
    if (flat_pm < 1) return fail(WL_EINVAL, "flatness below 0.001");
    wl_status st = allocate(h);
    if (st) return st;
    if (after) {
        CU(cudaEventRecord(h->ev_join, after));
        CU(cudaStreamWaitEvent(h->s, h->ev_join, 0));
    }
    if (!h->initialized) {
        st = initialise(h, ln_f_min, flat_pm);
        if (st) return st;
        h->launches += 2;
    } else if (ln_f_min != h->u || flat_pm != h->flat_pm) {
        return fail(WL_EINVAL, "a continued run must use the same ln_f_min and flatness");
    }
    h->running = h->nqueue;
    h->assembled = false;
    return WL_OK;
}

void set_slot(const Slot& slot, WalkArgs* a)
{
    a->slot_bytes = slot.bytes;
    a->off_sites = slot.off_sites;
    a->off_win = slot.off_win;
    a->off_rec = slot.off_rec;
    a->win_bins = slot.win;
    a->owner_mask = slot.owner_mask;
    a->stage_perm = slot.stage_perm;
    a->stage_sites = slot.stage_sites;
    a->off_perm = slot.off_perm;
    a->lone = slot.lone;
}

static cudaError_t walk_attrs(const ShapeKey& k, const Slot& slot, size_t smem, int threads, int* bps)
{
    WalkArgs a{};
    set_slot(slot, &a);
    a.g.shape = k.lattice == kTriangular ? kShapeTriangular : kShapeSquare;      // picks the kernel
    return walk_kernel_attrs(k.lattice, k.S, k.det, k.idx16, smem, threads, a, bps);
}

wl_status plan_shape(const ShapeKey& k, Shape* sh)
{
    int dev = 0;
    Gpu gpu{};
    CU(cudaGetDevice(&dev));
    CU(cudaDeviceGetAttribute(&gpu.sms, cudaDevAttrMultiProcessorCount, dev));
    CU(cudaDeviceGetAttribute(&gpu.per_block, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
    CU(cudaDeviceGetAttribute(&gpu.per_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev));
    CU(cudaDeviceGetAttribute(&gpu.reserved, cudaDevAttrReservedSharedMemoryPerBlock, dev));
    cudaError_t e = cudaSuccess;
    auto resident = [&](const Slot& slot, size_t smem, int threads) {
        int bps = 0;
        e = walk_attrs(k, slot, smem, threads, &bps);
        return e == cudaSuccess ? bps : -1;
    };
    switch (plan_shape(k, gpu, resident, sh)) {
    case Planned::ok: return WL_OK;
    case Planned::none_fits: return fail(WL_ECUDA, "no walker shape fits shared memory (S=%d)", k.S);
    default: return fail(WL_ECUDA, "walker attributes: %s", cudaGetErrorString(e));
    }
}

wl_status choose_shape(wl_ctx* h, int* S, Shape* sh)
{
    int m = h->mapping;
    if (m == 0) {
        std::lock_guard<std::mutex> lk(g_tune_mu);
        auto it = g_tune_cache.find({h->g.type, h->g.L, h->det});
        m = it != g_tune_cache.end() && it->second.best ? it->second.best : pick_mapping_default(h);
    }
    *S = m;
    h->last_mapping = m;
    return persistent_shape(h, m, h->nqueue, sh);
}

wl_status launch_slice_async(wl_ctx* h, int S, const Shape& sh) { return run_slice(h, S, sh, true); }

wl_status summary_status(wl_ctx* h, const Summary& sm) { return check_flags(h, sm); }

size_t handle_bytes(const wl_ctx* h) { return required_bytes(h->g, h->lo); }

wl_status assemble_copy_async(wl_ctx* h, double* dst, size_t cap, size_t* n_out)
{
    if (!h->initialized) return fail(WL_ESTATE, "no run to assemble");
    const LineDesc& a = h->lo.desc[h->ell_min];
    const LineDesc& b = h->lo.desc[h->ell_max];
    const size_t n = (size_t)(b.bin_off + b.nbins - a.bin_off);
    if (n_out) *n_out = n;
    if (!dst || cap < n) return fail(WL_EINVAL, "output capacity %zu < %zu bins", cap, n);
    CU(launch_assemble(h->d_desc, h->d_order, h->d_lng, h->d_hist, h->g.N, h->nqueue, h->u, h->d_out, h->s));
    CU(cudaMemcpyAsync(dst, h->d_out + a.bin_off, n * 8, cudaMemcpyDeviceToHost, h->s));
    h->assembled = true;
    return WL_OK;
}

int table_shift(double u)
{
    const double need = 32.0 * std::log(2.0);
    for (int q = 0; q < 40; ++q)
        if (4095.0 * std::ldexp(1.0, q) * u >= need) return q;
    return -1;
}

uint64_t table_entry(double u, int q, int i)
{
    volatile double x = (double)((uint64_t)i << q) * u;
    const long double v = std::ldexp(std::exp(-(long double)x), 32) + 0.5L;
    return (uint64_t)std::floor(v);
}

}  // namespace rt
}  // namespace wl

extern "C" {

const char* wl_last_error(void) { return g_err.c_str(); }

size_t wl_required_bytes(wl_lattice lattice, int L)
{
    LatInfo g;
    if (!lattice_info((int)lattice, L, &g)) return 0;
    Layout lo = make_layout(g);
    return required_bytes(g, lo);
}

wl_status wl_create(wl_lattice lattice, int L, wl_handle* out)
{
    if (!out) return fail(WL_EINVAL, "out is NULL");
    *out = nullptr;
    LatInfo g;
    if (!lattice_info((int)lattice, L, &g))
        return fail(WL_EINVAL, "unsupported lattice %d with L=%d (L >= 3, N <= 2^20)", (int)lattice, L);
    wl_ctx* h = new (std::nothrow) wl_ctx();
    if (!h) return fail(WL_ENOMEM, "host allocation failed");
    h->g = g;
    h->lo = make_layout(g);
    h->ell_min = 0;
    h->ell_max = h->lo.nlines - 1;
    *out = h;
    g_err.clear();
    return WL_OK;
}

wl_status wl_destroy(wl_handle h)
{
    if (!valid_handle(h)) return fail(WL_EINVAL, "NULL handle");
    free_all(h);
    delete h;
    return WL_OK;
}

wl_status wl_set_option(wl_handle h, const char* key, int64_t v)
{
    if (!valid_handle(h) || !key) return fail(WL_EINVAL, "NULL handle or key");
    const std::string k(key);
    const bool semantic = (k == "seed" || k == "deterministic" || k == "check_interval" || k == "check_per_bin" ||
                           k == "ell_min" || k == "ell_max" || k == "same_f_resets");
    if (semantic && h->initialized)
        return fail(WL_ESTATE, "option '%s' changes the walk; call wl_reset first", key);
    if (k == "seed") {
        if (v < 0 || v > 0xFFFFFFFFll) return fail(WL_EINVAL, "seed must fit 32 bits");
        h->seed = (uint32_t)v;
    } else if (k == "deterministic") {
        h->det = v ? 1 : 0;
    } else if (k == "check_interval") {
        if (v < 1 || v > 0x7FFFFFFFll) return fail(WL_EINVAL, "check_interval must be in [1, 2^31-1]");
        h->C = v;
    } else if (k == "check_per_bin") {
        if (v < 0 || v > (1ll << 24)) return fail(WL_EINVAL, "check_per_bin must be in [0, 2^24]");
        h->C_per_bin = v;
    } else if (k == "move_budget") {
        if (v < 0) return fail(WL_EINVAL, "move_budget must be >= 0");
        h->budget = v;
    } else if (k == "mapping") {
        if (!(v == 0 || v == 1 || v == 2 || v == 4 || v == 8 || v == 16 || v == 32))
            return fail(WL_EINVAL, "mapping must be 0, 1, 2, 4, 8, 16 or 32");
        h->mapping = (int)v;
    } else if (k == "form") {
        if (v != 0 && v != 1) return fail(WL_EINVAL, "form must be 0 or 1");
        h->form = (int)v;
    } else if (k == "stream") {
        h->user_stream = (cudaStream_t)(intptr_t)v;
        h->has_user_stream = true;
    } else if (k == "slice_moves") {
        if (v < 1) return fail(WL_EINVAL, "slice_moves must be >= 1");
        h->slice_moves = v;
    } else if (k == "slice_ms") {
        if (v < 0) return fail(WL_EINVAL, "slice_ms must be >= 0");
        h->slice_ms = v;
    } else if (k == "timeout_ms") {
        if (v < 0) return fail(WL_EINVAL, "timeout_ms must be >= 0");
        h->timeout_ms = v;
    } else if (k == "hbm_budget") {
        if (v < 0) return fail(WL_EINVAL, "hbm_budget must be >= 0");
        h->hbm_budget = v;
    } else if (k == "same_f_resets") {
        if (v < 0 || v > 1000000) return fail(WL_EINVAL, "same_f_resets must be in [0, 10^6]");
        h->same_f_resets = (int)v;
    } else if (k == "tail") {
        if (v != 0 && v != 1) return fail(WL_EINVAL, "tail must be 0 or 1");
        h->tail = (int)v;
    } else if (k == "ell_min" || k == "ell_max") {
        if (v < 0 || v >= h->lo.nlines) return fail(WL_EINVAL, "%s must be in [0, %d]", key, h->lo.nlines - 1);
        (k == "ell_min" ? h->ell_min : h->ell_max) = (int)v;
        h->sel.clear();
    } else {
        return fail(WL_EINVAL, "unknown option '%s'", key);
    }
    return WL_OK;
}

wl_status wl_get_option(wl_handle h, const char* key, int64_t* v)
{
    if (!valid_handle(h) || !key || !v) return fail(WL_EINVAL, "NULL argument");
    const std::string k(key);
    if (k == "seed") *v = h->seed;
    else if (k == "deterministic") *v = h->det;
    else if (k == "check_interval") *v = h->C;
    else if (k == "check_per_bin") *v = h->C_per_bin;
    else if (k == "move_budget") *v = h->budget;
    else if (k == "mapping") *v = h->mapping;
    else if (k == "form") *v = h->form;
    else if (k == "stream") *v = (int64_t)(intptr_t)h->user_stream;
    else if (k == "slice_moves") *v = h->slice_moves;
    else if (k == "timeout_ms") *v = h->timeout_ms;
    else if (k == "slice_ms") *v = h->slice_ms;
    else if (k == "tuned_mapping") {
        // the lane count the tuner settled on for this lattice and mode (0: not yet)
        std::lock_guard<std::mutex> lk(g_tune_mu);
        auto it = g_tune_cache.find({h->g.type, h->g.L, h->det});
        *v = it != g_tune_cache.end() ? it->second.best : 0;
    }
    else if (k == "block_per_line") *v = h->last_lone;
    else if (k == "hbm_budget") *v = h->hbm_budget;
    else if (k == "ell_min") *v = h->ell_min;
    else if (k == "same_f_resets") *v = h->same_f_resets;
    else if (k == "tail") *v = h->tail;
    else if (k == "ell_max") *v = h->ell_max;
    else if (k == "N") *v = h->g.N;
    else if (k == "NB") *v = h->g.NB;
    else if (k == "z") *v = h->g.z;
    else if (k == "k_step") *v = h->g.kstep;
    else if (k == "lines") *v = h->lo.nlines;
    else if (k == "bins") *v = h->lo.nbins_total;
    else if (k == "device_bytes") *v = (int64_t)(required_bytes(h->g, h->lo) + h->thermo_bytes);
    else return fail(WL_EINVAL, "unknown option '%s'", key);
    return WL_OK;
}

wl_status wl_reset(wl_handle h)
{
    if (!valid_handle(h)) return fail(WL_EINVAL, "NULL handle");
    if (h->ell_min > h->ell_max) return fail(WL_EINVAL, "ell_min > ell_max");
    h->initialized = false;
    h->assembled = false;
    return WL_OK;
}

wl_status wl_select_lines(wl_handle h, const int32_t* ells, int n)
{
    if (!valid_handle(h)) return fail(WL_EINVAL, "NULL handle");
    if (h->initialized) return fail(WL_ESTATE, "the line set changes the walk; call wl_reset first");
    if (n < 0 || (n > 0 && !ells)) return fail(WL_EINVAL, "bad line list");
    if (n == 0) {
        h->sel.clear();
        h->ell_min = 0;
        h->ell_max = h->lo.nlines - 1;
        return WL_OK;
    }
    std::vector<uint8_t> sel(h->lo.nlines, 0);
    int lo = h->lo.nlines, hi = -1;
    for (int x = 0; x < n; ++x) {
        const int l = ells[x];
        if (l < 0 || l >= h->lo.nlines) return fail(WL_EINVAL, "line %d outside [0, %d]", l, h->lo.nlines - 1);
        sel[l] = 1;
        lo = std::min(lo, l);
        hi = std::max(hi, l);
    }
    h->sel.swap(sel);
    h->ell_min = lo;
    h->ell_max = hi;
    return WL_OK;
}

wl_status wl_abort(wl_handle h)
{
    if (!valid_handle(h)) return fail(WL_EINVAL, "NULL handle");
    if (h->h_abort) *(volatile int32_t*)h->h_abort = 1;
    return WL_OK;
}

wl_status wl_run(wl_handle h, double ln_f_min, double flatness)
{
    if (!valid_handle(h)) return fail(WL_EINVAL, "NULL handle");
    const auto t_start = std::chrono::steady_clock::now();
    h->launches = 0;
    wl_status st = wl::rt::prepare(h, ln_f_min, flatness, h->has_user_stream ? h->user_stream : nullptr);
    if (st) return st;
    CU(launch_set_deadline(h->d_deadline, (uint64_t)h->timeout_ms * 1000000ull, h->s));
    CU(cudaEventRecord(h->ev0, h->s));
    st = h->form == 0 ? run_persistent(h, t_start) : run_plain(h);
    cudaError_t e = cudaEventRecord(h->ev1, h->s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(h->s);
    if (e == cudaSuccess) {
        float ms = 0;
        if (cudaEventElapsedTime(&ms, h->ev0, h->ev1) == cudaSuccess) h->walk_ms = ms;
    }
    if (h->has_user_stream) {
        cudaEventRecord(h->ev_join, h->s);
        cudaStreamWaitEvent(h->user_stream, h->ev_join, 0);
    }
    if (st) return st;
    if (e != cudaSuccess) return fail(WL_ECUDA, "run failed: %s", cudaGetErrorString(e));
    const Summary sm = *h->h_summary;
    int selected = 0;
    for (int l = h->ell_min; l <= h->ell_max; ++l) selected += line_selected(h, l);
    const int outside = h->lo.nlines - selected;
    if (sm.converged - outside < selected) return fail(WL_ENOTCONVERGED, "move budget reached before convergence");
    g_err.clear();
    return WL_OK;
}

wl_status wl_assemble(wl_handle h)
{
    if (!valid_handle(h)) return fail(WL_EINVAL, "NULL handle");
    if (!h->initialized) return fail(WL_ESTATE, "no run to assemble");
    if (h->has_user_stream) {
        CU(cudaEventRecord(h->ev_join, h->user_stream));
        CU(cudaStreamWaitEvent(h->s, h->ev_join, 0));
    }
    CU(cudaEventRecord(h->ev0, h->s));
    CU(launch_assemble(h->d_desc, h->d_order, h->d_lng, h->d_hist, h->g.N, h->nqueue, h->u, h->d_out, h->s));
    CU(cudaEventRecord(h->ev1, h->s));
    if (h->has_user_stream) {
        CU(cudaEventRecord(h->ev_join, h->s));
        CU(cudaStreamWaitEvent(h->user_stream, h->ev_join, 0));
    }
    CU(cudaEventSynchronize(h->ev1));
    float ms = 0;
    CU(cudaEventElapsedTime(&ms, h->ev0, h->ev1));
    h->assemble_ms = ms;
    h->assembled = true;
    return WL_OK;
}

wl_status wl_get_lng(wl_handle h, int ell, double* out, size_t cap, int* k_lo, int* k_step,
                     size_t* n_out)
{
    if (!valid_handle(h)) return fail(WL_EINVAL, "NULL handle");
    if (ell < 0 || ell > h->g.N) return fail(WL_EINVAL, "ell out of range");
    if (!h->assembled) return fail(WL_ESTATE, "call wl_assemble first");
    const int li = std::min(ell, h->g.N - ell);
    if (!line_selected(h, li)) return fail(WL_EINVAL, "line %d was not walked", ell);
    const LineDesc& d = h->lo.desc[li];
    if (n_out) *n_out = (size_t)d.nbins;
    if (k_lo) *k_lo = 0;
    if (k_step) *k_step = h->g.kstep;
    if (!out || cap < (size_t)d.nbins) return fail(WL_EINVAL, "output capacity %zu < %d bins", cap, d.nbins);
    CU(cudaMemcpyAsync(out, h->d_out + d.bin_off, (size_t)d.nbins * 8, cudaMemcpyDeviceToHost, h->s));
    CU(cudaStreamSynchronize(h->s));
    return WL_OK;
}

wl_status wl_get_surface(wl_handle h, double* out, size_t cap, int64_t* offsets, size_t offsets_cap,
                         size_t* n_out)
{
    if (!valid_handle(h)) return fail(WL_EINVAL, "NULL handle");
    if (!h->assembled) return fail(WL_ESTATE, "call wl_assemble first");
    const LineDesc& a = h->lo.desc[h->ell_min];
    const LineDesc& b = h->lo.desc[h->ell_max];
    const int64_t n = b.bin_off + b.nbins - a.bin_off;
    const int lines = h->ell_max - h->ell_min + 1;
    if (n_out) *n_out = (size_t)n;
    if (!out || cap < (size_t)n) return fail(WL_EINVAL, "output capacity %zu < %lld bins", cap, (long long)n);
    if (offsets) {
        if (offsets_cap < (size_t)lines + 1) return fail(WL_EINVAL, "offsets capacity too small");
        for (int l = 0; l < lines; ++l) offsets[l] = h->lo.desc[h->ell_min + l].bin_off - a.bin_off;
        offsets[lines] = n;
    }
    if (!h->sel.empty()) {
        // the lines between those of the set
        CU(launch_fill_unvisited(h->d_out + a.bin_off, (size_t)n, h->s));
        CU(launch_assemble(h->d_desc, h->d_order, h->d_lng, h->d_hist, h->g.N, h->nqueue, h->u, h->d_out, h->s));
    }
    CU(cudaMemcpyAsync(out, h->d_out + a.bin_off, (size_t)n * 8, cudaMemcpyDeviceToHost, h->s));
    CU(cudaStreamSynchronize(h->s));
    return WL_OK;
}

wl_status wl_get_stats(wl_handle h, wl_stats* out)
{
    if (!valid_handle(h) || !out) return fail(WL_EINVAL, "NULL argument");
    memset(out, 0, sizeof *out);
    for (int l = h->ell_min; l <= h->ell_max; ++l) out->lines += line_selected(h, l);
    out->mapping = h->last_mapping;
    out->form = h->form;
    out->launches = h->launches;
    out->walk_ms = h->walk_ms;
    out->assemble_ms = h->assemble_ms;
    if (h->allocated && cudaEventSynchronize(h->ev_i1) == cudaSuccess) {
        float ms = 0;
        if (cudaEventElapsedTime(&ms, h->ev_i0, h->ev_i1) == cudaSuccess) out->init_ms = ms;
        clear_stale_error();          // events not recorded yet
    }
    if (!h->initialized) return WL_OK;
    std::vector<LineState> st(h->lo.nlines);
    CU(cudaMemcpyAsync(st.data(), h->d_st, st.size() * sizeof(LineState), cudaMemcpyDeviceToHost, h->s));
    CU(cudaStreamSynchronize(h->s));
    out->min_stage = INT32_MAX;
    for (int l = h->ell_min; l <= h->ell_max; ++l) {
        if (!line_selected(h, l)) continue;
        const LineState& s = st[l];
        out->moves += s.t;
        out->accepts += s.accepts;
        out->checks += s.checks;
        out->batches += s.batches;
        out->lines_converged += s.status == 1;
        out->min_stage = std::min<int32_t>(out->min_stage, (int32_t)s.stage);
        out->max_stage = std::max<int32_t>(out->max_stage, (int32_t)s.stage);
    }
    return WL_OK;
}

wl_status wl_get_line_state(wl_handle h, int ell, int64_t* scal, int32_t* perm, uint8_t* spins,
                            int64_t* lng, int64_t* hist, uint8_t* visited)
{
    if (!valid_handle(h)) return fail(WL_EINVAL, "NULL handle");
    if (!h->initialized) return fail(WL_ESTATE, "no walker state yet");
    if (ell < 0 || ell >= h->lo.nlines) return fail(WL_EINVAL, "ell must be in [0, N/2]");
    const LineDesc& d = h->lo.desc[ell];
    const int N = h->g.N;
    if (ell >= h->ell_min && ell <= h->ell_max && !line_selected(h, ell)) {
        // between the lines of a set: not walked, and initialised only when asked for
        InitArgs a = init_args(h, h->u);
        a.st = nullptr;
        a.order = h->d_ident + ell;
        a.nlines = 1;
        CU(launch_init(init_lattice(h), h->lo.idx16, a, h->s));
    }
    if (scal) {
        LineState s;
        CU(cudaMemcpyAsync(&s, h->d_st + ell, sizeof s, cudaMemcpyDeviceToHost, h->s));
        CU(cudaStreamSynchronize(h->s));
        const int64_t v[8] = {s.k, s.t, s.F, s.stage, s.accepts, s.t_stage, s.status, s.checks};
        memcpy(scal, v, sizeof v);
    }
    if (perm) {
        const size_t isz = h->lo.idx16 ? 2 : 4;
        std::vector<uint8_t> raw((size_t)N * isz);
        CU(cudaMemcpyAsync(raw.data(), (uint8_t*)h->d_perm + (size_t)ell * h->lo.pstride * isz,
                           raw.size(), cudaMemcpyDeviceToHost, h->s));
        CU(cudaStreamSynchronize(h->s));
        for (int i = 0; i < N; ++i)
            perm[i] = isz == 2 ? (int32_t)((uint16_t*)raw.data())[i] : (int32_t)((uint32_t*)raw.data())[i];
    }
    if (spins) {
        std::vector<uint32_t> w(h->lo.W);
        CU(cudaMemcpyAsync(w.data(), h->d_spins + (size_t)ell * h->lo.W, w.size() * 4,
                           cudaMemcpyDeviceToHost, h->s));
        CU(cudaStreamSynchronize(h->s));
        for (int i = 0; i < N; ++i) spins[i] = (uint8_t)((w[i >> 5] >> (i & 31)) & 1u);
    }
    if (lng) {
        CU(cudaMemcpyAsync(lng, h->d_lng + d.bin_off, (size_t)d.nbins * 8, cudaMemcpyDeviceToHost, h->s));
        CU(cudaStreamSynchronize(h->s));
    }
    if (hist || visited) {
        std::vector<hist_t> hw(d.nbins);
        CU(cudaMemcpyAsync(hw.data(), h->d_hist + d.bin_off, (size_t)d.nbins * sizeof(hist_t),
                           cudaMemcpyDeviceToHost, h->s));
        CU(cudaStreamSynchronize(h->s));
        for (int b = 0; b < d.nbins; ++b) {
            if (hist) hist[b] = (int64_t)(hw[b] & ~kVisited);
            if (visited) visited[b] = (hw[b] & kVisited) ? 1 : 0;
        }
    }
    return WL_OK;
}

wl_status wl_thermo(wl_handle h, const double* T, int nT, const double* H, int nH, double* out)
{
    if (!valid_handle(h) || !T || !H || !out || nT < 1 || nH < 1) return fail(WL_EINVAL, "bad arguments");
    if (!h->assembled) return fail(WL_ESTATE, "call wl_assemble first");
    if (h->ell_min != 0 || h->ell_max != h->lo.nlines - 1 || !h->sel.empty())
        return fail(WL_ESTATE, "thermodynamics needs every line l = 0..N/2");
    for (int a = 0; a < nT; ++a)
        if (!(T[a] > 0.0)) return fail(WL_EINVAL, "temperatures must be > 0");
    const size_t nd = (size_t)nT + (size_t)nH + 6 * (size_t)nT * (size_t)nH;
    const size_t need = nd * sizeof(double) + thermo_scratch_bytes(h->lo.nlines, nT);
    // A small workspace is kept with the handle, inside its memory budget: to map and unmap
    // it on every call takes longer than a scan of a small surface.  A large one is given
    // back at the end of the call.
    const size_t held = required_bytes(h->g, h->lo);
    const bool keep = need <= kThermoKept && (h->hbm_budget == 0 || held + need <= (size_t)h->hbm_budget);
    if (keep && h->thermo_bytes < need) {
        if (h->d_thermo) CU(cudaFree(h->d_thermo));
        h->d_thermo = nullptr;
        h->thermo_bytes = 0;
        CU(cudaMalloc(&h->d_thermo, need));
        h->thermo_bytes = need;
    }
    void* once = nullptr;
    if (!keep) CU(cudaMallocAsync(&once, need, h->s));
    double* d = static_cast<double*>(keep ? h->d_thermo : once);
    cudaError_t e = cudaMemcpyAsync(d, T, nT * sizeof(double), cudaMemcpyHostToDevice, h->s);
    if (!e) e = cudaMemcpyAsync(d + nT, H, nH * sizeof(double), cudaMemcpyHostToDevice, h->s);
    if (!e) e = launch_thermo(h->d_desc, h->lo.nlines, h->d_out, h->g.N, h->g.NB, h->g.kstep, d, nT,
                              d + nT, nH, d + nT + nH, d + nd, h->s);
    if (!e) e = cudaMemcpyAsync(out, d + nT + nH, 6 * (size_t)nT * nH * sizeof(double),
                                cudaMemcpyDeviceToHost, h->s);
    if (once) cudaFreeAsync(once, h->s);
    if (!e) e = cudaStreamSynchronize(h->s);
    if (e) return fail(WL_ECUDA, "wl_thermo: %s", cudaGetErrorString(e));
    return WL_OK;
}

wl_status wl_get_exp_table(wl_handle h, uint64_t* table, int* q)
{
    if (!valid_handle(h)) return fail(WL_EINVAL, "NULL handle");
    if (!h->initialized || h->table64.empty()) return fail(WL_ESTATE, "no table before the first run");
    if (table) memcpy(table, h->table64.data(), kTableN * 8);
    if (q) *q = h->q;
    return WL_OK;
}

wl_status wl_accept_threshold(double ln_f_min, int deterministic, size_t n, const uint32_t* r,
                              int64_t* out)
{
    if (!(ln_f_min >= 1e-10 && ln_f_min <= 0.5)) return fail(WL_EINVAL, "ln_f_min must be in [1e-10, 0.5]");
    if (n == 0) return WL_OK;
    if (!r || !out) return fail(WL_EINVAL, "NULL argument");
    const int q = host_table_q(ln_f_min);
    uint64_t* d64 = nullptr;
    uint32_t *d32 = nullptr, *dr = nullptr;
    int64_t* dout = nullptr;
    std::vector<uint64_t> t64(kTableN), ref;
    std::vector<uint32_t> t32(kTableN);
    host_table(ln_f_min, q, ref);
    cudaError_t e = cudaMalloc(&d64, kTableN * 8);
    if (!e) e = cudaMalloc(&d32, kTableN * 4);
    if (!e) e = cudaMalloc(&dr, n * 4);
    if (!e) e = cudaMalloc(&dout, n * 8);
    if (!e) e = launch_exp_table(ln_f_min, q, d64, 0);
    if (!e) e = cudaMemcpy(t64.data(), d64, kTableN * 8, cudaMemcpyDeviceToHost);
    bool same = true;
    if (!e) {
        for (int i = 0; i < kTableN; ++i) same &= t64[i] == ref[i];
        t32[0] = 0xFFFFFFFFu;
        for (int i = 1; i < kTableN; ++i) t32[i] = (uint32_t)t64[i];
        e = cudaMemcpy(d32, t32.data(), kTableN * 4, cudaMemcpyHostToDevice);
    }
    if (!e) e = cudaMemcpy(dr, r, n * 4, cudaMemcpyHostToDevice);
    if (!e)
        e = launch_dmax(n, dr, deterministic ? 1 : 0, d32, q,
                        (float)(std::log(2.0) / (std::ldexp(1.0, q) * ln_f_min)),
                        (float)(1.0 / ln_f_min), dout, 0);
    if (!e) e = cudaMemcpy(out, dout, n * 8, cudaMemcpyDeviceToHost);
    cudaFree(d64);
    cudaFree(d32);
    cudaFree(dr);
    cudaFree(dout);
    if (e) return fail(WL_ECUDA, "wl_accept_threshold: %s", cudaGetErrorString(e));
    if (deterministic && !same) return fail(WL_EMISMATCH, "device exp table differs from the host table");
    return WL_OK;
}

wl_status wl_philox(size_t n, const uint32_t* ctr, const uint32_t* key, uint32_t* out)
{
    if (n == 0) return WL_OK;
    if (!ctr || !key || !out) return fail(WL_EINVAL, "NULL argument");
    uint32_t *dc = nullptr, *dk = nullptr, *dout = nullptr;
    cudaError_t e = cudaMalloc(&dc, n * 16);
    if (!e) e = cudaMalloc(&dk, n * 8);
    if (!e) e = cudaMalloc(&dout, n * 16);
    if (!e) e = cudaMemcpy(dc, ctr, n * 16, cudaMemcpyHostToDevice);
    if (!e) e = cudaMemcpy(dk, key, n * 8, cudaMemcpyHostToDevice);
    if (!e) e = launch_philox(n, dc, dk, dout, 0);
    if (!e) e = cudaMemcpy(out, dout, n * 16, cudaMemcpyDeviceToHost);
    cudaFree(dc);
    cudaFree(dk);
    cudaFree(dout);
    if (e) return fail(WL_ECUDA, "wl_philox: %s", cudaGetErrorString(e));
    return WL_OK;
}

}  // extern "C"
