// wl_kernels.cu -- walker initialisation, DOS assembly, the device-built exp
// threshold table, the Philox check kernel and the per-launch run summary.
#include <algorithm>
#include <cfloat>
#include <cmath>

#include "wl_kernels.cuh"

namespace wl {

// ---------------------------------------------------------------------------
// Walker initialisation (the initial state of the text around Eq. 3): one warp
// per line.  l up spins at the sites perm[0, l) of a partial Fisher-Yates
// shuffle (step t swaps perm[t] with perm[t + pick(r.x, N - t)], r = Philox
// counter (t, 0, 1, 0), key (l, seed)); U = perm[0, l), D = perm[l, N); ln g = 0,
// h = 0, ln f = 1 (F0 = round(1/u)); k0 counted from the spins.  The line l = 0
// has no exchange move: its single bin k = 0 is marked visited and it is done.
// The shuffle is a chain of l dependent swaps: it runs in shared memory where the
// list fits (A.stage; ~45 cycles a swap against ~600 from global memory: the four
// lines of the 256x256 lattice take 1.1 ms), one line per block of one warp.
// ---------------------------------------------------------------------------
template <int LAT, typename IDX>
__global__ void __launch_bounds__(32) init_kernel(const InitArgs A)
{
    extern __shared__ __align__(16) uint8_t smem[];
    const int lane = threadIdx.x & 31;
    const int li = A.order ? A.order[blockIdx.x] : (int)blockIdx.x;
    const LineDesc D = A.desc[li];
    const int N = A.g.N, W = A.g.W, ell = D.ell;
    IDX* gperm = reinterpret_cast<IDX*>(A.perm) + (size_t)li * A.pstride;
    IDX* perm = A.stage ? reinterpret_cast<IDX*>(smem) : gperm;
    uint32_t* sp = A.spins + (size_t)li * W;
    int64_t* lng = A.lng + D.bin_off;
    hist_t* hist = A.hist + D.bin_off;
    for (int n = lane; n < A.pstride; n += 32) perm[n] = (IDX)(n < N ? n : 0);
    for (int w = lane; w < W; w += 32) sp[w] = 0u;
    for (int b = lane; b < D.nbins; b += 32) {
        lng[b] = 0;
        hist[b] = 0ull;
    }
    __syncwarp();
    const uint2 key = make_uint2((uint32_t)ell, A.seed);
    const int tmax = ell < N - 1 ? ell : N - 1;
    for (int base = 0; base < tmax; base += 32) {
        const int t = base + lane;
        uint32_t j = 0;
        if (t < tmax) {
            const uint4 r = philox4x32_10(make_uint4((uint32_t)t, 0u, 1u, 0u), key);
            j = (uint32_t)t + pick(r.x, (uint32_t)(N - t));
        }
        const int cnt = tmax - base < 32 ? tmax - base : 32;
        for (int s = 0; s < cnt; ++s) {
            const uint32_t js = __shfl_sync(0xffffffffu, j, s);
            if (lane == 0) {
                const IDX x = perm[base + s];
                perm[base + s] = perm[js];
                perm[js] = x;
            }
        }
        __syncwarp();
    }
    if (A.stage)
        for (int n = lane; n < A.pstride; n += 32) gperm[n] = perm[n];
    for (int a = lane; a < ell; a += 32) {
        const uint32_t n = (uint32_t)perm[a];
        atomicOr(&sp[n >> 5], 1u << (n & 31u));
    }
    __syncwarp();
    int twice = 0;
    constexpr int z = Coord<LAT>::z;
    for (int n = lane; n < N; n += 32) {
        uint32_t nb[z];
        unsigned valid = (1u << z) - 1u;
        if constexpr (LAT == kSquareOpen) valid = open_neighbours(A.g, (uint32_t)n, nb);
        else neighbours<LAT>(A.g, (uint32_t)n, nb);
        const uint32_t sn = spin_at(sp, (uint32_t)n);
#pragma unroll
        for (int m = 0; m < z; ++m) twice += (int)(((valid >> m) & 1u) && sn != spin_at(sp, nb[m]));
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) twice += __shfl_xor_sync(0xffffffffu, twice, off);
    if (lane == 0 && A.st) {
        LineState s;
        s.k = twice / 2;
        s.t = 0;
        s.F = A.F0;
        s.stage = 0;
        s.accepts = 0;
        s.t_stage = 0;
        s.status = 0;
        s.checks = 0;
        s.batches = 0;
        if (ell == 0) {
            hist[s.k >> Coord<LAT>::kshift] = kVisited;
            s.F = 0;
            s.status = 1;
        }
        A.st[li] = s;
    }
}

// ---------------------------------------------------------------------------
// A caller's own walker state (wl_walk_noalloc): one block per running line checks
// that the list is a permutation whose first l entries are the up spins, that k is
// theirs and that there is a move to make.  The walkers take this for granted: every
// bin and site they reach, and with it every address, follows from it.  A line that
// fails gets the status and the flag of a broken invariant and is not walked.
// A site seen twice shows in a bit per site (up to 128 KB of shared memory).
// ---------------------------------------------------------------------------
constexpr int kCheckThreads = 128;

template <int LAT, typename IDX>
__global__ void __launch_bounds__(kCheckThreads) check_state_kernel(const InitArgs A, int32_t* flags)
{
    extern __shared__ uint32_t seen[];
    __shared__ int twice_all;
    const int li = blockIdx.x;
    if (A.st[li].status != 0) return;
    const LineDesc D = A.desc[li];
    const int N = A.g.N;
    const IDX* perm = reinterpret_cast<const IDX*>(A.perm) + (size_t)li * A.pstride;
    const uint32_t* sp = A.spins + (size_t)li * A.g.W;
    constexpr int z = Coord<LAT>::z;
    for (int w = threadIdx.x; w < A.g.W; w += kCheckThreads) seen[w] = 0u;
    if (threadIdx.x == 0) twice_all = 0;
    __syncthreads();
    int twice = 0, bad = D.ell < 1 || A.st[li].t < 0;
    for (int n = threadIdx.x; n < N; n += kCheckThreads) {
        const uint32_t e = (uint32_t)perm[n];
        if (e >= (uint32_t)N) {
            bad = 1;
        } else {
            const uint32_t bit = 1u << (e & 31u);
            bad |= (atomicOr(&seen[e >> 5], bit) & bit) != 0u;
            bad |= spin_at(sp, e) != (n < D.ell ? 1u : 0u);
        }
        uint32_t nb[z];
        neighbours<LAT>(A.g, (uint32_t)n, nb);
        const uint32_t sn = spin_at(sp, (uint32_t)n);
#pragma unroll
        for (int q = 0; q < z; ++q) twice += sn != spin_at(sp, nb[q]);
    }
    twice = group_sum<32>(0xffffffffu, twice);
    if ((threadIdx.x & 31) == 0) atomicAdd(&twice_all, twice);
    __syncthreads();
    bad |= A.st[li].k != twice_all / 2;
    if (__syncthreads_or(bad) && threadIdx.x == 0) {
        A.st[li].status = 3;
        atomicOr(flags, 8);
    }
}

template <int LAT, typename IDX>
static cudaError_t check_one(const InitArgs& a, int32_t* flags, cudaStream_t s)
{
    const size_t bits = (size_t)a.g.W * 4;
    if (bits > 40 * 1024) {
        const cudaError_t e = cudaFuncSetAttribute(check_state_kernel<LAT, IDX>,
                                                   cudaFuncAttributeMaxDynamicSharedMemorySize, 128 * 1024);
        if (e != cudaSuccess) return e;
    }
    check_state_kernel<LAT, IDX><<<a.nlines, kCheckThreads, bits, s>>>(a, flags);
    return cudaGetLastError();
}

cudaError_t launch_check_state(int lattice, bool idx16, const InitArgs& a, int32_t* flags, cudaStream_t s)
{
    clear_stale_error();
    if (lattice == kSquare)
        return idx16 ? check_one<kSquare, uint16_t>(a, flags, s) : check_one<kSquare, uint32_t>(a, flags, s);
    if (lattice == kTriangular)
        return idx16 ? check_one<kTriangular, uint16_t>(a, flags, s) : check_one<kTriangular, uint32_t>(a, flags, s);
    return idx16 ? check_one<kCubic, uint16_t>(a, flags, s) : check_one<kCubic, uint32_t>(a, flags, s);
}

template <int LAT, typename IDX>
static cudaError_t init_one(InitArgs a, cudaStream_t s)
{
    // any list that fits a block's shared memory
    const size_t list = (size_t)a.pstride * sizeof(IDX);
    int dev = 0, optin = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e != cudaSuccess) return e;
    a.stage = list <= (size_t)optin;
    if (a.stage && list > 48 * 1024) {
        e = cudaFuncSetAttribute(init_kernel<LAT, IDX>, cudaFuncAttributeMaxDynamicSharedMemorySize, optin);
        if (e != cudaSuccess) return e;
    }
    init_kernel<LAT, IDX><<<a.nlines, 32, a.stage ? list : 0, s>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_init(int lattice, bool idx16, const InitArgs& a, cudaStream_t s)
{
    clear_stale_error();
    if (a.nlines < 1) return cudaSuccess;
    if (lattice == kSquare) return idx16 ? init_one<kSquare, uint16_t>(a, s) : init_one<kSquare, uint32_t>(a, s);
    if (lattice == kTriangular)
        return idx16 ? init_one<kTriangular, uint16_t>(a, s) : init_one<kTriangular, uint32_t>(a, s);
    if (lattice == kCubic) return idx16 ? init_one<kCubic, uint16_t>(a, s) : init_one<kCubic, uint32_t>(a, s);
    return idx16 ? init_one<kSquareOpen, uint16_t>(a, s) : init_one<kSquareOpen, uint32_t>(a, s);
}

// Line states of lines that are not walked: converged, with no move made.
__global__ void blank_states_kernel(LineState* st, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) st[i] = LineState{0, 0, 0, 0, 0, 0, 1, 0, 0};
}

cudaError_t launch_blank_states(LineState* st, int n, cudaStream_t s)
{
    clear_stale_error();
    blank_states_kernel<<<(n + 255) / 256, 256, 0, s>>>(st, n);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Assembly (Eq. 4 applied once, g_kl of Eq. 2): one warp per line,
//   ln g_kl = ln C(N,l) + u lng[b] - (M + ln sum_visited exp(u lng[b] - M)),
// M the visited maximum; unvisited bins get -inf.  FP64.
// ---------------------------------------------------------------------------
__global__ void assemble_kernel(const LineDesc* desc, const int32_t* order, const int64_t* lng, const hist_t* hist,
                                int N, int nlines, double u, double* out)
{
    const int warps = blockDim.x >> 5;
    const int x = blockIdx.x * warps + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (x >= nlines) return;
    const int li = order[x];
    const LineDesc D = desc[li];
    const int64_t* lg = lng + D.bin_off;
    const hist_t* h = hist + D.bin_off;
    double* o = out + D.bin_off;
    double mx = -DBL_MAX;
    for (int b = lane; b < D.nbins; b += 32)
        if (h[b] & kVisited) mx = fmax(mx, u * (double)lg[b]);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, off));
    double sum = 0.0;
    for (int b = lane; b < D.nbins; b += 32)
        if (h[b] & kVisited) sum += exp(u * (double)lg[b] - mx);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, off);
    const double lse = mx + log(sum);
    const double lnC = lgamma((double)N + 1.0) - lgamma((double)D.ell + 1.0) -
                       lgamma((double)(N - D.ell) + 1.0);
    for (int b = lane; b < D.nbins; b += 32)
        o[b] = (h[b] & kVisited) ? lnC + u * (double)lg[b] - lse : -INFINITY;
}

cudaError_t launch_assemble(const LineDesc* desc, const int32_t* order, const int64_t* lng, const hist_t* hist, int N,
                            int nlines, double u, double* out, cudaStream_t s)
{
    clear_stale_error();
    const int warps = 8;
    assemble_kernel<<<(nlines + warps - 1) / warps, 32 * warps, 0, s>>>(desc, order, lng, hist, N, nlines, u, out);
    return cudaGetLastError();
}

__global__ void fill_unvisited_kernel(double* out, size_t n)
{
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
        out[i] = -INFINITY;
}

cudaError_t launch_fill_unvisited(double* out, size_t n, cudaStream_t s)
{
    clear_stale_error();
    fill_unvisited_kernel<<<1216, 256, 0, s>>>(out, n);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Exp threshold table, built on the device: t[i] = floor(2^32 exp(-x_i) + 1/2),
// x_i = (i 2^q) u as one IEEE double product.  exp is evaluated in
// double-double arithmetic (Dekker's exact products and sums): x = n ln2 + r
// with ln 2 split in two doubles, exp(r / 2^10) by its Taylor series to degree
// 10, then ten squarings; relative error ~1e-28, far below the 2^-33
// granularity of the rounding.
// ---------------------------------------------------------------------------
struct dd {
    double hi, lo;
};

__device__ __forceinline__ dd dd_two_sum(double a, double b)
{
    const double s = __dadd_rn(a, b);
    const double bb = __dsub_rn(s, a);
    const double e = __dadd_rn(__dsub_rn(a, __dsub_rn(s, bb)), __dsub_rn(b, bb));
    return {s, e};
}

__device__ __forceinline__ dd dd_norm(double a, double b)
{
    const double s = __dadd_rn(a, b);
    return {s, __dsub_rn(b, __dsub_rn(s, a))};
}

__device__ __forceinline__ dd dd_add(dd a, dd b)
{
    dd s = dd_two_sum(a.hi, b.hi);
    const dd t = dd_two_sum(a.lo, b.lo);
    s.lo = __dadd_rn(s.lo, t.hi);
    s = dd_norm(s.hi, s.lo);
    s.lo = __dadd_rn(s.lo, t.lo);
    return dd_norm(s.hi, s.lo);
}

__device__ __forceinline__ dd dd_mul(dd a, dd b)
{
    const double p = __dmul_rn(a.hi, b.hi);
    double e = __fma_rn(a.hi, b.hi, -p);
    e = __fma_rn(a.hi, b.lo, e);
    e = __fma_rn(a.lo, b.hi, e);
    return dd_norm(p, e);
}

__device__ __forceinline__ dd dd_mul_d(dd a, double b)
{
    const double p = __dmul_rn(a.hi, b);
    const double e = __fma_rn(a.lo, b, __fma_rn(a.hi, b, -p));
    return dd_norm(p, e);
}

__device__ dd dd_exp_neg(double x)   // exp(-x) for 0 <= x < 40
{
    const dd ln2 = {0x1.62e42fefa39efp-1, 0x1.abc9e3b39803fp-56};
    const double n = rint(x / ln2.hi);
    // r = n ln2 - x  (exact enough: |r| <= 0.35)
    dd r = dd_mul_d(ln2, n);
    r = dd_add(r, {-x, 0.0});
    r.hi = ldexp(r.hi, -10);
    r.lo = ldexp(r.lo, -10);
    // Taylor series of exp(r) - 1, Horner form: r (1 + r/2 (1 + r/3 (...)))
    dd s = {1.0, 0.0};
    for (int k = 10; k >= 1; --k) {
        dd term = dd_mul(s, r);
        // divide by k: term / k in double-double via multiplication by 1/k corrections
        const double qh = __ddiv_rn(term.hi, (double)k);
        const double rem = __fma_rn(-qh, (double)k, term.hi);
        const double ql = __ddiv_rn(__dadd_rn(rem, term.lo), (double)k);
        s = dd_add({1.0, 0.0}, dd_norm(qh, ql));
    }
    // s = exp(r); square ten times
    for (int k = 0; k < 10; ++k) s = dd_mul(s, s);
    // times 2^-n
    s.hi = ldexp(s.hi, -(int)n);
    s.lo = ldexp(s.lo, -(int)n);
    return s;
}

__global__ void exp_table_kernel(double u, int q, uint64_t* out)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= kTableN) return;
    const double x = __dmul_rn((double)((uint64_t)i << q), u);
    dd e = dd_exp_neg(x);
    // v = 2^32 e + 1/2, floor(v) with v = hi + lo
    const double hi = ldexp(e.hi, 32), lo = ldexp(e.lo, 32);
    const double fh = floor(hi);
    const double frac = __dadd_rn(__dadd_rn(__dsub_rn(hi, fh), lo), 0.5);
    out[i] = (uint64_t)fh + (uint64_t)floor(frac);
}

cudaError_t launch_exp_table(double u, int q, uint64_t* out, cudaStream_t s)
{
    clear_stale_error();
    exp_table_kernel<<<(kTableN + 255) / 256, 256, 0, s>>>(u, q, out);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Philox check kernel: one block per counter.
// ---------------------------------------------------------------------------
__global__ void philox_kernel(size_t n, const uint32_t* ctr, const uint32_t* key, uint32_t* out)
{
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const uint4 c = make_uint4(ctr[4 * i], ctr[4 * i + 1], ctr[4 * i + 2], ctr[4 * i + 3]);
    const uint2 k = make_uint2(key[2 * i], key[2 * i + 1]);
    const uint4 r = philox4x32_10(c, k);
    out[4 * i] = r.x;
    out[4 * i + 1] = r.y;
    out[4 * i + 2] = r.z;
    out[4 * i + 3] = r.w;
}

cudaError_t launch_philox(size_t n, const uint32_t* ctr, const uint32_t* key, uint32_t* out,
                          cudaStream_t s)
{
    if (n == 0) return cudaSuccess;
    clear_stale_error();
    philox_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(n, ctr, key, out);
    return cudaGetLastError();
}

// dmax of Eq. 3 (the walker's acceptance threshold on d) for n random words.
__global__ void dmax_kernel(size_t n, const uint32_t* r, int det, const uint32_t* tab, int q,
                            float seg_per_log2, float inv_u, int64_t* out)
{
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    out[i] = det ? dmax_det(r[i], tab, q, seg_per_log2) : dmax_prod(r[i], inv_u);
}

cudaError_t launch_dmax(size_t n, const uint32_t* r, int det, const uint32_t* tab, int q,
                        float seg_per_log2, float inv_u, int64_t* out, cudaStream_t s)
{
    if (n == 0) return cudaSuccess;
    clear_stale_error();
    dmax_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(n, r, det, tab, q, seg_per_log2, inv_u, out);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Run summary after each walker launch: one block reduces the line states.
// ---------------------------------------------------------------------------
__global__ void summary_kernel(const LineState* st, int nlines, int64_t budget,
                               const int32_t* flags, Summary* out)
{
    __shared__ long long s_moves[32], s_acc[32], s_chk[32], s_bat[32];
    __shared__ int s_active[32], s_conv[32], s_ovf[32], s_min[32], s_max[32];
    long long moves = 0, acc = 0, chk = 0, bat = 0;
    int active = 0, conv = 0, ovf = 0, mn = INT_MAX, mx = 0;
    for (int i = threadIdx.x; i < nlines; i += blockDim.x) {
        const LineState s = st[i];
        moves += s.t;
        acc += s.accepts;
        chk += s.checks;
        bat += s.batches;
        active += (s.status == 0 && s.t < budget);
        conv += (s.status == 1);
        ovf += (s.status == 2);
        mn = (int)s.stage < mn ? (int)s.stage : mn;
        mx = (int)s.stage > mx ? (int)s.stage : mx;
    }
    for (int off = 16; off > 0; off >>= 1) {
        moves += __shfl_xor_sync(0xffffffffu, moves, off);
        acc += __shfl_xor_sync(0xffffffffu, acc, off);
        chk += __shfl_xor_sync(0xffffffffu, chk, off);
        bat += __shfl_xor_sync(0xffffffffu, bat, off);
        active += __shfl_xor_sync(0xffffffffu, active, off);
        conv += __shfl_xor_sync(0xffffffffu, conv, off);
        ovf += __shfl_xor_sync(0xffffffffu, ovf, off);
        mn = min(mn, __shfl_xor_sync(0xffffffffu, mn, off));
        mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, off));
    }
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (lane == 0) {
        s_moves[w] = moves;
        s_acc[w] = acc;
        s_chk[w] = chk;
        s_bat[w] = bat;
        s_active[w] = active;
        s_conv[w] = conv;
        s_ovf[w] = ovf;
        s_min[w] = mn;
        s_max[w] = mx;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        Summary r = {0, 0, 0, 0, 0, 0, 0, INT_MAX, 0, 0};
        for (int x = 0; x < (int)(blockDim.x >> 5); ++x) {
            r.moves += s_moves[x];
            r.accepts += s_acc[x];
            r.checks += s_chk[x];
            r.batches += s_bat[x];
            r.active += s_active[x];
            r.converged += s_conv[x];
            r.overflow += s_ovf[x];
            r.min_stage = min(r.min_stage, s_min[x]);
            r.max_stage = max(r.max_stage, s_max[x]);
        }
        r.flags = *flags;
        *out = r;
    }
}

cudaError_t launch_summary(const LineState* st, int nlines, int64_t budget, const int32_t* flags,
                           Summary* out, cudaStream_t s)
{
    clear_stale_error();
    summary_kernel<<<1, 1024, 0, s>>>(st, nlines, budget, flags, out);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Thermodynamics from the assembled surface (Eq. 2 with the energy of Eq. 1):
// Z = sum_{k,l} g_kl exp(-E_kl / T), E_kl = -(N_B - 2k) - H M, M = 2l - N; line l > N/2
// is line N - l.  FP64.
//
// The field term is the same for all of a line, so the sum over k is taken once per
// (T, line) and the fields are then a sum over lines: bins x nT exponentials and not
// 2 x bins x nT x nH, spread over (lines x nT) warps and not nT x nH blocks.  FP64 is
// slow on this GPU, and most bins of a line weigh nothing at a given T, so the line's
// maximum is found first and only bins within e^-46 of it (1e-20) take an exponential:
// a line of 4097 bins loses less than a rounding of its sum, and of its second moment
// less than 1e-20 (2 N_B)^2 a bin, 3e-12 at 64x64, where squares of energies that cancel
// lose more.  Moments are kept about the line's likeliest bin and then about the mean,
// where the variances of C and chi do not cancel.  32x32, 64 T x 3 H: 7.8 ms as one block per point with an exponential for
// every bin and mirror, 0.6 ms this way.
// ---------------------------------------------------------------------------
struct LineSum {
    double mx;             // max over visited bins of ln g - E / T at H = 0 (-inf: none)
    double s0, s1, s2;     // sums of w, w c, w c^2: w = exp(. - mx), c = bond energy - ref
    double ref;            // bond energy of the bin at the maximum
};

__device__ __forceinline__ double warp_sum(double v)
{
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    return v;
}

constexpr double kNegligible = 46.0;

__global__ void thermo_lines_kernel(const LineDesc* desc, int nlines, const double* lng, int NB, int kstep, const double* T,
                                    LineSum* out)
{
    const int li = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (li >= nlines) return;
    const LineDesc D = desc[li];
    const double* g = lng + D.bin_off;
    const double beta = 1.0 / T[blockIdx.y];
    // bond energy of bin b: -(N_B - 2 k), k = kstep b
    auto bond = [&](int b) { return (double)(2 * kstep * b - NB); };
    double mx = -INFINITY;
    int at = 0;
#pragma unroll 4
    for (int b = lane; b < D.nbins; b += 32) {
        const double x = g[b] - beta * bond(b);
        if (x > mx) {
            mx = x;
            at = b;
        }
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        const double m2 = __shfl_xor_sync(0xffffffffu, mx, off);
        const int a2 = __shfl_xor_sync(0xffffffffu, at, off);
        if (m2 > mx || (m2 == mx && a2 < at)) {
            mx = m2;
            at = a2;
        }
    }
    const double ref = bond(at);
    double s0 = 0.0, s1 = 0.0, s2 = 0.0;
#pragma unroll 4
    for (int b = lane; b < D.nbins; b += 32) {
        const double x = g[b] - beta * bond(b) - mx;
        if (x > -kNegligible) {
            const double w = exp(x), c = bond(b) - ref;
            s0 += w;
            s1 += w * c;
            s2 += w * c * c;
        }
    }
    s0 = warp_sum(s0);
    s1 = warp_sum(s1);
    s2 = warp_sum(s2);
    if (lane == 0) out[(size_t)blockIdx.y * nlines + li] = LineSum{mx, s0, s1, s2, ref};
}

// Sums over the block, the same in every thread (blocks of 256).
template <int n>
__device__ __forceinline__ void block_sums(double (&v)[n])
{
    __shared__ double part[8][n];
    __syncthreads();
#pragma unroll
    for (int q = 0; q < n; ++q) {
        v[q] = warp_sum(v[q]);
        if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5][q] = v[q];
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < n; ++q) {
        v[q] = 0.0;
        for (int w = 0; w < 8; ++w) v[q] += part[w][q];
    }
}

// One block per (T, H): the lines' sums with the field's weight, both l and N - l.
__global__ void __launch_bounds__(256) thermo_points_kernel(const LineDesc* desc, int nlines, const LineSum* sums, int N,
                                                            const double* T, const double* H, int nH, double* out)
{
    const int pt = blockIdx.x;
    const double beta = 1.0 / T[pt / nH], h = H[pt % nH];
    const LineSum* S = sums + (size_t)(pt / nH) * nlines;
    __shared__ double s_mx[8];
    double mx = -INFINITY;
    for (int i = threadIdx.x; i < nlines; i += 256) {
        const double M = (double)(2 * desc[i].ell - N);
        mx = fmax(mx, S[i].mx + fabs(beta * h * M));       // of the line and its mirror
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, off));
    if ((threadIdx.x & 31) == 0) s_mx[threadIdx.x >> 5] = mx;
    __syncthreads();
    for (int w = 0; w < 8; ++w) mx = fmax(mx, s_mx[w]);
    // for each line (and its mirror): weight, energies about `e`, magnetisation about `m`
    auto over_lines = [&](auto&& add) {
        for (int i = threadIdx.x; i < nlines; i += 256) {
            const LineSum s = S[i];
            if (s.mx == -INFINITY) continue;
            const int l = desc[i].ell;
            const double M = (double)(2 * l - N);
            add(s, M, exp(s.mx + beta * h * M - mx));
            if (N - l != l) add(s, -M, exp(s.mx - beta * h * M - mx));
        }
    };
    double a[4] = {0.0, 0.0, 0.0, 0.0};
    over_lines([&](const LineSum& s, double M, double w) {
        a[0] += w * s.s0;
        a[1] += w * (s.s1 + (s.ref - h * M) * s.s0);
        a[2] += w * s.s0 * M;
        a[3] += w * s.s0 * fabs(M);
    });
    block_sums(a);
    const double z = a[0], e = a[1] / z, m = a[2] / z;
    double v[2] = {0.0, 0.0};
    over_lines([&](const LineSum& s, double M, double w) {
        const double d = s.ref - h * M - e;
        v[0] += w * (s.s2 + 2.0 * d * s.s1 + d * d * s.s0);
        v[1] += w * s.s0 * (M - m) * (M - m);
    });
    block_sums(v);
    if (threadIdx.x == 0) {
        double* o = out + (size_t)pt * 6;
        o[0] = (mx + log(z)) / N;
        o[1] = e / N;
        o[2] = v[0] / z * beta * beta / N;
        o[3] = m / N;
        o[4] = a[3] / z / N;
        o[5] = v[1] / z * beta / N;
    }
}

size_t thermo_scratch_bytes(int nlines, int nT)
{
    // temperatures are taken in groups whose line sums fit 2 MB (one at least): a group of
    // a large surface has work for all SMs all the same
    const size_t one = (size_t)nlines * sizeof(LineSum);
    return one * std::min<size_t>((size_t)nT, std::max<size_t>(1, ((size_t)2 << 20) / one));
}

cudaError_t launch_thermo(const LineDesc* desc, int nlines, const double* lng, int N, int NB,
                          int kstep, const double* T, int nT, const double* H, int nH, double* out,
                          void* scratch, cudaStream_t s)
{
    if (nT * nH == 0) return cudaSuccess;
    clear_stale_error();
    LineSum* sums = static_cast<LineSum*>(scratch);
    const int group = (int)std::min<size_t>(thermo_scratch_bytes(nlines, nT) / ((size_t)nlines * sizeof(LineSum)), 32768);
    for (int t = 0; t < nT; t += group) {
        const int n = std::min(group, nT - t);
        thermo_lines_kernel<<<dim3((nlines + 3) / 4, n), 128, 0, s>>>(desc, nlines, lng, NB, kstep, T + t, sums);
        thermo_points_kernel<<<n * nH, 256, 0, s>>>(desc, nlines, sums, N, T + t, H, nH, out + (size_t)t * nH * 6);
    }
    return cudaGetLastError();
}

__global__ void deadline_kernel(uint64_t* deadline, uint64_t timeout_ns)
{
    *deadline = timeout_ns ? globaltimer_ns() + timeout_ns : 0ull;
}

cudaError_t launch_set_deadline(uint64_t* deadline, uint64_t timeout_ns, cudaStream_t s)
{
    clear_stale_error();
    deadline_kernel<<<1, 1, 0, s>>>(deadline, timeout_ns);
    return cudaGetLastError();
}

__global__ void begin_slice_kernel(uint64_t* slice_end, uint64_t slice_ns, int32_t* first, int walkers, int nqueue)
{
    *slice_end = globaltimer_ns() + slice_ns;
    const int at = first[1];
    first[0] = at;
    first[1] = (at + walkers) % nqueue;
}

cudaError_t launch_begin_slice(uint64_t* slice_end, uint64_t slice_ns, int32_t* first, int walkers, int nqueue,
                               cudaStream_t s)
{
    clear_stale_error();
    begin_slice_kernel<<<1, 1, 0, s>>>(slice_end, slice_ns, first, walkers, nqueue);
    return cudaGetLastError();
}

cudaError_t launch_walk(int lattice, int S, bool det, bool idx16, dim3 grid, dim3 block,
                        size_t smem, cudaStream_t s, const WalkArgs& a)
{
    if (a.lone) return idx16 ? launch_lone(det, grid, block, smem, s, a, nullptr) : cudaErrorInvalidValue;
    if (lattice == kSquare) return launch_walk_square(S, det, idx16, grid, block, smem, s, a, nullptr);
    if (lattice == kSquareP2)
        return launch_walk_square_p2(S, det, idx16, grid, block, smem, s, a, nullptr);
    if (lattice == kTriangular)
        return launch_walk_triangular(S, det, idx16, grid, block, smem, s, a, nullptr);
    if (lattice == kSquareOpen)
        return launch_walk_square_open(S, det, idx16, grid, block, smem, s, a, nullptr);
    return launch_walk_cubic(S, det, idx16, grid, block, smem, s, a, nullptr);
}

cudaError_t walk_kernel_attrs(int lattice, int S, bool det, bool idx16, size_t smem, int block_threads,
                              const WalkArgs& a, int* blocks_per_sm)
{
    const dim3 z(0), b(block_threads);
    if (a.lone) return idx16 ? launch_lone(det, z, b, smem, 0, a, blocks_per_sm) : cudaErrorInvalidValue;
    if (lattice == kSquare) return launch_walk_square(S, det, idx16, z, b, smem, 0, a, blocks_per_sm);
    if (lattice == kSquareP2)
        return launch_walk_square_p2(S, det, idx16, z, b, smem, 0, a, blocks_per_sm);
    if (lattice == kTriangular)
        return launch_walk_triangular(S, det, idx16, z, b, smem, 0, a, blocks_per_sm);
    if (lattice == kSquareOpen)
        return launch_walk_square_open(S, det, idx16, z, b, smem, 0, a, blocks_per_sm);
    return launch_walk_cubic(S, det, idx16, z, b, smem, 0, a, blocks_per_sm);
}

}  // namespace wl
