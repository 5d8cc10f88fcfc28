// wl_walk.cuh -- the Wang-Landau walker kernel for micromagnetic lines
// (arXiv:1302.2320, the procedure around Eq. 3 and Eq. 4).
//
// One walker = one line l = S consecutive lanes of a warp ("group").  A batch
// covers the steps t .. t+S-1:
//   draw -- lane m holds the random numbers of step t+m, drawn one batch
//     ahead: the list slots a, b and dmax, the largest ln g increase that
//     Eq. 3 accepts with this step's random word (see dmax_det / dmax_prod);
//   propose -- lane m evaluates its exchange against the state at the start of
//     the batch: sites i = U[a], j = D[b] and the change of k, and collects the
//     earlier proposals that could change either (below);
//   chain -- the group's first lane alone takes the steps in order: one load of
//     ln g at the target bin, one 64-bit compare, one store of ln g at the bin
//     the step ends in.
// The chain is the serial part of the method.  It costs ~18 instructions a step
// whether the step is accepted or not, all its operands but the target's ln g
// are known before it starts, and its critical path is one shared-memory load,
// the compare and a select.
//
// What an accepted exchange of (i_e, j_e) does to a later proposal: if that one
// uses the same list slot (equivalently: names site i_e or j_e, the lists
// holding distinct sites) its sites are no longer U[a], D[b]; if i_e or j_e
// neighbours its sites, its change of k is another.  Every site has a byte that
// names the lane proposing it (its "owner"; of several lanes proposing one site
// the last to write), so a proposal learns the owners of its sites and their
// neighbours from the same bytes that hold their spins.  The chain keeps the
// set of owners whose site an accepted step has moved; a step that sees one of
// them stops the chain, the accepted exchanges are applied, the group evaluates
// that one step again from the lists and spins as they now are, and the chain
// goes on.  A step whose evaluation is out of date is always seen: its sites
// and their neighbours at the start of the batch include every site through
// which an earlier step can have reached it, also when a re-evaluated step took
// a site that entered its slot within the batch (that site was itself proposed
// in the batch, so it has an owner).
// Random numbers are keyed by t, so the committed chain is the sequential
// chain, bit for bit, for every S and both forms.  Batches never cross a
// flatness check (t multiple of C) or the end of the slice.
//
// ln g of the bins around the walker lives in a shared-memory window, written
// back when the walker nears an edge of it, at every check and at the end.  A
// visit adds F to a bin's ln g and 1 to its count, so the counts are not kept
// while walking: storing the window recovers them as (ln g - ln g before) / F.
//
// Lattices too large for a block per line walk in this form (plan_shape), and "tail" = 0,
// other lane counts than 32 and one launch per line.  A line of many up spins takes
// 160 cycles a move alone (256x256, where resolving the accepted steps with all lanes
// took 500), 17 a move and SM when there are enough lines to fill it; a line of few up
// spins, whose batches keep running into themselves, up to 1000.
#pragma once

#include "wl_device.cuh"

namespace wl {

template <int S>
__device__ __forceinline__ unsigned group_mask(int gbase)
{
    if constexpr (S == 32) return 0xffffffffu;
    else return ((1u << S) - 1u) << gbase;
}

// The predicate of each lane of the group as bits 0 .. S-1.
template <int S>
__device__ __forceinline__ unsigned group_ballot(unsigned gmask, int gbase, bool p)
{
    const unsigned b = __ballot_sync(gmask, p);
    if constexpr (S == 32) return b;
    else return (b >> gbase) & ((1u << S) - 1u);
}

// Flatness (80%/80% convention, fraction x = flat_pm/1000, exact integers):
// n visited bins, Ssum = their histogram total, c = bins with
// 1000*n*h >= flat_pm*Ssum; flat iff 1000*c >= flat_pm*n.
// Both passes issue kFlatUnroll independent loads per lane: the histogram lies in
// L2, and one load at a time makes a check cost its latency times bins / S.
constexpr int kFlatUnroll = 8;

template <int S>
__device__ bool group_flat(const hist_t* hist, int nbins, int m, unsigned gmask, int flat_pm)
{
    int64_t n = 0;
    uint64_t ssum = 0;
    for (int b0 = m; b0 < nbins; b0 += S * kFlatUnroll) {
        hist_t h[kFlatUnroll];
#pragma unroll
        for (int q = 0; q < kFlatUnroll; ++q) h[q] = b0 + q * S < nbins ? hist[b0 + q * S] : 0ull;
#pragma unroll
        for (int q = 0; q < kFlatUnroll; ++q)
            if (h[q] & kVisited) {
                n += 1;
                ssum += h[q] & ~kVisited;
            }
    }
    n = group_sum<S>(gmask, n);
    ssum = group_sum<S>(gmask, ssum);
    if (n == 0) return false;
    int64_t c = 0;
    // products of up to ~2^77: compared in 128-bit integers
    const unsigned __int128 rhs = (unsigned __int128)flat_pm * ssum;
    const unsigned __int128 scale = (unsigned __int128)(1000 * n);
    for (int b0 = m; b0 < nbins; b0 += S * kFlatUnroll) {
        hist_t h[kFlatUnroll];
#pragma unroll
        for (int q = 0; q < kFlatUnroll; ++q) h[q] = b0 + q * S < nbins ? hist[b0 + q * S] : 0ull;
#pragma unroll
        for (int q = 0; q < kFlatUnroll; ++q)
            if ((h[q] & kVisited) && scale * (h[q] & ~kVisited) >= rhs) c += 1;
    }
    c = group_sum<S>(gmask, c);
    return 1000 * c >= (int64_t)flat_pm * n;
}

// Stage step after a flat histogram: the constant shift that puts the visited
// minimum of ln g at zero stands in for the normalisation of Eq. 4 (Eq. 4 is
// applied exactly at assembly); the histogram is reset, visited bits kept.
template <int S>
__device__ void group_stage_step(int64_t* lng, hist_t* hist, int nbins, int m, unsigned gmask)
{
    int64_t mn = INT64_MAX;
    for (int b = m; b < nbins; b += S)
        if (hist[b] & kVisited) mn = lng[b] < mn ? lng[b] : mn;
    mn = group_min<S>(gmask, mn);
    for (int b = m; b < nbins; b += S) {
        const hist_t h = hist[b];
        if (h & kVisited) lng[b] -= mn;
        hist[b] = h & kVisited;
    }
    __syncwarp(gmask);
}

// Visits behind an increase d of a bin's ln g: d / F, exact.  Every round takes a
// quotient estimated from below to one part in 2^18, so counts below 2^18 need
// two at most (the float helpers keep the FP64 pipe out of it).
__device__ __forceinline__ uint64_t visits_of(int64_t d, int64_t F, float inv_f)
{
    uint64_t rem = (uint64_t)d, n = 0;
    while (rem >= (uint64_t)F) {
        uint64_t e = (uint64_t)float_floor_i64(u64_to_float_rz(rem) * inv_f);
        e = e ? e : 1;
        n += e;
        rem -= e * (uint64_t)F;
    }
    return n;
}

// 1 / F rounded so that the estimates of visits_of never exceed the quotient.
__device__ __forceinline__ float inverse_below(int64_t F)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(u64_to_float_rz((uint64_t)F)));
    return r * (1.0f - 0x1p-18f);
}

// Store the window [wb, wb + wn) of ln g; the visits made since it was loaded
// are added to the histogram and mark their bins visited.  Counts reaching 2^62
// (far beyond any run) are reported as an overflow.
template <int S>
__device__ __forceinline__ bool window_store(const int64_t* wl, int64_t* lng, hist_t* hist, int wb,
                                             int wn, int m, int64_t F)
{
    constexpr int U = 4;      // independent loads per lane and round
    bool ovf = false;
    const float inv_f = inverse_below(F);
    for (int x0 = m; x0 < wn; x0 += U * S) {
        int64_t d[U];
        hist_t h[U];
#pragma unroll
        for (int q = 0; q < U; ++q) {
            const int x = x0 + q * S;
            d[q] = x < wn ? wl[x] - lng[wb + x] : 0;
            h[q] = x < wn ? hist[wb + x] : 0ull;
        }
#pragma unroll
        for (int q = 0; q < U; ++q) {
            const int x = x0 + q * S;
            if (d[q]) {
                h[q] += visits_of(d[q], F, inv_f);
                ovf |= (h[q] & ~kVisited) >= (1ull << 62);
                hist[wb + x] = h[q] | kVisited;
                lng[wb + x] = wl[x];
            }
        }
    }
    return ovf;
}

template <int S>
__device__ __forceinline__ void window_load(int64_t* wl, const int64_t* lng, int wb, int wn, int m)
{
#pragma unroll 4
    for (int x = m; x < wn; x += S) wl[x] = lng[wb + x];
}

__device__ __forceinline__ int window_base(int bc, int nbins, int win)
{
    int wb = bc - win / 2;
    if (wb > nbins - win) wb = nbins - win;
    return wb < 0 ? 0 : wb;
}

template <bool DET>
__device__ __forceinline__ Draw draw_step(uint64_t t, uint2 key, uint32_t ell, uint32_t nd,
                                          const WalkArgs& A)
{
    const uint4 r = philox4x32_10(make_uint4((uint32_t)t, (uint32_t)(t >> 32), 0u, 0u), key);
    Draw d;
    d.a = pick(r.x, ell);
    d.b = pick(r.y, nd);
    d.dmax = DET ? dmax_det(r.z, A.table, A.q, A.seg_per_log2) : dmax_prod(r.z, A.inv_u);
    return d;
}

// The spins and the owners of the sites proposed in the current batch.
// BYTES: one byte per site in shared memory, the spin at the start of the batch
// in bit 7 and the owner's lane in bits 0..6 (kNoOwner: none), so that one load
// answers both questions.
// Otherwise (a lattice larger than shared memory): packed spins in global memory
// and owners in a shared table indexed by the low bits of the site; sites that
// share an entry share an owner, which can only add evaluations.
constexpr uint32_t kNoOwner = 0x40u;

template <bool BYTES>
struct Sites {
    uint8_t* own;      // BYTES: N bytes; otherwise mask + 1 owners
    uint32_t* sp;      // packed spins (not BYTES)
    uint32_t mask;
    __device__ __forceinline__ uint32_t peek(uint32_t n) const
    {
        if constexpr (BYTES) return own[n];
        else return own[n & mask] | (spin_at(sp, n) << 7);
    }
    __device__ __forceinline__ void mark(uint32_t n, uint32_t spin, uint32_t lane) const
    {
        if constexpr (BYTES) own[n] = (uint8_t)((spin << 7) | lane);
        else own[n & mask] = (uint8_t)lane;
    }
    // no owner, and (BYTES) the spin
    __device__ __forceinline__ void clear(uint32_t n, uint32_t spin) const
    {
        if constexpr (BYTES) own[n] = (uint8_t)((spin << 7) | kNoOwner);
        else own[n & mask] = (uint8_t)kNoOwner;
    }
};

// 1 << owner of a site byte, 0 for kNoOwner (a PTX shift by 32 or more gives 0).
__device__ __forceinline__ uint32_t owner_bit(uint32_t v)
{
    uint32_t r;
    asm("shl.b32 %0, 1, %1;" : "=r"(r) : "r"(v & 0x7Fu));
    return r;
}

// Owners next to the two sites of a proposal: of up and of down neighbours of i
// and of j (the up ones own a site that an accepted step turns down, and so on).
struct Near {
    uint32_t iu, id, ju, jd;
};

// The sites of the batch that have turned since its start, by owner: up sites
// turned down, down sites turned up.  Every owner owns one site of each kind.
struct Turned {
    uint32_t up, down;
};

// The change of k when i (up) and j (down) exchange.  NEAR: with the spins as the
// bytes hold them, and the owners around; otherwise (BYTES) with the spins as
// they are after `turned`.
template <int LAT, bool BYTES, bool NEAR>
__device__ __forceinline__ int exchange_dk(const Geo& g, const Sites<BYTES>& st, uint32_t i, uint32_t j,
                                           const Turned& turned, Near* near)
{
    constexpr int z = Coord<LAT>::z;
    uint32_t ni[z], nj[z];
    unsigned vi = (1u << z) - 1u, vj = vi;
    if constexpr (LAT == kSquareOpen) {
        vi = open_neighbours(g, i, ni);
        vj = open_neighbours(g, j, nj);
    } else {
        neighbours<LAT>(g, i, ni);
        neighbours<LAT>(g, j, nj);
    }
    int ui = 0, uj = 0, a = 0;
    Near o{0u, 0u, 0u, 0u};
#pragma unroll
    for (int q = 0; q < z; ++q) {
        const uint32_t pi = st.peek(ni[q]), pj = st.peek(nj[q]);
        int si = (int)(pi >> 7), sj = (int)(pj >> 7);
        const uint32_t oi = owner_bit(pi), oj = owner_bit(pj);
        if constexpr (BYTES && !NEAR) {
            si ^= (oi & (si ? turned.up : turned.down)) != 0u;
            sj ^= (oj & (sj ? turned.up : turned.down)) != 0u;
        }
        bool adj = ni[q] == j;
        if constexpr (LAT == kSquareOpen) {
            if (!((vi >> q) & 1u)) si = 0, adj = false;
            if (!((vj >> q) & 1u)) sj = 0;
        }
        ui += si;
        uj += sj;
        a += adj;
        if constexpr (NEAR) {
            const bool hi = LAT != kSquareOpen || ((vi >> q) & 1u), hj = LAT != kSquareOpen || ((vj >> q) & 1u);
            const uint32_t mi = hi ? oi : 0u, mj = hj ? oj : 0u;
            const uint32_t fi = 0u - (pi >> 7), fj = 0u - (pj >> 7);
            o.iu |= mi & fi;
            o.id |= mi & ~fi;
            o.ju |= mj & fj;
            o.jd |= mj & ~fj;
        }
    }
    if constexpr (NEAR) *near = o;
    int dk = 2 * (ui - uj + a);
    // with site degrees z_i, z_j: dk = 2 (u_i - u_j + a_ij) - z_i + z_j
    if constexpr (LAT == kSquareOpen) dk += __popc(vj) - __popc(vi);
    return dk;
}

// What the chain needs of the steps of a batch, in shared memory:
//   a {dmax (two words), the owners whose move makes the step out of date, its
//     bin step in bytes of the window}
//   b {the owner of its up site, of its down site, as bits}
//   c the owners around (Near), read when the step is out of date
template <int S>
struct Steps {
    uint4 a[S];
    uint4 c[S];
    uint2 b[S];
};

// State of the chain (held by the group's first lane while it runs).
struct Chain {
    uint32_t xa;     // shared address of the current bin in the window
    int64_t u;       // its ln g
    uint32_t moved;  // owners with a site that an accepted step has moved
    Turned turned;
    uint32_t accm;   // accepted steps of the batch
    int s;           // steps taken
};

// K steps of the chain from step c.s on, or up to the first that is out of date.
// Written in PTX for the predication: the compiler turns the updates of an
// accepted step into selects and every exit into a divergent branch with its
// own reconvergence, ~30 instructions a step against 20 here.  The serial path
// of a step is: target address, load, compare, select.  The load is issued before
// the out-of-date test; its address is then wrong by a few bins at most, inside
// the slot's guard.  The window always holds every visit, so a step with no
// change of bin needs no case of its own: it reads ln g of its own bin and is
// accepted, dmax being >= 0.
#define WL_REC(q, oa, ob)                                         \
    "ld.shared.v4.u32 {l" #q ", h" #q ", z" #q ", k" #q "}, [%7+" #oa "];\n\t" \
    "ld.shared.v2.u32 {i" #q ", j" #q "}, [%8+" #ob "];\n\t"
#define WL_STEP(q, bit, next, bra)                                \
    "add.u32 ta, %0, k" #q ";\n\t"                                \
    "ld.shared.s64 g, [ta];\n\t"                                  \
    next                                                          \
    "and.b32 t, z" #q ", %2;\n\t"                                 \
    "setp.ne.u32 p, t, 0;\n\t"                                    \
    "@p " bra " X" #q ";\n\t"                                     \
    "mov.b64 d, {l" #q ", h" #q "};\n\t"                          \
    "add.s64 d, d, %1;\n\t"                                       \
    "add.s64 %1, %1, %9;\n\t"                                     \
    "setp.le.s64 p, g, d;\n\t"                                    \
    "add.s64 g, g, %9;\n\t"                                       \
    "@p mov.u32 %0, ta;\n\t"                                      \
    "@p mov.b64 %1, g;\n\t"                                       \
    "st.shared.s64 [%0], %1;\n\t"                                 \
    "@p lop3.b32 %2, %2, i" #q ", j" #q ", 0xFE;\n\t"             \
    "@p xor.b32 %3, %3, i" #q ";\n\t"                             \
    "@p xor.b32 %4, %4, j" #q ";\n\t"                             \
    "@p or.b32 %5, %5, " #bit ";\n\t"
#define WL_REGS(q) ".reg .b32 l" #q ", h" #q ", z" #q ", k" #q ", i" #q ", j" #q ";\n\t"
#define WL_EXIT(q) "X" #q ": mov.u32 %6, " #q ";\n\t bra DONE;\n\t"
#define WL_CHAIN_OPERANDS                                                                   \
    : "+r"(c.xa), "+l"(c.u), "+r"(c.moved), "+r"(c.turned.up), "+r"(c.turned.down), "+r"(acc), "=r"(n) \
    : "r"(ra), "r"(rb), "l"(F) : "memory"

#define WL_CHAIN_8(bra)                                                                     \
    WL_REGS(0) WL_REGS(1) WL_REGS(2) WL_REGS(3) WL_REGS(4) WL_REGS(5) WL_REGS(6) WL_REGS(7) \
    WL_REC(0, 0, 0) WL_REC(1, 16, 8)                                                        \
    WL_STEP(0, 1, WL_REC(2, 32, 16), bra) WL_STEP(1, 2, WL_REC(3, 48, 24), bra)             \
    WL_STEP(2, 4, WL_REC(4, 64, 32), bra) WL_STEP(3, 8, WL_REC(5, 80, 40), bra)             \
    WL_STEP(4, 16, WL_REC(6, 96, 48), bra) WL_STEP(5, 32, WL_REC(7, 112, 56), bra)          \
    WL_STEP(6, 64, "", bra) WL_STEP(7, 128, "", bra)                                        \
    "mov.u32 %6, 8;\n\tbra DONE;\n\t"                                                      \
    WL_EXIT(0) WL_EXIT(1) WL_EXIT(2) WL_EXIT(3) WL_EXIT(4) WL_EXIT(5) WL_EXIT(6) WL_EXIT(7)
#define WL_CHAIN_4(bra)                                                                     \
    WL_REGS(0) WL_REGS(1) WL_REGS(2) WL_REGS(3)                                             \
    WL_REC(0, 0, 0) WL_REC(1, 16, 8)                                                        \
    WL_STEP(0, 1, WL_REC(2, 32, 16), bra) WL_STEP(1, 2, WL_REC(3, 48, 24), bra)             \
    WL_STEP(2, 4, "", bra) WL_STEP(3, 8, "", bra)                                           \
    "mov.u32 %6, 4;\n\tbra DONE;\n\t"                                                      \
    WL_EXIT(0) WL_EXIT(1) WL_EXIT(2) WL_EXIT(3)
#define WL_CHAIN_1(bra)                                                                     \
    WL_REGS(0) WL_REC(0, 0, 0) WL_STEP(0, 1, "", bra)                                       \
    "mov.u32 %6, 1;\n\tbra DONE;\n\t" WL_EXIT(0)
#define WL_CHAIN(steps)                                                                     \
    asm volatile("{\n\t.reg .pred p;\n\t.reg .b32 ta, t;\n\t.reg .b64 g, d;\n\t"         \
                 steps "DONE:\n\t}" WL_CHAIN_OPERANDS)

// ALONE: the only chain of its warp, whose exits are uniform (128x128, 32 lanes a
// walker: 21.7 ms against 22.9 without the promise).  Leaders of several groups run
// theirs together and leave them at different steps: theirs are not.
template <int K, bool ALONE>
__device__ __forceinline__ int chain_steps(Chain& c, uint32_t ra, uint32_t rb, int64_t F)
{
    static_assert(K == 8 || K == 4 || K == 1, "chain_steps");
    uint32_t n, acc = 0u;
    ra += 16u * (uint32_t)c.s;
    rb += 8u * (uint32_t)c.s;
    if constexpr (K == 8) {
        if constexpr (ALONE) WL_CHAIN(WL_CHAIN_8("bra.uni"));
        else WL_CHAIN(WL_CHAIN_8("bra"));
    } else if constexpr (K == 4) {
        if constexpr (ALONE) WL_CHAIN(WL_CHAIN_4("bra.uni"));
        else WL_CHAIN(WL_CHAIN_4("bra"));
    } else {
        if constexpr (ALONE) WL_CHAIN(WL_CHAIN_1("bra.uni"));
        else WL_CHAIN(WL_CHAIN_1("bra"));
    }
    c.accm |= acc << c.s;
    c.s += (int)n;
    return (int)n;
}

// Take steps c.s .. lim-1; 0: all taken, 1: step c.s has to be evaluated again
// by the group, 2: the walker is near an edge of its window (tested every kSub
// steps; lo and hi leave the margin that kSub steps can use up).
// An out-of-date step whose own sites are where they were only has another
// change of k, by the sites around it that have turned: that is a count of owner
// bits (BYTES: owners are exact), and the step is taken here.
constexpr int kSub = 8;

template <int S, int KS, bool BYTES>
__device__ __forceinline__ int run_chain(Chain& c, Steps<S>* steps, int lim, int64_t F, uint32_t lo, uint32_t hi)
{
    const uint32_t ra = (uint32_t)__cvta_generic_to_shared(steps->a);
    const uint32_t rb = (uint32_t)__cvta_generic_to_shared(steps->b);
    while (c.s < lim) {
        if (c.xa < lo || c.xa > hi) return 2;
        const int left = lim - c.s;
        bool fresh;
        if (S >= 8 && left >= 8) fresh = chain_steps<8, S == 32>(c, ra, rb, F) == 8;
        else if (S >= 4 && left >= 4) fresh = chain_steps<4, S == 32>(c, ra, rb, F) == 4;
        else fresh = chain_steps<1, S == 32>(c, ra, rb, F) == 1;
        if (fresh) continue;
        if constexpr (!BYTES) {
            return 1;
        } else {
            const uint2 b = steps->b[c.s];
            if ((b.x | b.y) & c.moved) return 1;
            const uint4 o = steps->c[c.s];
            const int d = __popc(o.z & c.turned.up) - __popc(o.x & c.turned.up) + __popc(o.y & c.turned.down) -
                          __popc(o.w & c.turned.down);
            steps->a[c.s].z = 0u;
            steps->a[c.s].w += (uint32_t)(d * (16 >> KS));
        }
    }
    return 0;
}

// Walk line `li` for up to A.slice_moves moves (or to its budget, or to
// convergence).  perm points at the line's list (shared or global memory), st at
// its spins; wl is the group's window, steps its step records (shared memory).
// All lanes of the group hold identical copies of the scalar state.
template <int LAT, int S, bool DET, typename IDX, bool BYTES>
__device__ void walk_line(const WalkArgs& A, int li, int m, int gbase, unsigned gmask, IDX* perm,
                          const Sites<BYTES>& st, int64_t* wl, Steps<S>* steps)
{
    constexpr int zb = Coord<LAT>::zbin;  // largest bin step of one move
    constexpr int ks = Coord<LAT>::kshift;
    constexpr int kMargin = kSub * (zb + 1);
    const LineDesc D = A.desc[li];
    LineState* P = A.st + li;
    int64_t t = P->t, F = P->F, stage = P->stage, accepts = P->accepts;
    int64_t t_stage = P->t_stage, status = P->status, checks = P->checks;
    int64_t batches = P->batches;
    int k = (int)P->k;
    if (status != 0) return;
    const int ell = D.ell, nbins = D.nbins;
    const uint32_t nd = (uint32_t)(A.g.N - ell);
    int64_t* lng = A.lng + D.bin_off;
    hist_t* hist = A.hist + D.bin_off;
    const uint2 key = make_uint2((uint32_t)ell, A.seed);
    int64_t end = t + A.slice_moves;
    if (end > A.budget) end = A.budget;
    // flatness check interval of this line: longer for lines with more bins
    const int64_t C = A.C_per_bin > 0 && A.C_per_bin * nbins > A.C ? A.C_per_bin * nbins : A.C;

    int stop = 0;
    int bc = k >> ks;
    if (bc < 0 || bc >= nbins) {
        stop = 4;                 // not a state of this line
        bc = 0;
        end = t;
    }
    const int wn = nbins < A.win_bins ? nbins : A.win_bins;
    int wb = window_base(bc, nbins, A.win_bins);
    window_load<S>(wl, lng, wb, wn, m);
    __syncwarp(gmask);
    const uint32_t wa = (uint32_t)__cvta_generic_to_shared(wl);
    Chain c{};
    c.xa = wa + 8u * (uint32_t)(bc - wb);
    c.u = wl[bc - wb];

    Draw d = draw_step<DET>((uint64_t)(t + m), key, (uint32_t)ell, nd, A);

    while (t < end && !stop) {
        const int64_t next_check = (t / C + 1) * C;
        const int64_t seg_end = next_check < end ? next_check : end;
        int64_t left = seg_end - t;       // moves before the next check or the slice end

        while (left > 0) {
            const int lim = left < S ? (int)left : S;
            // -- propose: step t + m against the state at the start of the batch
            const uint32_t i0 = (uint32_t)perm[d.a];
            const uint32_t j0 = (uint32_t)perm[ell + d.b];
            st.mark(i0, 1u, (uint32_t)m);
            st.mark(j0, 0u, (uint32_t)m);
            // the next batch's draw (independent of this batch: it hides the latencies here)
            const Draw dn = draw_step<DET>((uint64_t)(t + S + m), key, (uint32_t)ell, nd, A);
            __syncwarp(gmask);
            Near near;
            int dk = exchange_dk<LAT, BYTES, true>(A.g, st, i0, j0, Turned{0u, 0u}, &near);
            const uint32_t oi = owner_bit(st.peek(i0)), oj = owner_bit(st.peek(j0));
            steps->a[m] = make_uint4((uint32_t)d.dmax, (uint32_t)((uint64_t)d.dmax >> 32),
                                     (near.iu | near.id | near.ju) | (near.jd | oi | oj), (uint32_t)((dk >> ks) * 8));
            steps->b[m] = make_uint2(oi, oj);
            if constexpr (BYTES) steps->c[m] = make_uint4(near.iu, near.id, near.ju, near.jd);
            __syncwarp(gmask);
            if constexpr (!BYTES) {
                st.clear(i0, 1u);
                st.clear(j0, 0u);
            }
            uint32_t i = i0, j = j0;      // the sites the step exchanges, once it is taken
            // -- the chain, with out-of-date steps evaluated again as they come up
            const uint32_t lo = wb > 0 ? wa + 8u * kMargin : wa;
            const uint32_t hi = wb + wn < nbins ? wa + 8u * (uint32_t)(wn - 1 - kMargin)
                                                : wa + 8u * (uint32_t)(wn - 1);
            c.moved = 0u;
            c.turned = Turned{0u, 0u};
            c.accm = 0u;
            c.s = 0;
            unsigned applied = 0u;
            for (;;) {
                int why = 0;
                if (m == 0) why = run_chain<S, ks, BYTES>(c, steps, lim, F, lo, hi);
                __syncwarp(gmask);
                // steps taken, reason and bin of the first lane
                const uint32_t pk = __shfl_sync(gmask, ((c.xa - wa) & 0xFFFFFu) | ((uint32_t)c.s << 20) | ((uint32_t)why << 28), gbase);
                c.accm = __shfl_sync(gmask, c.accm, gbase);
                c.s = (int)((pk >> 20) & 0x3Fu);
                c.xa = wa + (pk & 0xFFFFFu);
                why = (int)(pk >> 28);
                // the lists (distinct slots: a second step on a slot is out of date)
                if (((c.accm & ~applied) >> m) & 1u) {
                    perm[d.a] = (IDX)j;
                    perm[ell + d.b] = (IDX)i;
                    if constexpr (!BYTES) {
                        atomicAnd(&st.sp[i >> 5], ~(1u << (i & 31u)));
                        atomicOr(&st.sp[j >> 5], 1u << (j & 31u));
                    }
                }
                applied = c.accm;
                if constexpr (BYTES) {
                    c.turned.up = __shfl_sync(gmask, c.turned.up, gbase);
                    c.turned.down = __shfl_sync(gmask, c.turned.down, gbase);
                }
                __syncwarp(gmask);
                if (why != 1) break;
                // step c.s again, from the lists and spins as they now are
                const uint32_t ac = __shfl_sync(gmask, d.a, gbase + c.s);
                const uint32_t bb = __shfl_sync(gmask, d.b, gbase + c.s);
                const uint32_t i2 = (uint32_t)perm[ac], j2 = (uint32_t)perm[ell + bb];
                dk = exchange_dk<LAT, BYTES, false>(A.g, st, i2, j2, c.turned, nullptr);
                if (m == c.s) {
                    i = i2;
                    j = j2;
                    steps->a[m].z = 0u;
                    steps->a[m].w = (uint32_t)((dk >> ks) * 8);
                    if constexpr (BYTES) {
                        // its sites by kind and owner: turning them toggles those bits
                        const uint32_t pi = st.peek(i2), pj = st.peek(j2);
                        const uint32_t bi = owner_bit(pi), bj = owner_bit(pj);
                        steps->b[m] = make_uint2((pi >> 7 ? bi : 0u) | (pj >> 7 ? bj : 0u),
                                                 (pi >> 7 ? 0u : bi) | (pj >> 7 ? 0u : bj));
                    }
                }
                __syncwarp(gmask);
            }
            if constexpr (BYTES) {
                // every owner writes back its two sites
                if (oi == 1u << m) st.clear(i0, ((c.turned.up >> m) & 1u) ^ 1u);
                if (oj == 1u << m) st.clear(j0, (c.turned.down >> m) & 1u);
                __syncwarp(gmask);
            }
            const int taken = c.s;
            accepts += __popc(c.accm);
            batches += 1;
            const int x = (int)(c.xa - wa) >> 3;
            bc = wb + x;
            if (taken == 0 || x < 0 || x >= wn) {
                stop = 4;                  // never: a step from inside the margins stays inside
                break;
            }
            t += taken;
            left -= taken;
            if (c.xa < lo || c.xa > hi) {
                // re-centre the window
                if (group_ballot<S>(gmask, gbase, window_store<S>(wl, lng, hist, wb, wn, m, F))) stop = 2;
                __syncwarp(gmask);
                wb = window_base(bc, nbins, A.win_bins);
                window_load<S>(wl, lng, wb, wn, m);
                __syncwarp(gmask);
                c.xa = wa + 8u * (uint32_t)(bc - wb);
            }
            d = dn;
            if (taken != S) d = draw_step<DET>((uint64_t)(t + m), key, (uint32_t)ell, nd, A);
            if (stop) break;
        }
        if (stop) break;

        if (t == next_check) {
            // window -> global, then test flatness over the line
            __syncwarp(gmask);
            if (group_ballot<S>(gmask, gbase, window_store<S>(wl, lng, hist, wb, wn, m, F))) {
                stop = 2;
                break;
            }
            __syncwarp(gmask);
            checks += 1;
            const bool flat = group_flat<S>(hist, nbins, m, gmask, A.flat_pm);
            // extra reset at unchanged f within the first R checks of a stage (the
            // remark after Eq. 4): histogram reset, ln g shifted
            const bool again = !flat && A.same_f_resets > 0 && (t - t_stage) / C <= A.same_f_resets;
            if (flat || again) {
                group_stage_step<S>(lng, hist, nbins, m, gmask);
                window_load<S>(wl, lng, wb, wn, m);
                __syncwarp(gmask);
                c.u = wl[bc - wb];
            }
            if (flat) {
                stage += 1;
                t_stage = t;
                F >>= 2;                     // ln f -> ln f / 4
                if (F == 0) {                // ln f < ln f_min
                    status = 1;
                    break;
                }
            }
            // stop requests are read by one lane and broadcast, so the group
            // stays converged; a time-limited slice ends here without an error
            int req = 0;
            if (m == 0) {
                const uint64_t now = globaltimer_ns();
                if (A.slice_end_ns && *A.slice_end_ns && now > *A.slice_end_ns) req = 5;
                if (A.deadline_ns && *A.deadline_ns && now > *A.deadline_ns) req = 1;
                if (A.abort_flag && *A.abort_flag) req = 3;
            }
            req = __shfl_sync(gmask, req, gbase);
            if (req) stop = req;
        }
    }
    // window -> global (a converged line was stored at its last check)
    if (stop != 4 && F != 0) {
        __syncwarp(gmask);
        if (group_ballot<S>(gmask, gbase, window_store<S>(wl, lng, hist, wb, wn, m, F)) && stop == 0)
            stop = 2;
    }
    if (stop == 2) status = 2;
    if (stop == 4) status = 3;
    if (m == 0) {
        P->k = (int64_t)bc << ks;
        P->t = t;
        P->F = F;
        P->stage = stage;
        P->accepts = accepts;
        P->t_stage = t_stage;
        P->status = status;
        P->checks = checks;
        P->batches = batches;
        if (stop == 1) atomicOr(A.flags, 1);
        if (stop == 3) atomicOr(A.flags, 2);
        if (stop == 2) atomicOr(A.flags, 4);
        if (stop == 4) atomicOr(A.flags, 8);
    }
    __syncwarp(gmask);
}

// Copy n 32-bit words with the group's lanes (16-byte chunks when aligned).
template <int S>
__device__ __forceinline__ void group_copy(uint32_t* dst, const uint32_t* src, int nwords, int m)
{
    if (((reinterpret_cast<uintptr_t>(dst) | reinterpret_cast<uintptr_t>(src)) & 15u) == 0) {
        const int n4 = nwords >> 2;
        uint4* d4 = reinterpret_cast<uint4*>(dst);
        const uint4* s4 = reinterpret_cast<const uint4*>(src);
        for (int x = m; x < n4; x += S) d4[x] = s4[x];
        for (int x = (n4 << 2) + m; x < nwords; x += S) dst[x] = src[x];
    } else {
        for (int x = m; x < nwords; x += S) dst[x] = src[x];
    }
}

// Packed spins -> one byte per site (no owners) and back, a 32-site word per lane
// and round, four sites at a time: the products spread a nibble's bits over the
// bytes of a word and gather them again (no two partial products meet).
template <int S>
__device__ __forceinline__ void sites_load(uint8_t* own, const uint32_t* sp, int N, int m)
{
    uint32_t* o = reinterpret_cast<uint32_t*>(own);
#pragma unroll 2
    for (int w = m; w * 32 < N; w += S) {
        const uint32_t v = sp[w];
#pragma unroll
        for (int b = 0; b < 8; ++b)
            o[w * 8 + b] = (((((v >> (4 * b)) & 0xFu) * 0x00204081u) & 0x01010101u) << 7) | (kNoOwner * 0x01010101u);
    }
}

template <int S>
__device__ __forceinline__ void sites_store(uint32_t* sp, const uint8_t* own, int N, int m)
{
    const uint32_t* o = reinterpret_cast<const uint32_t*>(own);
    for (int w = m; w * 32 < N; w += S) {
        uint32_t v = 0u;
#pragma unroll
        for (int b = 0; b < 8; ++b)
            v |= (((((o[w * 8 + b] >> 7) & 0x01010101u) * 0x01020408u) >> 24) & 0xFu) << (4 * b);
        sp[w] = v;
    }
}

// Persistent walker: every group pops lines from the work queue until it is
// empty.  With one group and a one-entry queue the same kernel is the plain
// one-launch-per-line form.  A group's slot of shared memory: the list (when
// staged), the window, the sites, the step records (plan_slot in wl_plan.h).
template <int LAT, int S, bool DET, typename IDX, bool BYTES>
__global__ void walk_kernel(const WalkArgs A)
{
    extern __shared__ __align__(16) uint8_t smem[];
    const int lane = threadIdx.x & 31;
    const int m = lane % S;
    const int gbase = lane - m;
    const unsigned gmask = group_mask<S>(gbase);
    const int gid = threadIdx.x / S;
    uint8_t* slot = smem + (size_t)gid * (size_t)A.slot_bytes;
    int64_t* wl = reinterpret_cast<int64_t*>(slot + A.off_win);
    static_assert(sizeof(Steps<S>) <= (kStepBytes * S + 15) / 16 * 16, "plan_slot");
    Steps<S>* steps = reinterpret_cast<Steps<S>*>(slot + A.off_rec);
    Sites<BYTES> st{slot + A.off_sites, nullptr, (uint32_t)A.owner_mask};
    if constexpr (!BYTES) {
        for (int x = m; x <= A.owner_mask; x += S) st.own[x] = (uint8_t)kNoOwner;
        __syncwarp(gmask);
    }
    // per-line strides are padded to 16 bytes: pstride list entries, W spin words
    const int pstride = A.pstride, W = A.g.W;
    const int perm_words = (int)((size_t)pstride * sizeof(IDX) / 4);

    for (;;) {
        int qi = 0;
        if (m == 0) qi = atomicAdd(A.qnext, 1);
        qi = __shfl_sync(gmask, qi, gbase);
        if (qi >= A.nqueue) break;
        const int li = queue_line(A, qi);
        if (A.st[li].status != 0) continue;
        IDX* gperm = reinterpret_cast<IDX*>(A.perm) + (size_t)li * pstride;
        uint32_t* gsp = A.spins + (size_t)li * W;
        IDX* perm = gperm;
        if (A.stage_perm) {
            perm = reinterpret_cast<IDX*>(slot);
            group_copy<S>(reinterpret_cast<uint32_t*>(perm), reinterpret_cast<const uint32_t*>(gperm),
                          perm_words, m);
        }
        if constexpr (BYTES) sites_load<S>(st.own, gsp, A.g.N, m);
        else st.sp = gsp;
        __syncwarp(gmask);
        walk_line<LAT, S, DET, IDX, BYTES>(A, li, m, gbase, gmask, perm, st, wl, steps);
        if (A.stage_perm)
            group_copy<S>(reinterpret_cast<uint32_t*>(gperm), reinterpret_cast<const uint32_t*>(perm),
                          perm_words, m);
        if constexpr (BYTES) sites_store<S>(gsp, st.own, A.g.N, m);
        __syncwarp(gmask);
    }
}

}  // namespace wl
