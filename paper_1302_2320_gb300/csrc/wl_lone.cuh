// wl_lone.cuh -- the walker for lines whose state fits a share of an SM's shared memory:
// one block per line, made for the time of one step (arXiv:1302.2320, the procedure
// around Eq. 3 and Eq. 4).  plan_shape chooses between it and batches (wl_walk.cuh).
//
// The chain of a line is serial, and the time to the end of a surface is that of its
// slowest line, so what counts is the latency from one decision to the next.  No step
// is evaluated on a guess, so a line of few up spins or a tiny lattice, where
// neighbouring steps draw the same list slots all the time, walks as fast as any other:
// ~120 cycles a step (square 16x16 to 64x64, cubic 8^3, triangular 32x32; batches: 160
// to 1000, and the walker before both 180 to 420).  From decision to decision there are
//   - the change of the words around the two sites (below), then two loads of words;
//   - the proposed bin, one load of ln g at it, the 64-bit compare.
// Everything else a step needs lies off that path:
//   - the second warp draws the random numbers, up to three batches of 32 steps
//     ahead, into a ring in shared memory (they depend on the step number only);
//   - every site has a word with its number of up neighbours, so that a proposal
//     needs two loads; an exchange changes the words of the 2z sites around it, one
//     lane each, with one shared-memory reduction;
//   - the sites in the next step's list slots are loaded a step ahead; where it
//     shares a slot with the step being decided, the decision says what is there;
//   - the neighbours of a step's sites are worked out while ln g is on its way.
// A shared-memory instruction of one warp takes 2.5 (load) to 4 (store) cycles to
// issue, which is what the rest of a step is made of.  Forms that were slower: one
// thread that reads the 2z neighbours' spins itself (15 loads, 7 stores: 180 cycles a
// step); the next step evaluated for both outcomes of the pending one, in two halves of
// each word (116 where slots are rarely shared, 200 where they often are, and with two
// codes for the two the instruction cache suffers where handles share an SM).
//
// Sites are kept as the addresses of their words past the start of the shared memory;
// rows have a power-of-two stride, (y << s) | x, so that coordinates need no division
// and a list entry no address arithmetic.
//
// WORD: bytes of a site's word.  With 4 a step is shorter (119 cycles against 126: no
// shift into place); with 1 a line takes little shared memory, so that more of them
// share an SM and fill each other's gaps (96x96: 6 instead of 2 an SM, 27 cycles a move
// and SM; 64x64, 7 an SM with either: 23 and 24), and 256x256 fits.  What bounds 7 to 12
// walkers on an SM together is issue (57 to 70 % of its slots, ~51 instructions a step
// with the drawing warp's) and the shared-memory pipe (63 to 74 %, 14 cycles a step).
#pragma once

#include "wl_walk.cuh"

namespace wl {

// The ring of draws: per step {dmax (two words), U slot, D slot} and the same with the
// slots the other way round, for the lanes of the down site.
constexpr int kRing = 96;                  // steps (3 batches of 32)
constexpr int kRingMore = 3;               // the first records again past the end: a step reads up to 3 ahead
constexpr int kLoneThreads = 64;           // one warp walks, one draws

// The lattice is a run-time matter but for the second axis of the triangular one's
// diagonals (TRI): requests for different lattices that share an SM then run the same
// code, and do not drive each other's out of its instruction cache (eight requests of
// five lattices: 121 ms with a kernel for each lattice, each 26 ms alone).
__device__ __forceinline__ uint32_t site_code(const Geo& g, uint32_t n)
{
    const uint32_t L = (uint32_t)g.L, r = divL(g, n), x = n - r * L;
    if (g.shape == kShapeCubic) {
        const uint32_t z = divL(g, r), y = r - z * L;
        return (((z << g.cshift) | y) << g.cshift) | x;
    }
    return ((r + (g.shape == kShapeOpen ? 1u : 0u)) << g.cshift) | x;
}

__device__ __forceinline__ uint32_t code_site(const Geo& g, uint32_t c)
{
    const uint32_t L = (uint32_t)g.L, x = c & g.cmask;
    if (g.shape == kShapeCubic) {
        const uint32_t y = (c >> g.cshift) & g.cmask, z = c >> (2 * g.cshift);
        return (z * L + y) * L + x;
    }
    return ((c >> g.cshift) - (g.shape == kShapeOpen ? 1u : 0u)) * L + x;
}

// The word of site n (LoneLane).
template <int LAT>
__device__ __forceinline__ uint32_t site_word(const Geo& g, const uint32_t* sp, uint32_t n)
{
    constexpr int z = Coord<LAT>::z;
    uint32_t nb[z];
    int u = 0;
    if constexpr (LAT == kSquareOpen) {
        const unsigned v = open_neighbours(g, n, nb);
#pragma unroll
        for (int q = 0; q < z; ++q) u += (int)((v >> q) & 1u & spin_at(sp, nb[q]));
        u = 2 * u - __popc(v);
    } else {
        neighbours<LAT>(g, n, nb);
#pragma unroll
        for (int q = 0; q < z; ++q) u += (int)spin_at(sp, nb[q]);
    }
    return (uint32_t)(8 * u) + (LAT == kSquareOpen ? 32u : 0u);
}

// Shared memory by 32-bit address (generic pointers cost 64-bit address arithmetic).
// Volatile, so that they stay in the order written here.
__device__ __forceinline__ uint32_t lds16(uint32_t a)
{
    uint32_t v;
    asm volatile("{.reg .u16 h;\n\tld.shared.u16 h, [%1];\n\tcvt.u32.u16 %0, h;}" : "=r"(v) : "r"(a) : "memory");
    return v;
}
template <int WORD>
__device__ __forceinline__ uint32_t lds_word(uint32_t a)      // the word of the site at a
{
    uint32_t v;
    if constexpr (WORD == 4)
        asm volatile("ld.shared.u32 %0, [%1+1024];" : "=r"(v) : "r"(a) : "memory");
    else
        asm volatile("ld.shared.u8 %0, [%1+1024];" : "=r"(v) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ uint2 lds64u(uint32_t a)
{
    uint2 v;
    asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ int64_t lds64(uint32_t a)
{
    int64_t v;
    asm volatile("ld.shared.s64 %0, [%1];" : "=l"(v) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ void sts64(uint32_t a, int64_t v)
{
    asm volatile("st.shared.s64 [%0], %1;" ::"r"(a), "l"(v) : "memory");
}
__device__ __forceinline__ void sts16(uint32_t a, uint32_t v)
{
    asm volatile("{.reg .u16 h;\n\tcvt.u16.u32 h, %1;\n\tst.shared.u16 [%0], h;}" ::"r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ void red_word(uint32_t a, uint32_t v)     // a: a multiple of 4
{
    asm volatile("red.shared.add.u32 [%0+1024], %1;" ::"r"(a), "r"(v) : "memory");
}
static_assert(kLow == 1024u, "the offset in lds_word and red_word");

// The two warps of a block keep step at a barrier per batch of 32 steps.  The lanes of a
// warp come to it together, and its form allows for those that do not.
__device__ __forceinline__ void lone_barrier()
{
    __syncwarp();
    asm volatile("barrier.sync 1, 64;" ::: "memory");
}

// The lanes of the walking warp.  Lane q < z stands for neighbour q of the pending
// step's up site, lane z + q for neighbour q of its down site.  The others go along, so
// that no step branches: they load and store the same, and each has a word of its own
// in the place of a neighbour's; the first of them counts the accepted steps in its.
//
// A word holds 8 for every up neighbour, the bytes of one bin of ln g: half the change
// of k.  With open boundaries bins are half as wide, and a word holds 16 for every up
// neighbour less 8 for every neighbour, plus 32; a missing neighbour is a word of the
// border around the lattice, which nobody reads.  Words stay within 0 .. 255, so that
// what is added to one of the four in 32 bits never reaches the next.
template <bool TRI, int WORD>
struct LoneLane {
    uint32_t swap;                   // 16 for the lanes of the down site: their order in a ring record
    int32_t sign;                    // own word less the other's, as up less down
    uint32_t unit;                   // added if the sites are neighbours
    uint32_t accept;                 // what an accepted step adds to this lane's word
    uint32_t scale;                  // 0 for a lane without a neighbour
    uint32_t s0, m0, e0, d0, w0;     // along one axis: shift, mask, coordinate at the edge, step, step at the edge
    uint32_t s1, m1, e1, d1, w1;     // along the other (triangular diagonals)

    __device__ __forceinline__ void setup(const Geo& g, int lane, uint32_t spare)
    {
        const int z = g.shape == kShapeTriangular || g.shape == kShapeCubic ? 6 : 4;
        const bool open = g.shape == kShapeOpen;
        unit = open ? 16u : 8u;
        const int q = lane % z;
        const bool down = ((lane / z) & 1) != 0;
        swap = down ? 16u : 0u;
        sign = down ? -1 : 1;
        accept = down ? unit : 0u - unit;            // the up site goes, the down site comes
        const uint32_t e = (uint32_t)g.L - 1u;
        auto axis = [&](int ax, bool plus, uint32_t& s, uint32_t& mk, uint32_t& ed, uint32_t& d, uint32_t& w) {
            s = (uint32_t)(ax * g.cshift) + (WORD == 4 ? 2u : 0u);
            const uint32_t u = 1u << s;
            mk = g.cmask;
            ed = plus ? e : 0u;
            d = plus ? u : 0u - u;
            w = open ? d : plus ? 0u - e * u : e * u;
        };
        // neighbours in the order of neighbours<LAT>: +-x, +-y, (+-z | the diagonals)
        s1 = m1 = d1 = w1 = 0u;
        e1 = 1u;
        if (TRI && q >= 4) {
            axis(0, q == 4, s0, m0, e0, d0, w0);
            axis(1, q == 5, s1, m1, e1, d1, w1);
        } else {
            axis(q >> 1, (q & 1) == 0, s0, m0, e0, d0, w0);
        }
        scale = 1u;
        if (lane >= 2 * z) {
            scale = d1 = w1 = 0u;
            accept = lane == 2 * z ? 1u : 0u;
            d0 = w0 = spare - kLow + 4u * (uint32_t)lane;
        }
    }

    // Address of the word of this lane's neighbour of the site at c.
    __device__ __forceinline__ uint32_t neighbour(uint32_t c) const
    {
        uint32_t n = (((c >> s0) & m0) == e0 ? w0 : d0) + c * scale;
        if constexpr (TRI) n += ((c >> s1) & m1) == e1 ? w1 : d1;
        return n;
    }
};

// A walker's state: the pending step (this lane's own site and the other one, its
// neighbour, the bin it proposes), the sites of the step after it, and the list slots of
// both and of the one after that.  Sites are the addresses of their words; xa, ta and u
// are the same in every lane.
struct Lone {
    uint32_t xa;            // address of the current bin
    uint32_t ta;            // address of the bin the pending step proposes
    int64_t u;              // ln g of the current bin
    uint32_t own, oth, nb;  // pending step
    uint32_t add;           // what it adds to the four words around nb's if accepted
    uint32_t own1, oth1;    // the step after it
    uint2 slot0, slot1, slot2;      // own, other
};

// The pending step's neighbour of this lane and the bin it proposes, from the words wo
// and wt of its sites.
template <bool TRI, int WORD>
__device__ __forceinline__ void lone_propose(Lone& w, const LoneLane<TRI, WORD>& L, uint32_t wo, uint32_t wt)
{
    w.nb = L.neighbour(w.own);
    const uint32_t at = w.xa + (__any_sync(0xffffffffu, w.nb == w.oth) ? L.unit : 0u);
    w.add = L.accept;
    if constexpr (WORD == 1) {
        w.add = __funnelshift_l(0u, L.accept, w.nb << 3);     // by 8 (nb & 3)
        w.nb &= ~3u;
    }
    w.ta = at + (uint32_t)((int32_t)(wo - wt) * L.sign);
}

// One step: decide the pending one, write it back, propose the next.  `at`: the pending
// step's record in the ring, in this lane's order.  The order of the memory accesses is
// the order they are written in here: the reduction first and the words right behind
// it, the stores the next decision does not wait for after them.
template <bool TRI, int WORD>
__device__ __forceinline__ void lone_step(Lone& w, const LoneLane<TRI, WORD>& L, uint32_t at, int64_t F)
{
    const int64_t gt = lds64(w.ta);
    const int64_t dmax = lds64(at);
    const bool p = gt <= w.u + dmax;
    // what the two slots hold now, and the next step's sites with it
    const uint32_t no = p ? w.oth : w.own, nt = p ? w.own : w.oth;
    w.own = w.slot1.x == w.slot0.x ? no : w.own1;
    w.oth = w.slot1.y == w.slot0.y ? nt : w.oth1;
    red_word(w.nb, p ? w.add : 0u);
    __syncwarp();
    const uint32_t wo = lds_word<WORD>(w.own), wt = lds_word<WORD>(w.oth);
    w.xa = p ? w.ta : w.xa;
    w.u = (p ? gt : w.u) + F;
    sts16(w.slot0.x, no);                // the lanes of either site write its slot
    sts64(w.xa, w.u);
    __syncwarp();
    w.own1 = lds16(w.slot2.x);
    w.oth1 = lds16(w.slot2.y);
    w.slot0 = w.slot1;
    w.slot1 = w.slot2;
    w.slot2 = lds64u(at + 104u);
    lone_propose<TRI, WORD>(w, L, wo, wt);
}

template <bool TRI, int WORD, int K>
__device__ __forceinline__ void lone_block(Lone& w, const LoneLane<TRI, WORD>& L, uint32_t& at, int64_t F)
{
#pragma unroll
    for (int q = 0; q < K; ++q) lone_step<TRI, WORD>(w, L, at + 32u * q, F);
    at += 32u * K;
}

// Take n <= 16 steps, from the record at `at` on, in blocks: the end of a loop's body
// costs ~75 cycles (the compiler lets the loops of a kernel yield whose warps part
// before a barrier).  16x16, l = 4: 126 cycles a step in blocks of 8, 118 of 16.
template <bool TRI, int WORD>
__device__ __forceinline__ void lone_run(Lone& w, const LoneLane<TRI, WORD>& L, uint32_t at, int n, int64_t F)
{
    if (n == 16) {
        lone_block<TRI, WORD, 16>(w, L, at, F);
        return;
    }
#pragma unroll 1
    for (; n >= 4; n -= 4) lone_block<TRI, WORD, 4>(w, L, at, F);
#pragma unroll 1
    for (; n > 0; --n) lone_block<TRI, WORD, 1>(w, L, at, F);
}

// The drawing warp: batches of 32 steps from t on, until the walker is done.
template <bool DET>
__device__ __forceinline__ void lone_draw(const WalkArgs& A, int64_t t, int ell, uint4* ring, uint32_t perm,
                                          const volatile uint64_t* last, int lane)
{
    const uint2 key = make_uint2((uint32_t)ell, A.seed);
    const uint32_t nd = (uint32_t)(A.g.N - ell);
    auto fill = [&](uint64_t k, uint32_t at) {
        const Draw d = draw_step<DET>((uint64_t)t + 32u * k + (uint64_t)lane, key, (uint32_t)ell, nd, A);
        const uint32_t sa = perm + 2u * d.a, sb = perm + 2u * ((uint32_t)ell + d.b);
        const uint4 r = make_uint4((uint32_t)d.dmax, (uint32_t)((uint64_t)d.dmax >> 32), sa, sb);
        const uint4 q = make_uint4(r.x, r.y, sb, sa);
        at += (uint32_t)lane;
        ring[2u * at] = r;
        ring[2u * at + 1u] = q;
        if (at < kRingMore) {
            ring[2u * (kRing + at)] = r;
            ring[2u * (kRing + at) + 1u] = q;
        }
    };
    fill(0u, 0u);
    fill(1u, 32u);
    lone_barrier();
    uint32_t at = 64u;
    for (uint64_t k = 2u;; ++k) {            // the k-th barrier
        fill(k, at);
        at = at == 64u ? 0u : at + 32u;
        lone_barrier();
        if (*last == k) break;
    }
}

// The walking warp: line `li` for up to A.slice_moves moves (or to its budget, or
// to convergence); the bookkeeping between steps as in walk_line.
template <bool TRI, int WORD>
__device__ __forceinline__ void lone_walk(const WalkArgs& A, int li, int m, uint8_t* sm, const uint4* ring,
                                          uint32_t* spare, volatile uint64_t* last)
{
    const bool open = A.g.shape == kShapeOpen;
    const int ks = open ? 0 : 1;
    const int zb = open ? 8 : A.g.shape == kShapeTriangular || A.g.shape == kShapeCubic ? 6 : 4;    // Coord::zbin
    const int kMargin = 16 * zb;         // a run of steps stays inside the window
    constexpr unsigned all = 0xffffffffu;
    const LineDesc D = A.desc[li];
    LineState* P = A.st + li;
    // what only a check needs stays in memory: registers are few
    int64_t t = P->t, F = P->F;
    const int nbins = D.nbins;
    int64_t* lng = A.lng + D.bin_off;
    hist_t* hist = A.hist + D.bin_off;
    // a turn's share of the moves of this launch
    const int64_t moves = A.turns > 1 && A.slice_moves > A.budget ? A.budget : A.slice_moves;
    int64_t end = t + (A.turns > 1 ? (moves + A.turns - 1) / A.turns : moves);
    if (end > A.budget) end = A.budget;
    const int64_t C = A.C_per_bin > 0 && A.C_per_bin * nbins > A.C ? A.C_per_bin * nbins : A.C;

    int stop = 0;
    int bc = (int)P->k >> ks;
    if (bc < 0 || bc >= nbins) {
        stop = 4;                 // not a state of this line
        bc = 0;
        end = t;
    }
    const int wn = nbins < A.win_bins ? nbins : A.win_bins;
    int wb = window_base(bc, nbins, A.win_bins);
    int64_t* wl = reinterpret_cast<int64_t*>(sm + A.off_win);
    window_load<32>(wl, lng, wb, wn, m);
    __syncwarp(all);
    const uint32_t wa = (uint32_t)__cvta_generic_to_shared(wl);
    LoneLane<TRI, WORD> L;
    L.setup(A.g, m, (uint32_t)__cvta_generic_to_shared(spare));
    const uint32_t ring_at = (uint32_t)__cvta_generic_to_shared(ring) + L.swap;
    uint32_t* counter = spare + (zb == 6 ? 12 : 8);       // the first lane past the neighbours
    Lone w{};
    w.xa = wa + 8u * (uint32_t)(bc - wb);
    w.u = wl[bc - wb];
    if (m == 0) *counter = 0u;
    lone_barrier();               // the first two batches are drawn
    uint64_t barriers = 1u;
    if (t < end) {
        // the first step is pending, the second loaded, the third's slots at hand
        w.slot0 = lds64u(ring_at + 8u);
        w.slot1 = lds64u(ring_at + 40u);
        w.slot2 = lds64u(ring_at + 72u);
        w.own = lds16(w.slot0.x);
        w.oth = lds16(w.slot0.y);
        w.own1 = lds16(w.slot1.x);
        w.oth1 = lds16(w.slot1.y);
        const uint32_t wo = lds_word<WORD>(w.own), wt = lds_word<WORD>(w.oth);
        lone_propose<TRI, WORD>(w, L, wo, wt);
    }
    __syncwarp(all);

    uint32_t pos = 0u;                       // steps since t0, modulo 2^32
    uint32_t at = ring_at;                   // the pending step's record
    uint32_t lo = 0u, hi = 0u;               // the bins a run of 16 steps may start from
    auto set_margins = [&]() {
        lo = wb > 0 ? wa + 8u * (uint32_t)kMargin : wa;
        hi = wa + 8u * (uint32_t)(wn - 1 - (wb + wn < nbins ? kMargin : 0));
    };
    set_margins();
    while (t < end && !stop) {
        const int64_t next_check = (t / C + 1) * C;
        int64_t seg_end = next_check < end ? next_check : end;
        if (seg_end - t > (1ll << 30)) seg_end = t + (1ll << 30);
        int64_t left = seg_end - t;
        while (left > 0) {
            const uint32_t in = pos & 15u;
            const int n = left < 16 - (int)in ? (int)left : 16 - (int)in;
            lone_run<TRI, WORD>(w, L, at, n, F);
            pos += (uint32_t)n;
            at += 32u * (uint32_t)n;
            left -= n;
            if (w.xa < lo || w.xa > hi) {
                const uint32_t xa = w.xa;
                bc = wb + ((int)(xa - wa) >> 3);
                if (xa < wa || bc - wb >= wn) {
                    stop = 4;              // never: a run from inside the margins stays inside
                } else {
                    // re-centre the window
                    __syncwarp(all);
                    if (__any_sync(all, window_store<32>(wl, lng, hist, wb, wn, m, F))) stop = 2;
                    __syncwarp(all);
                    wb = window_base(bc, nbins, A.win_bins);
                    window_load<32>(wl, lng, wb, wn, m);
                    __syncwarp(all);
                    const uint32_t to = wa + 8u * (uint32_t)(bc - wb);
                    w.ta += to - xa;
                    w.xa = to;
                    set_margins();
                }
            }
            if ((pos & 31u) == 0u) {
                lone_barrier();
                ++barriers;
                if (at == ring_at + 32u * kRing) at = ring_at;
            }
            if (stop) break;
        }
        t = seg_end - left;
        bc = wb + ((int)(w.xa - wa) >> 3);
        // a segment is short enough for the 32-bit counter
        __syncwarp(all);
        if (m == 0) {
            P->accepts += *counter;
            *counter = 0u;
        }
        __syncwarp(all);
        if (stop) break;

        if (t == next_check) {
            // window -> global, then test flatness over the line
            __syncwarp(all);
            if (__ballot_sync(all, window_store<32>(wl, lng, hist, wb, wn, m, F))) {
                stop = 2;
                break;
            }
            __syncwarp(all);
            if (m == 0) P->checks += 1;
            const bool flat = group_flat<32>(hist, nbins, m, all, A.flat_pm);
            const bool again = !flat && A.same_f_resets > 0 && (t - P->t_stage) / C <= A.same_f_resets;
            if (flat || again) {
                group_stage_step<32>(lng, hist, nbins, m, all);
                window_load<32>(wl, lng, wb, wn, m);
                __syncwarp(all);
                w.u = wl[bc - wb];
            }
            if (flat) {
                __syncwarp(all);
                if (m == 0) {
                    P->stage += 1;
                    P->t_stage = t;
                }
                __syncwarp(all);
                F >>= 2;                     // ln f -> ln f / 4
                if (F == 0) break;           // ln f < ln f_min
            }
            int req = 0;
            if (m == 0) {
                const uint64_t now = globaltimer_ns();
                if (A.slice_end_ns && *A.slice_end_ns && now > *A.slice_end_ns) req = 5;
                if (A.deadline_ns && *A.deadline_ns && now > *A.deadline_ns) req = 1;
                if (A.abort_flag && *A.abort_flag) req = 3;
            }
            req = __shfl_sync(all, req, 0);
            if (req) stop = req;
        }
    }
    // the pending step is dropped: it is drawn again next time
    if (stop != 4 && F != 0) {
        __syncwarp(all);
        if (__ballot_sync(all, window_store<32>(wl, lng, hist, wb, wn, m, F)) && stop == 0) stop = 2;
    }
    if (m == 0) {
        if (F == 0) P->status = 1;
        if (stop == 2) P->status = 2;
        if (stop == 4) P->status = 3;
        P->k = (int64_t)bc << ks;
        P->batches += (t - P->t + 31) / 32;
        P->t = t;
        P->F = F;
        if (stop == 1) atomicOr(A.flags, 1);
        if (stop == 3) atomicOr(A.flags, 2);
        if (stop == 2) atomicOr(A.flags, 4);
        if (stop == 4) atomicOr(A.flags, 8);
        *last = barriers + 1u;           // the next one
    }
    __syncwarp(all);
    lone_barrier();
}

// Turn r of a line: once the block that has the turn before it, an earlier entry of the
// queue and so running or done, is through with it.  Not taken when the slice is over,
// or when that takes a second: the line goes on in the next slice.
__device__ __noinline__ bool lone_turn(const WalkArgs& A, int li, int r)
{
    for (int n = 0; n < (1 << 20); ++n) {
        const uint64_t now = globaltimer_ns();
        if (A.slice_end_ns && *A.slice_end_ns && now > *A.slice_end_ns) return false;
        if (A.deadline_ns && *A.deadline_ns && now > *A.deadline_ns) return false;
        if (A.abort_flag && *A.abort_flag) return false;
        int done;
        asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(done) : "l"(A.turn + li) : "memory");
        if (done >= r) return true;
        __nanosleep(1000);
    }
    return false;
}
__device__ __forceinline__ void turn_done(int32_t* turn, int done)
{
    __threadfence();
    asm volatile("st.release.gpu.global.s32 [%0], %1;" ::"l"(turn), "r"(done) : "memory");
}

// One block per line: shared memory holds the words of the sites, the list, the window,
// the ring of draws.
//
// Registers for 10 blocks on an SM: a burst of eight requests (square, triangular,
// cubic, open; 10 blocks an SM) takes 29 ms, 38 with room for 8, when the last request
// waits for the others; alone a step costs the same (119 and 120 cycles).  Triangular
// lattices keep more (122 cycles a step against 129).
template <bool TRI, bool DET, int WORD>
__global__ void __launch_bounds__(kLoneThreads, TRI && WORD == 4 ? 8 : 10) lone_kernel(const WalkArgs A)
{
    extern __shared__ __align__(16) uint8_t smem[];
    const int th = threadIdx.x, warp = th >> 5, lane = th & 31;
    if ((uint32_t)__cvta_generic_to_shared(smem) != kLow) {      // never: plan_shape
        if (th == 0) atomicOr(A.flags, 8);
        return;
    }
    uint16_t* perm = reinterpret_cast<uint16_t*>(smem + A.off_perm);
    uint4* ring = reinterpret_cast<uint4*>(smem + A.off_rec);
    int32_t* ctl = reinterpret_cast<int32_t*>(ring + 2 * (kRing + kRingMore));    // the line; who walks; the barrier at which the walker is done
    if (th == 0) {
        // The SM deals its warps out to four schedulers in order of their slots: were
        // it always the first warp of a block that walks, all walkers would share two
        // of them.  Any choice is right; this one spreads them over all four.
        uint32_t slot;
        asm volatile("mov.u32 %0, %%warpid;" : "=r"(slot));
        ctl[1] = (int32_t)((slot >> 2) & 1u);
    }
    uint64_t* last = reinterpret_cast<uint64_t*>(ctl + 2);
    uint32_t* spare = reinterpret_cast<uint32_t*>(ctl + 4);
    const int N = A.g.N, pstride = A.pstride;
    int turn = 0;
    for (;;) {
        if (th == 0) {
            const int qi = atomicAdd(A.qnext, 1);
            const int r = A.turns > 1 ? qi / A.nqueue : 0;       // the line's turn
            const int x = qi - r * A.nqueue;
            int li = r < (A.turns > 1 ? A.turns : 1) && x < A.nqueue ? queue_line(A, x) : -1;
            if (li >= 0 && r > 0 && !lone_turn(A, li, r)) li = -2;
            ctl[0] = li;
            *last = 0u;
            turn = r;
        }
        __syncthreads();
        const int li = ctl[0];
        if (li == -1) break;
        if (li >= 0 && A.st[li].status == 0) {
            uint16_t* gperm = reinterpret_cast<uint16_t*>(A.perm) + (size_t)li * pstride;
            uint32_t* gsp = A.spins + (size_t)li * A.g.W;
            if (A.g.shape == kShapeOpen) {           // the border: far from either end of a byte
                for (int x = th; x < A.off_perm; x += kLoneThreads) smem[x] = WORD == 4 && (x & 3) ? 0u : 128u;
                __syncthreads();
            }
            for (int n = th; n < N; n += kLoneThreads) {
                perm[n] = (uint16_t)(WORD * site_code(A.g, gperm[n]));
                const uint32_t u = A.g.shape == kShapeTriangular ? site_word<kTriangular>(A.g, gsp, (uint32_t)n)
                                   : A.g.shape == kShapeCubic    ? site_word<kCubic>(A.g, gsp, (uint32_t)n)
                                   : A.g.shape == kShapeOpen     ? site_word<kSquareOpen>(A.g, gsp, (uint32_t)n)
                                                                 : site_word<kSquare>(A.g, gsp, (uint32_t)n);
                const uint32_t c = site_code(A.g, (uint32_t)n);
                if constexpr (WORD == 4)
                    reinterpret_cast<uint32_t*>(smem)[c] = u;
                else
                    smem[c] = (uint8_t)u;
            }
            const int64_t t = A.st[li].t;
            const int ell = A.desc[li].ell;
            __syncthreads();
            if (warp == ctl[1])
                lone_walk<TRI, WORD>(A, li, lane, smem, ring, spare, last);
            else
                lone_draw<DET>(A, t, ell, ring, (uint32_t)__cvta_generic_to_shared(perm), last, lane);
            __syncthreads();
            // the list, and from it the spins
            uint32_t* sp = reinterpret_cast<uint32_t*>(smem);
            for (int x = th; x * 32 < N; x += kLoneThreads) sp[x] = 0u;
            __syncthreads();
            for (int n = th; n < N; n += kLoneThreads) {
                const uint32_t s = code_site(A.g, perm[n] / (uint32_t)WORD);
                gperm[n] = (uint16_t)s;
                if (n < ell) atomicOr(&sp[s >> 5], 1u << (s & 31u));
            }
            __syncthreads();
            for (int x = th; x * 32 < N; x += kLoneThreads) gsp[x] = sp[x];
        }
        __syncthreads();
        if (th == 0 && li >= 0 && A.turns > 1) turn_done(A.turn + li, turn + 1);
    }
}

}  // namespace wl
