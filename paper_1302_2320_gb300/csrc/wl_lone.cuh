// wl_lone.cuh -- the walker for few lines: one block per line, made for the time
// of one step (arXiv:1302.2320, the procedure around Eq. 3 and Eq. 4).
//
// The chain of a line is serial, and the time to the end of a surface is that of
// its slowest line, so what counts here is the latency from one decision to the
// next: one load of ln g at the proposed bin (~29 cycles), the compare and the
// selects behind it.  Nothing about a step is guessed, so a line with few up spins
// or a tiny lattice, where neighbouring steps meet all the time, walks nearly as
// fast as any other.  What else a step needs is kept off that path:
//   - the second warp draws the random numbers, up to three batches of 32 steps
//     ahead, into a ring in shared memory (they depend on the step number only);
//   - every site has a word with its number of up neighbours, so that a proposal
//     needs two loads; an exchange changes the words of the 2z sites around it, one
//     lane each, with a shared-memory reduction;
//   - the sites of step m+2 are loaded while step m is pending;
//   - while ln g of step m is on its way, step m+1 is evaluated for both of its
//     outcomes.  A site's word holds its count now in the low half and its count
//     if the pending step is accepted in the high half.  A proposal adds its changes
//     to the high halves when it becomes the pending one; its decision adds them to
//     the low halves or takes them back.  The difference of two words then holds
//     both changes of k of step m+1, and the decision picks one by a shift.
// Steps that draw a list slot of one of the two steps before them (flags made with
// the draws) wait for the decision first.
//
// A shared-memory instruction of one warp takes 2.5 (load) to 4 (store) cycles to
// issue, which is what a step is made of: an earlier form in which one thread read
// the 2z neighbours' spins (15 loads, 7 stores a step) took 180 cycles a step.
//
// Sites are kept as the addresses of their words, whose rows have a power-of-two
// stride, so that coordinates need no division and a list entry no address
// arithmetic: 4 ((y << s) | x) past a base aligned to a row (cubic: a plane).
#pragma once

#include "wl_walk.cuh"

namespace wl {

// The ring of draws: per step {dmax (two words), U slot, D slot} and the same with the
// slots the other way round, for the lanes of the down site.
constexpr int kRing = 128;                 // steps (4 batches of 32)
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

// 8 for every up neighbour of site n (open boundaries: 16, less 8 for every neighbour).
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
    return (uint32_t)(8 * u);
}

// Shared memory by 32-bit address (generic pointers cost 64-bit address arithmetic).
// Volatile, so that they stay in the order written here.
__device__ __forceinline__ uint32_t lds16(uint32_t a)
{
    uint32_t v;
    asm volatile("{.reg .u16 h;\n\tld.shared.u16 h, [%1];\n\tcvt.u32.u16 %0, h;}" : "=r"(v) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ uint32_t lds32(uint32_t a)
{
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
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
__device__ __forceinline__ uint4 lds128(uint32_t a)
{
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a) : "memory");
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
__device__ __forceinline__ void reds(uint32_t a, uint32_t v)
{
    asm volatile("red.shared.add.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}

__device__ __forceinline__ void lone_barrier() { asm volatile("bar.sync 1, 64;" ::: "memory"); }

constexpr uint32_t kBias = 128u;            // keeps the two halves of a difference of words apart
constexpr uint32_t kBoth = 0x10001u;        // a number in both halves

// The lanes of the walking warp.  Lane q < z stands for neighbour q of the pending
// step's up site, lane z + q for neighbour q of its down site; the next 2z lanes
// stand for the neighbours of the step after it in the same way, so that one
// reduction writes back the pending step and makes the next one pending.  The
// lanes past those go along, so that no step branches: they load and store the
// same, and each has a word of its own in the place of a neighbour's; the first of
// them counts the accepted steps in its.
//
// A word holds 8 for every up neighbour, the bytes of one bin of ln g: half the change
// of k.  With open boundaries bins are half as wide, and a word holds 16 for every up
// neighbour less 8 for every neighbour; a missing neighbour is a word of the border
// around the lattice, which nobody reads.
template <bool TRI>
struct LoneLane {
    uint32_t swap;                   // 16 for the lanes of the down site: their order in a ring record
    int32_t sign;                    // own word less the other's, as up less down
    uint32_t ahead;                  // all ones in the lanes of the step after the pending one
    uint32_t accept, reject;         // what the decision adds to this lane's word
    uint32_t next;                   // what becoming the pending step adds to it
    uint32_t both;                   // what an accepted step adds where nothing is pending
    uint32_t scale;                  // 0 for a lane without a neighbour
    uint32_t apart, touching;        // bias of a difference whose sites are not, are neighbours
    uint32_t s0, m0, e0, d0, w0;     // along one axis: shift, mask, coordinate at the edge, step, step at the edge
    uint32_t s1, m1, e1, d1, w1;     // along the other (triangular diagonals)

    __device__ __forceinline__ void setup(const Geo& g, int lane, uint32_t words, uint32_t spare)
    {
        const int z = g.shape == kShapeTriangular || g.shape == kShapeCubic ? 6 : 4;
        const bool open = g.shape == kShapeOpen;
        const uint32_t unit = open ? 16u : 8u;
        const int q = lane % z;
        const bool down = ((lane / z) & 1) != 0;
        swap = down ? 16u : 0u;
        sign = down ? -1 : 1;
        apart = kBias * kBoth;
        touching = (kBias + unit) * kBoth;
        const uint32_t delta = down ? unit : 0u - unit;    // the up site goes, the down site comes
        ahead = lane >= 2 * z && lane < 4 * z ? 0xFFFFFFFFu : 0u;
        next = ahead & (delta << 16);
        accept = ahead ? next : delta;
        reject = ahead ? next : 0u - (delta << 16);
        both = ahead ? 0u : delta * kBoth;
        const uint32_t e = (uint32_t)g.L - 1u;
        auto axis = [&](int ax, bool plus, uint32_t& s, uint32_t& mk, uint32_t& ed, uint32_t& d, uint32_t& w) {
            s = (uint32_t)(ax * g.cshift) + 2u;
            const uint32_t u = 1u << s;
            // the outermost coordinate is what is left of the address, base and all
            const bool outer = ax == (g.shape == kShapeCubic ? 2 : 1);
            mk = outer ? 0xFFFFFFFFu : g.cmask;
            ed = (plus ? e : 0u) + (outer ? words >> s : 0u);
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
        if (lane >= 4 * z) {
            scale = d1 = w1 = reject = 0u;
            accept = both = lane == 4 * z ? 1u : 0u;
            d0 = w0 = spare + 4u * (uint32_t)lane;
        }
    }

    // Address of the word of this lane's neighbour of the site at c.
    __device__ __forceinline__ uint32_t neighbour(uint32_t c) const
    {
        uint32_t n = (((c >> s0) & m0) == e0 ? w0 : d0) + c * scale;
        if constexpr (TRI) n += ((c >> s1) & m1) == e1 ? w1 : d1;
        return n;
    }
    __device__ __forceinline__ uint32_t bias(bool adjacent) const { return adjacent ? touching : apart; }
};

// A walker's state: the pending step (this lane's own site and the other one, the
// bin it proposes), the step after it, the list slots of the one after that.  Sites are
// the addresses of their words; xa, ta and u are the same in every lane.
struct Lone {
    uint32_t xa;            // address of the current bin
    uint32_t ta;            // address of the bin the pending step proposes
    int64_t u;              // ln g of the current bin
    uint32_t own, oth;      // pending step
    uint32_t own1, oth1;    // the step after it
    uint32_t nb;            // this lane's neighbour of its step
    uint32_t bias;          // of the next step's difference: kBias, and a unit more if its sites are neighbours
    uint2 slots;            // of the step after next: own, other
};

// One step: decide the pending one, evaluate the next, load the one after.
// `at`: the pending step's record in the ring, in this lane's order.  WAIT: the next
// step or the one after it shares a list slot with the pending one.  The loads come
// before the stores as far as they may: the compiler keeps their order, and a load
// that waits behind a store waits for the decision.
template <bool TRI, bool WAIT>
__device__ __forceinline__ void lone_step(Lone& w, const LoneLane<TRI>& L, uint32_t at, int64_t F)
{
    const int64_t gt = lds64(w.ta);
    const uint4 r = lds128(at);
    uint2 s1 = make_uint2(0u, 0u);
    if constexpr (WAIT) s1 = lds64u(at + 40u);
    bool p;
    auto decide = [&]() {
        p = gt <= w.u + (int64_t)(((uint64_t)r.y << 32) | r.x);
        w.xa = p ? w.ta : w.xa;
        w.u = (p ? gt : w.u) + F;
    };
    if constexpr (WAIT) {
        // what the next step finds in a slot it shares is known with the decision
        decide();
        const uint32_t no = p ? w.oth : w.own, nt = p ? w.own : w.oth;
        w.own1 = s1.x == r.z ? no : w.own1;
        w.oth1 = s1.y == r.w ? nt : w.oth1;
        reds(w.nb, (p ? L.accept : L.reject) & ~L.ahead);
        sts16(r.z, no);
        sts64(w.xa, w.u);
        __syncwarp();
    }
    const uint32_t wo = lds32(w.own1), wt = lds32(w.oth1);
    const uint32_t own2 = lds16(w.slots.x), oth2 = lds16(w.slots.y);
    w.slots = lds64u(at + 104u);
    __syncwarp();
    if constexpr (WAIT) {
        const uint32_t n1 = L.neighbour(w.own1);
        w.bias = L.bias(__any_sync(0xffffffffu, n1 == w.oth1));
        reds(n1, L.next);
    }
    // the change of k as bytes of ln g, in both halves
    const uint32_t d = (uint32_t)((int32_t)(wo - wt) * L.sign) + w.bias;
    // the lanes ahead take the step after next, the others the next; only the
    // former see whether its sites are neighbours
    const uint32_t nb = L.neighbour(L.ahead ? own2 : w.own1);
    const uint32_t bias = L.bias(__any_sync(0xffffffffu, nb == (oth2 & L.ahead)));
    if constexpr (!WAIT) {
        decide();
        sts64(w.xa, w.u);
        sts16(r.z, p ? w.oth : w.own);             // the lanes of either site write its list slot
        reds(w.nb, p ? L.accept : L.reject);       // the pending step is decided, the next is pending
    }
    // with the pending step rejected (WAIT: decided), or accepted
    w.ta = w.xa + __byte_perm(d, 0u, !WAIT && p ? 0x4432u : 0x4410u) - kBias;
    w.own = w.own1;
    w.oth = w.oth1;
    w.own1 = own2;
    w.oth1 = oth2;
    w.nb = nb;
    w.bias = bias;
    __syncwarp();
}

template <bool TRI, int K, bool WAIT>
__device__ __forceinline__ void lone_block(Lone& w, const LoneLane<TRI>& L, uint32_t& at, int64_t F)
{
#pragma unroll
    for (int q = 0; q < K; ++q) lone_step<TRI, WAIT>(w, L, at + 32u * q, F);
    at += 32u * K;
}

// One step where most would wait: decided, written back, and only then the next one
// evaluated.  Nothing is pending in the words (their halves are the same), so an
// accepted step needs one reduction and the next but one is not looked at ahead.
template <bool TRI>
__device__ __forceinline__ void dense_step(Lone& w, const LoneLane<TRI>& L, uint32_t at, int64_t F)
{
    const int64_t gt = lds64(w.ta);
    const uint4 r = lds128(at);
    const uint2 s1 = lds64u(at + 40u);
    const bool p = gt <= w.u + (int64_t)(((uint64_t)r.y << 32) | r.x);
    // what the next step finds in a slot it shares is known with the decision
    const uint32_t no = p ? w.oth : w.own, nt = p ? w.own : w.oth;
    w.own = s1.x == r.z ? no : w.own1;
    w.oth = s1.y == r.w ? nt : w.oth1;
    reds(w.nb, p ? L.both : 0u);
    w.xa = p ? w.ta : w.xa;
    w.u = (p ? gt : w.u) + F;
    sts16(r.z, no);
    sts64(w.xa, w.u);
    __syncwarp();
    const uint32_t wo = lds32(w.own), wt = lds32(w.oth);
    w.own1 = lds16(w.slots.x);
    w.oth1 = lds16(w.slots.y);
    w.slots = lds64u(at + 104u);
    __syncwarp();
    w.nb = L.neighbour(w.own);
    const uint32_t bias = L.bias(__any_sync(0xffffffffu, w.nb == w.oth));
    const uint32_t d = (uint32_t)((int32_t)(wo - wt) * L.sign) + bias;
    w.ta = w.xa + (d & 0xFFFFu) - kBias;
}

// Between the two ways: the pending step's changes leave the words' high halves, or
// enter them (and the step after it is looked at).
template <bool TRI>
__device__ __forceinline__ void to_dense(Lone& w, const LoneLane<TRI>& L)
{
    reds(w.nb, L.reject & ~L.ahead);
    __syncwarp();
}
template <bool TRI>
__device__ __forceinline__ void from_dense(Lone& w, const LoneLane<TRI>& L)
{
    const uint32_t n1 = L.neighbour(w.own1);
    w.bias = L.bias(__any_sync(0xffffffffu, n1 == w.oth1));
    reds(w.nb, 0u - (L.reject & ~L.ahead));
    w.nb = L.ahead ? n1 : w.nb;
    __syncwarp();
}

// Take n <= 32 steps, from the record at `at` on; waits: their wait flags.  The end of
// a loop's body costs ~75 cycles here (the compiler lets the loops of a kernel yield
// whose warps part before a barrier), and so do the turns between two kinds of step.
// So steps go in blocks: 64x64, l = 2048, takes 182 cycles a step one at a time, 143
// two, 115 four, 106 eight.  A flagged step among others costs ~350 cycles; from
// three in a batch on (few up spins, a tiny lattice) all steps go the dense way.
constexpr int kToDense = 3, kFromDense = 1;

template <bool TRI>
__device__ __forceinline__ void lone_run(Lone& w, const LoneLane<TRI>& L, bool& dense, uint32_t at, int n, uint32_t waits,
                                         int64_t F)
{
    const int flags = __popc(waits);
    if (dense ? flags <= kFromDense : flags >= kToDense) {
        dense = !dense;
        if (dense) to_dense<TRI>(w, L);
        else from_dense<TRI>(w, L);
    }
    if (dense) {
#pragma unroll 1
        for (; n >= 8; n -= 8) {
#pragma unroll
            for (int q = 0; q < 8; ++q) dense_step<TRI>(w, L, at + 32u * q, F);
            at += 256u;
        }
#pragma unroll 1
        for (; n > 0; --n) {
            dense_step<TRI>(w, L, at, F);
            at += 32u;
        }
        return;
    }
    for (;;) {
        const int clear = waits ? __ffs((int)waits) - 1 : 32;      // steps before the next flag
        int k = clear < n ? clear : n;
        n -= k;
        waits = clear < 31 ? waits >> (clear + 1) : 0u;
#pragma unroll 1
        for (; k >= 8; k -= 8) lone_block<TRI, 8, false>(w, L, at, F);
        if (k & 4) lone_block<TRI, 4, false>(w, L, at, F);
        if (k & 2) lone_block<TRI, 2, false>(w, L, at, F);
        if (k & 1) lone_block<TRI, 1, false>(w, L, at, F);
        if (n == 0) break;
        lone_block<TRI, 1, true>(w, L, at, F);
        n -= 1;
        if (n == 0) break;
    }
}

// The drawing warp: batches of 32 steps from t on, until the walker is done.
template <bool DET>
__device__ __forceinline__ void lone_draw(const WalkArgs& A, int64_t t, int ell, uint4* ring, uint32_t* waits, uint32_t perm,
                                          const volatile int32_t* done, int lane)
{
    const uint2 key = make_uint2((uint32_t)ell, A.seed);
    const uint32_t nd = (uint32_t)(A.g.N - ell);
    uint32_t prev_a = 0xFFFFFFFFu, prev_b = 0xFFFFFFFFu;      // slots of the batch before
    auto fill = [&](uint32_t k) {
        const Draw d = draw_step<DET>((uint64_t)t + 32u * (uint64_t)k + (uint64_t)lane, key, (uint32_t)ell, nd, A);
        // a step waits for its decision when the next one or the one after it draws
        // one of its slots; here: this step and the two before it, of this batch or
        // of the end of the last
        uint32_t a[3] = {d.a, 0u, 0u}, b[3] = {d.b, 0u, 0u};
#pragma unroll
        for (int back = 1; back <= 2; ++back) {
            const uint32_t a0 = __shfl_up_sync(0xffffffffu, d.a, back), b0 = __shfl_up_sync(0xffffffffu, d.b, back);
            const uint32_t a1 = __shfl_sync(0xffffffffu, prev_a, (lane + 32 - back) & 31);
            const uint32_t b1 = __shfl_sync(0xffffffffu, prev_b, (lane + 32 - back) & 31);
            a[back] = lane >= back ? a0 : a1;
            b[back] = lane >= back ? b0 : b1;
        }
        const bool wait = a[0] == a[2] || b[0] == b[2] || a[1] == a[2] || b[1] == b[2];
        prev_a = d.a;
        prev_b = d.b;
        const uint32_t sa = perm + 2u * d.a, sb = perm + 2u * ((uint32_t)ell + d.b);
        const uint4 r = make_uint4((uint32_t)d.dmax, (uint32_t)((uint64_t)d.dmax >> 32), sa, sb);
        const uint4 q = make_uint4(r.x, r.y, sb, sa);
        const uint32_t at = (32u * k + (uint32_t)lane) & (kRing - 1);
        ring[2u * at] = r;
        ring[2u * at + 1u] = q;
        if (at < kRingMore) {
            ring[2u * (kRing + at)] = r;
            ring[2u * (kRing + at) + 1u] = q;
        }
        // the flag is for the step two before
        const uint32_t flags = __ballot_sync(0xffffffffu, wait);
        if (lane == 0) waits[k & 3u] = flags;
    };
    fill(0);
    fill(1);
    lone_barrier();
    for (uint32_t k = 2;; ++k) {
        fill(k);
        lone_barrier();
        if (*done) break;
    }
}

// The walking warp: line `li` for up to A.slice_moves moves (or to its budget, or
// to convergence); the bookkeeping between steps as in walk_line.
template <bool TRI>
__device__ __forceinline__ void lone_walk(const WalkArgs& A, int li, int m, uint8_t* sm, const uint4* ring, const uint32_t* waits,
                                          uint32_t words, uint32_t* spare, volatile int32_t* done)
{
    const bool open = A.g.shape == kShapeOpen;
    const int ks = open ? 0 : 1;
    const int zb = open ? 8 : A.g.shape == kShapeTriangular || A.g.shape == kShapeCubic ? 6 : 4;    // Coord::zbin
    const int kMargin = 32 * zb;         // a run of steps stays inside the window
    constexpr unsigned all = 0xffffffffu;
    const LineDesc D = A.desc[li];
    LineState* P = A.st + li;
    int64_t t = P->t, F = P->F, stage = P->stage, accepts = P->accepts;
    int64_t t_stage = P->t_stage, status = P->status, checks = P->checks;
    const int64_t t0 = t, batches = P->batches;
    const int nbins = D.nbins;
    int64_t* lng = A.lng + D.bin_off;
    hist_t* hist = A.hist + D.bin_off;
    int64_t end = t + A.slice_moves;
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
    LoneLane<TRI> L;
    L.setup(A.g, m, words, (uint32_t)__cvta_generic_to_shared(spare));
    const uint32_t ring_at = (uint32_t)__cvta_generic_to_shared(ring) + L.swap;
    uint32_t* counter = spare + (zb == 6 ? 24 : 16);      // the first lane past the neighbours
    Lone w{};
    w.xa = wa + 8u * (uint32_t)(bc - wb);
    w.u = wl[bc - wb];
    if (m == 0) *counter = 0u;
    lone_barrier();               // the first two batches are drawn
    if (t < end) {
        // the first step is pending, the second loaded, the third's slots at hand
        uint2 sl = lds64u(ring_at + 8u);
        w.own = lds16(sl.x);
        w.oth = lds16(sl.y);
        sl = lds64u(ring_at + 40u);
        w.own1 = lds16(sl.x);
        w.oth1 = lds16(sl.y);
        w.slots = lds64u(ring_at + 72u);
        const uint32_t n0 = L.neighbour(w.own), n1 = L.neighbour(w.own1);
        const uint32_t d = (uint32_t)((int32_t)(lds32(w.own) - lds32(w.oth)) * L.sign) +
                           L.bias(__any_sync(all, n0 == w.oth));
        w.ta = w.xa + (d & 0xFFFFu) - kBias;
        w.bias = L.bias(__any_sync(all, n1 == w.oth1));
        w.nb = L.ahead ? n1 : n0;
        __syncwarp(all);
        reds(n0, L.next);
    }
    __syncwarp(all);

    bool dense = false;
    while (t < end && !stop) {
        const int64_t next_check = (t / C + 1) * C;
        const int64_t seg_end = next_check < end ? next_check : end;
        while (t < seg_end) {
            const uint32_t pos = (uint32_t)(t - t0), k = pos >> 5;
            const int batch = 32 - (int)(pos & 31u);
            const int n = seg_end - t < batch ? (int)(seg_end - t) : batch;
            const uint32_t lo = wb > 0 ? wa + 8u * kMargin : wa;
            const uint32_t hi = wa + 8u * (uint32_t)(wn - 1 - (wb + wn < nbins ? kMargin : 0));
            const uint32_t wm = (waits[k & 3u] >> 2) | (waits[(k + 1u) & 3u] << 30);
            lone_run<TRI>(w, L, dense, ring_at + 32u * (pos & (kRing - 1)), n, wm >> (pos & 31u), F);
            __syncwarp(all);
            const uint32_t xa = w.xa;
            bc = wb + ((int)(xa - wa) >> 3);
            if (xa < wa || bc - wb >= wn) {
                stop = 4;                  // never: a run from inside the margins stays inside
                break;
            }
            t += n;
            if ((pos >> 24) != ((uint32_t)(t - t0) >> 24)) {      // long before the counter overflows
                accepts += *counter;
                __syncwarp(all);
                if (m == 0) *counter = 0u;
                __syncwarp(all);
            }
            if (xa < lo || xa > hi) {
                // re-centre the window
                if (__any_sync(all, window_store<32>(wl, lng, hist, wb, wn, m, F))) stop = 2;
                __syncwarp(all);
                wb = window_base(bc, nbins, A.win_bins);
                window_load<32>(wl, lng, wb, wn, m);
                __syncwarp(all);
                const uint32_t to = wa + 8u * (uint32_t)(bc - wb);
                w.ta += to - xa;
                w.xa += to - xa;
            }
            if (((uint32_t)(t - t0) & 31u) == 0u) lone_barrier();
            if (stop) break;
        }
        if (stop) break;

        if (t == next_check) {
            // window -> global, then test flatness over the line
            __syncwarp(all);
            if (__ballot_sync(all, window_store<32>(wl, lng, hist, wb, wn, m, F))) {
                stop = 2;
                break;
            }
            __syncwarp(all);
            checks += 1;
            const bool flat = group_flat<32>(hist, nbins, m, all, A.flat_pm);
            const bool again = !flat && A.same_f_resets > 0 && (t - t_stage) / C <= A.same_f_resets;
            if (flat || again) {
                group_stage_step<32>(lng, hist, nbins, m, all);
                window_load<32>(wl, lng, wb, wn, m);
                __syncwarp(all);
                w.u = wl[bc - wb];
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
    if (stop == 2) status = 2;
    if (stop == 4) status = 3;
    if (m == 0) {
        P->k = (int64_t)bc << ks;
        P->t = t;
        P->F = F;
        P->stage = stage;
        P->accepts = accepts + *counter;
        P->t_stage = t_stage;
        P->status = status;
        P->checks = checks;
        P->batches = batches + (t - t0 + 31) / 32;
        if (stop == 1) atomicOr(A.flags, 1);
        if (stop == 3) atomicOr(A.flags, 2);
        if (stop == 2) atomicOr(A.flags, 4);
        if (stop == 4) atomicOr(A.flags, 8);
        *done = 1;
    }
    __syncwarp(all);
    lone_barrier();
}

// One block per line: shared memory holds the words of the sites (and one more), the
// list, the window, the ring of draws.
template <bool TRI, bool DET>
__global__ void __launch_bounds__(kLoneThreads) lone_kernel(const WalkArgs A)
{
    extern __shared__ __align__(16) uint8_t smem[];
    const int th = threadIdx.x, warp = th >> 5, lane = th & 31;
    const uint32_t base = (uint32_t)__cvta_generic_to_shared(smem);
    // the words start at a whole row (cubic: plane) of addresses
    const uint32_t row = 4u << (A.g.shape == kShapeCubic ? 2 * A.g.cshift : A.g.cshift);
    const uint32_t words_at = (base + row - 1u) / row * row;
    uint32_t* words = reinterpret_cast<uint32_t*>(smem + (words_at - base));
    uint16_t* perm = reinterpret_cast<uint16_t*>(smem + A.off_perm);
    uint4* ring = reinterpret_cast<uint4*>(smem + A.off_rec);
    uint32_t* waits = reinterpret_cast<uint32_t*>(ring + 2 * (kRing + kRingMore));
    int32_t* ctl = reinterpret_cast<int32_t*>(waits + 4);         // the line; the walker is done; who walks
    if (th == 0) {
        // The SM deals its warps out to four schedulers in order of their slots: were
        // it always the first warp of a block that walks, all walkers would share two
        // of them.  Any choice is right; this one spreads them over all four.
        uint32_t slot;
        asm volatile("mov.u32 %0, %%warpid;" : "=r"(slot));
        ctl[2] = (int32_t)((slot >> 2) & 1u);
    }
    uint32_t* spare = reinterpret_cast<uint32_t*>(ctl + 4);
    const int N = A.g.N, pstride = A.pstride;
    for (;;) {
        if (th == 0) {
            const int qi = atomicAdd(A.qnext, 1);
            ctl[0] = qi < A.nqueue ? A.order[qi] : -1;
            ctl[1] = 0;
        }
        __syncthreads();
        const int li = ctl[0];
        if (li < 0) break;
        if (A.st[li].status == 0) {
            uint16_t* gperm = reinterpret_cast<uint16_t*>(A.perm) + (size_t)li * pstride;
            uint32_t* gsp = A.spins + (size_t)li * A.g.W;
            for (int n = th; n < N; n += kLoneThreads) {
                perm[n] = (uint16_t)(words_at + 4u * site_code(A.g, gperm[n]));
                const uint32_t u = A.g.shape == kShapeTriangular ? site_word<kTriangular>(A.g, gsp, (uint32_t)n)
                                   : A.g.shape == kShapeCubic    ? site_word<kCubic>(A.g, gsp, (uint32_t)n)
                                   : A.g.shape == kShapeOpen     ? site_word<kSquareOpen>(A.g, gsp, (uint32_t)n)
                                                                 : site_word<kSquare>(A.g, gsp, (uint32_t)n);
                words[site_code(A.g, (uint32_t)n)] = u * kBoth;
            }
            const int64_t t = A.st[li].t;
            const int ell = A.desc[li].ell;
            __syncthreads();
            if (warp == ctl[2])
                lone_walk<TRI>(A, li, lane, smem, ring, waits, words_at, spare, ctl + 1);
            else
                lone_draw<DET>(A, t, ell, ring, waits, (uint32_t)__cvta_generic_to_shared(perm), ctl + 1, lane);
            __syncthreads();
            // the list, and from it the spins
            for (int x = th; x * 32 < N; x += kLoneThreads) words[x] = 0u;
            __syncthreads();
            for (int n = th; n < N; n += kLoneThreads) {
                const uint32_t s = code_site(A.g, (perm[n] - words_at) >> 2);
                gperm[n] = (uint16_t)s;
                if (n < ell) atomicOr(&words[s >> 5], 1u << (s & 31u));
            }
            __syncthreads();
            for (int x = th; x * 32 < N; x += kLoneThreads) gsp[x] = words[x];
        }
        __syncthreads();
    }
}

}  // namespace wl
