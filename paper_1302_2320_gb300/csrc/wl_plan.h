// wl_plan.h -- how the walkers of a launch share the GPU: the slots of shared memory of
// the two walkers (wl_lone.cuh, wl_walk.cuh) and the choice between them.  Host code
// without CUDA, so that its choices can be checked without a GPU; wl_api.cu supplies the
// device's limits.
#pragma once

#include <algorithm>
#include <cstddef>
#include <cstdint>

namespace wl {

// kSquareP2: the square lattice when L is a power of two (coordinates by
// shift and mask); the same lattice and bond set as kSquare.
// kSquareOpen: the square lattice with open boundaries (sites on an edge have
// fewer neighbours; k takes every value, so bins have step 1).
enum LatticeType : int { kSquare = 0, kTriangular = 1, kCubic = 2, kSquareP2 = 3, kSquareOpen = 4 };

// A lattice at run time, whatever its kernel specialisation.
enum LatticeShape : int { kShapeSquare = 0, kShapeTriangular = 1, kShapeCubic = 2, kShapeOpen = 3 };

constexpr int kStepBytes = 40;     // shared bytes of a lane's step record (Steps in wl_walk.cuh)
constexpr uint32_t kLow = 1024u;   // address at which a block's shared memory starts (wl_lone.cuh): behind the system's share

namespace rt {

// A walker's slot of shared memory.
struct Slot {
    int bytes = 0, off_perm = 0, off_sites = 0, off_win = 0, off_rec = 0;
    int win = 0;                 // bins of the ln g window
    int owner_mask = 0;
    bool stage_sites = false, stage_perm = false;
    int lone = 0;            // a block per line: bytes of a site's word; else 0
};

// Launch shape of the persistent form for S lanes per walker.
struct Shape {
    unsigned grid = 0, block = 0;
    size_t smem = 0;
    Slot slot;
};

// What the shape of a launch depends on.
struct ShapeKey {
    int lattice;         // kernel specialisation (LatticeType)
    int S;               // lanes per walker
    bool det, idx16;
    int L, N, pstride;
    int max_bins;        // bins of the largest line
    int lines;           // walkers wanted at once
    bool lone;           // few lines may get a block each (wl_lone.cuh)
};

// The limits of a device: SMs, and shared memory of a block, of an SM, and kept back by
// the system in every block.
struct Gpu {
    int sms, per_block, per_sm, reserved;
};

// Where running lines outnumber the blocks of a block per line, they take turns, so that
// all blocks have work until the end of the slice and not the last round's few (2^18 moves
// each, 1569 lines of 56x56 on 1520 blocks: 37.7 -> 26.7 ms; 2049 lines of 64x64 on 1520:
// 40.4 -> 33.2).  Turns of 2^14 moves and more: loading and storing a line takes ~50 us,
// a turn 1.3 ms; one turn where the moves of a slice would make turns of a second.  Lines
// that are done need no block: late in a walk to ln f_min one turn is enough.
inline int line_turns(const Shape& sh, int64_t running, int64_t moves)
{
    if (!sh.slot.lone || running <= (int64_t)sh.grid || moves > (1 << 26)) return 1;
    return (int)std::max<int64_t>(1, std::min<int64_t>(8, moves >> 14));
}

inline size_t align16(size_t x) { return (x + 15) & ~(size_t)15; }

// A walker's slot: the list (staged or not), the sites, the window, the step
// records.  The window is what is left of `room` bytes, up to the whole line; the
// chain loads ln g before it knows that a step is out of date, a few bins off at most:
// a guard on both sides keeps that inside the slot.
inline bool plan_slot(const ShapeKey& k, bool sites, bool perm, size_t room, int least_win, Slot* o)
{
    constexpr int kGuard = 8 * 8 * (12 + 1);      // kSub steps of the largest bin step, in bytes
    constexpr int kOwners = 4096;
    const int min_win = std::min(k.max_bins, least_win);
    Slot s;
    size_t at = perm ? (size_t)k.pstride * (k.idx16 ? 2 : 4) : 0;
    s.stage_perm = perm;
    s.stage_sites = sites;
    s.off_sites = (int)at;
    s.owner_mask = kOwners - 1;
    at += sites ? ((size_t)k.N + 31) / 32 * 32 : (size_t)kOwners;
    at = std::max<size_t>(align16(at), kGuard);
    s.off_win = (int)at;
    const size_t after = std::max<size_t>(align16((size_t)k.S * kStepBytes), kGuard);
    if (at + (size_t)min_win * 8 + 16 + after > room) return false;
    s.win = (int)std::min<size_t>((size_t)k.max_bins, (room - 16 - at - after) / 8);
    at += align16((size_t)s.win * 8);
    s.off_rec = (int)at;
    s.bytes = (int)align16(at + after);
    *o = s;
    return true;
}

// The slot of a line with a block of its own (wl_lone.cuh): the words of the sites
// by code, the list, the window, the ring.  The window needs no guard: a step is
// evaluated from the state it is taken from, and every state is a line's own, by the
// library's initialisation or by the exact check of a caller's (check_state_kernel).
inline bool plan_lone(const ShapeKey& k, int word, size_t room, Slot* o)
{
    if (!k.idx16) return false;
    const bool open = k.lattice == kSquareOpen;      // with a border around it
    size_t stride = 1;
    while (stride < (size_t)k.L + (open ? 1 : 0)) stride <<= 1;
    const size_t codes = (k.lattice == kCubic ? stride : 1) * stride * ((size_t)k.L + (open ? 2 : 0));
    if (word * codes > 65536) return false;          // a list entry holds an address
    // two margins of 16 steps of the largest bin step, and 64 bins to walk between them
    const int zb = k.lattice == kSquareOpen ? 8 : k.lattice == kTriangular || k.lattice == kCubic ? 6 : 4;
    const int min_win = std::min(k.max_bins, 32 * zb + 64);
    Slot s;
    s.lone = word;
    size_t at = align16(word * codes);
    s.off_perm = (int)at;
    at += (size_t)k.pstride * 2;
    s.off_win = (int)at;
    const size_t ring = (96 + 3) * 32 + 16 + 128;   // the draws, control words, spare words
    if (at + (size_t)min_win * 8 + 16 + ring > room) return false;
    s.win = (int)std::min<size_t>((size_t)k.max_bins, (room - 16 - at - ring) / 8);
    at += align16((size_t)s.win * 8);
    s.off_rec = (int)at;
    s.bytes = (int)(at + ring);
    *o = s;
    return true;
}

// Cycles a move takes its walker (GB300), for the choice between shapes.
// A block per line (wl_lone.cuh), words of 4 bytes or of one: 119 and 126 with up to 4 on
// an SM, one for each scheduler.  With more on an SM a move alone takes 153 and 159 (5 or
// 6), 162 and 168 (7 or 8), 197 (9 or 10, in turns; 64x64).  In a whole surface the loads
// of lines, checks and windows weigh as well, and more of them hide more of that: with 4
// and 5 on an SM 112x112 takes 163 and 173 cycles a move.  kLoneCrowd is what ranks whole
// surfaces rightly: the ratios of moves alone (1.29, 1.36, 1.58) in its place choose 4 and
// not 5 on an SM at 112x112 (26.6 and not 22.7 ms for 2^15 moves) and cubic 20^3 (17.0 and
// 14.3), and 10 and not 8 at 56x56 (28.2 and 27.2 ms, 2^18).
// Rounds of a block per line are lines / blocks as they are, also where lines take no
// turns: the lines of the last round have an SM to fewer, and are faster.  Counted whole
// they gain 3 % at 64x64 (a continuation without allocation, 7 and not 10 on an SM) and
// lose 5 % at 56x56, 7 % at triangular 58x58 and 18 % at cubic 20^3.
// Batches (wl_walk.cuh): 191 with 7 on an SM and the lists staged (96x96), 272 with 16
// on an SM and the lists in global memory (96x96) or 12 and staged (64x64); and what a
// surface's lines of few up spins take longer, whose batches keep running into
// themselves.
// Where the line between the two lies, block per line and batches, ms for 2^15 moves of
// all lines: square 112x112 21.7 and 24.4, 116x116 27.4 and 24.4, 128x128 33.6 and 23.0;
// triangular 112x112 23.2 and 24.6, 120x120 30.3 and 26.7; cubic 23^3 24.9 and 26.5, 24^3
// 37.2 and 26.1.  With production acceptance a block per line is the same within 1 % and
// batches take from 4 % more to 13 % less there (116x116: 29.9).  Open boundaries cross
// earlier, between 100x100 (17.1 and 20.1) and 108x108 (20.6 and 18.4; 112x112: 25.8 and
// 17.3), which the figures below, those of square lattices, do not know.
inline constexpr double kLoneCycles[2] = {119.0, 126.0}, kLoneCrowd[4] = {1.0, 1.2, 1.27, 1.58}, kBatchIssue = 17.0, kBatchSlowest = 600.0;

// Either a block of two warps per line, or one warp per block with 32 / S walkers,
// whichever takes its walkers less time for a move of all of them.  The shape spreads the
// walkers over the SMs and gives each the shared memory its share of an SM leaves.  When
// walkers in batches do not all fit at once with their lists staged, the lists stay in
// global memory if that takes fewer rounds: they are read once per batch, so they cost a
// batch one L2 latency, while a round more costs a whole walk.
//
// resident(slot, smem, threads): how many blocks of the kernel that the slot selects an SM
// holds at once, negative if that cannot be told, which ends the planning.
enum class Planned { ok, none_fits, unknown };

template <class Resident>
Planned plan_shape(const ShapeKey& k, const Gpu& gpu, Resident&& resident, Shape* sh)
{
    const int sms = gpu.sms, per_block = gpu.per_block, per_sm = gpu.per_sm, reserved = gpu.reserved;
    const int groups = 32 / k.S;
    const int need = (k.lines + groups - 1) / groups;       // blocks wanted
    const int want = std::min((need + sms - 1) / sms, 32);  // per SM
    auto room_of = [&](int blocks) {   // bytes of a block with this many on an SM
        const int b = std::min(per_block, per_sm / blocks - reserved - 128) / 128 * 128;
        return b > 0 ? (size_t)b : (size_t)0;
    };
    double best = 0.0;
    int best_blocks = 0;
    // a block per line: as many as fit, each with its share of the shared memory; words of
    // a byte where that makes room for enough more of them (wl_lone.cuh)
    for (int word : {4, 1}) {
        if (!k.lone || gpu.reserved != (int)kLow) break;      // its addresses count from kLow
        auto cycles = [&](int on_sm) {
            return kLoneCycles[word == 1] * kLoneCrowd[std::min(3, std::max(0, (on_sm - 3) / 2))];
        };
        const int want = std::min((k.lines + sms - 1) / sms, 32);
        for (int b = want; b > 0; --b) {
            Slot slot;
            if (!plan_lone(k, word, room_of(b), &slot)) continue;
            const int bps = resident(slot, (size_t)slot.bytes, 64);
            if (bps < 0) return Planned::unknown;
            if (bps < b) continue;
            // rounds as a fraction (above)
            const double cost = std::max(1.0, (double)k.lines / (sms * b)) * cycles(b);
            if (best_blocks != 0 && cost >= best) continue;
            best = cost;
            best_blocks = b;
            sh->slot = slot;
            sh->grid = (unsigned)std::min(k.lines, sms * b);
            sh->block = 64;
            sh->smem = slot.bytes;
        }
    }
    auto room = [&](int blocks) {      // bytes per walker with this many blocks on an SM
        const int b = std::min(per_block, per_sm / blocks - reserved) / 128 * 128;
        return b > 0 ? (size_t)b / groups / 16 * 16 : (size_t)0;
    };
    struct Mode {
        bool sites, perm;
        double cycles;                 // a lone walker's cycles per move, to weigh rounds
    };
    const Mode modes[3] = {{true, true, 190.0}, {true, false, 200.0}, {false, false, 250.0}};
    // Windows of 384 bins where there are six neighbours, 256 otherwise; with one lane a
    // walker, of which 32 share a block, 384 may leave room for none (triangular from
    // 58x58 on, cubic from 15^3): then 256, still more than twice the two margins of 56.
    const bool six = k.lattice == kTriangular || k.lattice == kCubic;
    bool fits = false;
    for (const int least_win : {six ? 384 : 256, 256}) {
        if (fits) break;
        for (const Mode& m : modes) {
            if (m.sites && !k.idx16) continue;
            int b = want;
            Slot slot;
            while (b > 0 && !plan_slot(k, m.sites, m.perm, room(b), least_win, &slot)) --b;
            if (b == 0) continue;
            const int bps = resident(slot, (size_t)groups * slot.bytes, 32);
            if (bps < 0) return Planned::unknown;
            b = std::min(b, bps);
            if (b < 1) continue;
            fits = true;
            const double rounds = (double)((need + sms * b - 1) / (sms * b));
            const double cost = rounds * std::max(m.cycles, kBatchIssue * b * groups) + kBatchSlowest;
            if (best_blocks == 0 || cost < best) {
                if (!plan_slot(k, m.sites, m.perm, room(b), least_win, &slot)) continue;
                best = cost;
                best_blocks = b;
                sh->slot = slot;
                sh->grid = (unsigned)std::max(1, std::min(need, sms * b));
                sh->block = 32;
                sh->smem = (size_t)groups * slot.bytes;
            }
        }
    }
    return best_blocks ? Planned::ok : Planned::none_fits;
}

}  // namespace rt
}  // namespace wl
