// X-engine on the 5th-generation tensor cores (tcgen05, sm_103a).
//
// Paper: Sec. 1 (cross-multiply every pair of antennas per channel and
// accumulate), Sec. 4 (the cross-multiply dominates the load; the paper
// converts the FFT output to a narrower type with prescaling before it).
//
// For one channel k the spectra of a pass form the real matrix A whose rows
// are the real and imaginary parts of every antenna (spectra along the
// contraction axis); the Gram matrix G = A A^T holds every product the
// visibilities need.  Antennas come in blocks of 64 (128 rows at most); for
// a pair of blocks (b1 <= b2) with local antennas i' < nb1 and j' < nb2
// (block rows 2 i' = Re, 2 i' + 1 = Im:
//   Re V_ij = G[2i'][2j'] + G[2i'+1][2j'+1],  Im V_ij = G[2i'+1][2j'] - G[2i'][2j'+1].)
// Each block pair is a dense contraction D[128 x Nn] += A_b1[128 x 16|32] *
// A_b2^T on the tensor cores, operands loaded by TMA (rows past the antenna
// count are zero-filled), FP32 accumulators in TMEM.  With several blocks a
// pair of CTAs takes two blocks against two at a time.  For a diagonal pair
// both operands are the same shared-memory tile.
//
// Precisions (operands in shared memory, K-major; FP16 tiles of 32 spectra in
// 64-byte rows with the 64-byte swizzle, FP8 tiles of 128 in 128-byte rows
// with the 128-byte swizzle; rows 2 i' and 2 i' + 1 of a block are the real
// and imaginary parts of its antenna i'):
//   mode 0 (FP32-accurate): two FP16 planes sigma_i x = hi + lo, sigma_i a
//           power of two per antenna.  Diagonal pairs issue Dhh += hi hi^T
//           and Dhl += hi lo^T and form G = Dhh + Dhl + Dhl^T; off-diagonal
//           pairs issue hi hi^T, hi lo^T and lo hi^T into one accumulator
//           (lo lo^T is below 2^-22); V_ij is descaled by 1/(sigma_i sigma_j).
//   mode 1: one FP16 plane (pre-scaled per antenna and channel).
//   mode 2: one FP8-E4M3 plane (pre-scaled), kind::f8f6f4.
//
// One launch may serve several correlators ("modes") of different N and K
// that share the precision: work items (mode, channel, block pair or group,
// range of spectra) are enumerated mode by mode and dealt round-robin to
// persistent CTAs (several blocks: CTA pairs) of 10 warps:
//   warp 0    TMA producer                -> stage ring (full/empty mbarriers)
//   warp 1    TMEM allocator + MMA issuer -> two TMEM accumulator sets
//   warps 2-9 epilogue: TMEM -> registers, summed over windows -> G in shared
//             memory -> V -> FP64 accumulator (or FP32 partials)
// What the MMA warp does per stage sets the pace, not the tensor pipe: a loop
// of one lane spent ~1500 clocks on a stage of 8 MMAs (128 clocks each),
// ~100 an MMA, on descriptors built for each and copied to uniform registers,
// and ~130 a wait.  Now the warp runs whole, one elected lane issues, and a
// descriptor is the stage's plus a constant: 130 antennas, K = 2048, 1500
// spectra FP16 418 -> 352 us, N = 11, K = 4096, 1024 spectra 94 -> 63 us.
// The tensor core's FP32 accumulation into TMEM is biased (it loses about one
// unit in the last place per accumulate, always toward zero), so TMEM only
// accumulates one window of W spectra; the epilogue adds the windows with
// round-to-nearest FP32 arithmetic.  The two accumulator sets let the
// epilogue drain window n while the MMAs fill window n+1.
// Every mbarrier wait is bounded by a global-timer deadline; on expiry the
// kernel records a status code, drains its own copies and MMAs, frees TMEM
// and returns.
#include "xengine_tc.h"
#include "scales.cuh"
#include "tc_ptx.cuh"

#include <cuda.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <cstdio>
#include <vector>

namespace gbcorr {
namespace {

using namespace tc;

constexpr int kTcThreads = 320;     // producer, MMA, 8 epilogue warps
constexpr int kRows = 128;          // MMA M = TMA box rows = one antenna block
constexpr uint32_t kTmemCols = 512; // two accumulator sets of 256 columns
constexpr int kVB = 2;              // accumulator loads in flight per epilogue thread
constexpr int kVCols = 16;          // baselines per antenna in one staging round
constexpr int kVRow = kVCols + 1;   // float2 per staging row (+1: bank offset)

struct TcModeArgs {
    int N, C, P;
    int nblk, npairs;         // antenna blocks of 64 and the work groups of a channel
    int n_split;
    int item_base, n_items;   // items: block pair fastest, then channel, then split
    int64_t S_pad, S_item;
    int64_t tiles;            // k-tiles of the pass (balanced deal)
    int cap_tiles;            // k-tiles of a workspace plane (the lo plane's first tile)
    uint32_t box_bytes;       // bytes one TMA box of this mode lands in shared memory
    int64_t unit_base;        // first work unit of this mode (balanced deal)
    float2* partial;          // [n_split][C][P] FP32 partials (n_split > 1)
    double2* acc;             // [C][P] FP64 accumulator
    int* ticket;              // [C] arrival counters of a single block (n_split > 1), zero between launches
    const float* scale;       // [N][C] pre-cast scales (modes 1, 2)
    const float* split;       // [N] two-plane pre-scales sigma_i (mode 0)
    int assign;               // acc is known to hold zeros: store instead of adding
};

struct TcArgs {
    CUtensorMap tmap[kMaxTcModes];
    TcModeArgs md[kMaxTcModes];
    int n_modes, total_items;
    int stages, KT, W;
    int kt_shift;             // log2(KT): the single-lane roles avoid 64-bit division
    int atoms;                // k-tiles of KT spectra per pipeline stage
    int row_bytes;            // bytes of one tile row: 64 (FP16 modes) or 128 (FP8)
    int gs_floats;            // epilogue G buffer (largest 2nb x (2nb + 1) of the modes; FP32 mode + 2 kRows)
    int slot_rows;            // rows of one operand tile slot in shared memory (<= 128)
    int* status;
    unsigned long long timeout_ns;
    int withhold;             // test hook: CTA 0 does not load its first k-tile
    int balanced;             // 1: contiguous deal of weighted k-tiles; 0: round-robin items
    int64_t units;            // total work units of the balanced deal
    int u32;                  // units times CTAs fit 32 bits: cheap divisions
};

struct Item {
    int m, k, b1, b2, nbB, sp, pr;
};

// One CTA's share of an item: k-tiles [s_beg, s_end) of the pass, the
// item's slot among the CTAs sharing it and their number.
struct Piece {
    Item itm;
    int64_t s_beg, s_end;
    int slot, nslots;
};

// Work groups of a channel.  One antenna block (N <= 64): the single
// diagonal block pair.  Several blocks: two blocks (b1, b1 + 1; the A rows of
// the two CTAs of a pair) against two blocks (b2, b2 + 1; half of the B rows
// in each CTA), b1 <= b2, both even: 4 blocks (N = 256 antennas) take 3
// groups.  nbB is the number of B blocks that exist.
__host__ __device__ __forceinline__ int groups_of(int nblk) {
    const int nb2 = (nblk + 1) >> 1;
    return nb2 * (nb2 + 1) / 2;
}

__host__ __device__ __forceinline__ void group_decode(int gi, int nblk, int& b1, int& b2, int& nbB) {
    const int nb2 = (nblk + 1) >> 1;
    int r = 0;
    while (gi >= nb2 - r) {
        gi -= nb2 - r;
        ++r;
    }
    b1 = 2 * r;
    b2 = 2 * (r + gi);
    nbB = nblk - b2 < 2 ? nblk - b2 : 2;
}

// Columns of a group: its B rows, rounded up to 64 (half of them in each CTA
// and in each half of the epilogue's warps, in whole 16-baseline rounds).
__host__ __device__ __forceinline__ int group_cols(int N, int b2) {
    const int c = (2 * N - 128 * b2 + 63) & ~63;
    return c < 256 ? c : 256;
}

// Work units per k-tile: 2 for the single diagonal pair (one tile loaded,
// two MMAs in FP32 mode); for a group, one per tile that a CTA loads (on the
// diagonal its A tile is also its half of B) plus one.  Each item
// (with k-tiles) starts with kEndUnits more, standing for the cost of an
// item's end (~4 k-tiles); they hold no k-tile.
constexpr int kEndUnits = 8;

__host__ __device__ __forceinline__ int64_t item_units(int64_t tiles, int w) {
    return tiles > 0 ? kEndUnits + tiles * w : 0;
}
__host__ __device__ __forceinline__ int pair_units(int gi, int nblk) {
    if (nblk == 1) return 2;
    int b1, b2, nbB;
    group_decode(gi, nblk, b1, b2, nbB);
    return b2 != b1 ? 3 : 2;
}

// How far the groups of the channel whose first item is g0 are turned.
__host__ __device__ __forceinline__ int group_turn(int g0, int npairs, int G) {
    const int step = (npairs + 1 - G % npairs) % npairs;
    return (int)((int64_t)step * (g0 / G) % npairs);
}

// Item g of the round-robin deal to G workers.
__device__ __forceinline__ Item decode_item(const TcArgs& a, int g, int G) {
    int m = 0;
    while (m + 1 < a.n_modes && g >= a.md[m + 1].item_base) ++m;
    const TcModeArgs& d = a.md[m];
    int l = g - d.item_base;
    Item it;
    it.m = m;
    // group fastest: the CTAs that take one channel's groups at the same
    // time share its block tiles through L2.  The order of a channel's groups
    // is turned by one deal round after another so that a worker's group
    // index steps by one per round, whatever G is modulo npairs: groups cost
    // 2 or 3 units, and with G a multiple of npairs a worker would only ever
    // see one of them
    int pr = l % d.npairs;
    l /= d.npairs;
    if (d.npairs > 1) pr = (pr + group_turn(d.item_base + l * d.npairs, d.npairs, G)) % d.npairs;
    it.pr = pr;
    it.k = l % d.C;
    it.sp = l / d.C;
    group_decode(pr, d.nblk, it.b1, it.b2, it.nbB);
    return it;
}

__device__ __forceinline__ int block_ants(int N, int b) { return min(64, N - 64 * b); }

// The pieces of one CTA, in the same order for every role.
//
// Balanced deal: every mode's items (block pair major, channel fastest) are
// laid end to end as k-tiles of pair_units() units each, U units in all; CTA
// c owns the k-tiles whose first unit u has floor(u G / U) = c, so every CTA
// gets the same work to within one k-tile, whatever the channel count.  An
// item cut between CTAs is combined by the last of them (ticket).
// Round-robin deal (tile choices fixed by the caller): item g goes to CTA
// g mod G, its range is split number sp of n_split equal ranges.
struct PieceCursor {
    int m, pr, k, g;
    int64_t ibase, lo, hi;
};

// x / y for non-negative operands of the balanced deal.  The cursors divide
// several times per piece, on one lane and before its first load: ~150 clocks
// each in 64 bits, a few in 32.
__device__ __forceinline__ int64_t deal_div(const TcArgs& a, int64_t x, int64_t y) {
    return a.u32 ? (int64_t)((uint32_t)x / (uint32_t)y) : x / y;
}
__device__ __forceinline__ int64_t ceil_div(const TcArgs& a, int64_t x, int64_t y) {
    return deal_div(a, x + y - 1, y);
}

template <bool WIDE>
__device__ __forceinline__ void cursor_init(const TcArgs& a, PieceCursor& c) {
    c.g = WIDE ? blockIdx.x >> 1 : blockIdx.x;
    c.m = a.n_modes;
    if (WIDE || !a.balanced) return;
    const int64_t G = gridDim.x;
    c.lo = ceil_div(a, (int64_t)blockIdx.x * a.units, G);
    c.hi = ceil_div(a, (int64_t)(blockIdx.x + 1) * a.units, G);
    for (int m = 0; m < a.n_modes; ++m) {
        const TcModeArgs& d = a.md[m];
        int64_t base = d.unit_base;
        for (int pr = 0; pr < d.npairs; ++pr) {
            const int64_t iu = item_units(d.tiles, pair_units(pr, d.nblk));
            const int64_t pu = iu * d.C;
            if (c.lo < base + pu) {
                c.m = m;
                c.pr = pr;
                c.k = (int)deal_div(a, c.lo - base, iu);
                c.ibase = base + (int64_t)c.k * iu;
                return;
            }
            base += pu;
        }
    }
}

template <bool WIDE>
__device__ __forceinline__ bool next_piece(const TcArgs& a, PieceCursor& c, Piece& p) {
    if (WIDE || !a.balanced) {
        if (c.g >= a.total_items) return false;
        const int G = WIDE ? gridDim.x >> 1 : gridDim.x;      // workers: CTA pairs or CTAs
        p.itm = decode_item(a, c.g, G);
        const TcModeArgs& d = a.md[p.itm.m];
        p.s_beg = (int64_t)p.itm.sp * d.S_item;
        p.s_end = min(d.S_pad, p.s_beg + d.S_item);
        p.slot = p.itm.sp;
        p.nslots = d.n_split;
        c.g += G;
        return true;
    }
    const int64_t G = gridDim.x;
    while (c.m < a.n_modes && c.ibase < c.hi) {
        const TcModeArgs& d = a.md[c.m];
        const int w = pair_units(c.pr, d.nblk);
        const int64_t t0 = c.ibase + kEndUnits;          // first unit of k-tile 0
        const int64_t j0 = c.lo > t0 ? ceil_div(a, c.lo - t0, w) : 0;
        const int64_t j1 = c.hi > t0 ? min(d.tiles, ceil_div(a, c.hi - t0, w)) : 0;
        const bool mine = j0 < j1;
        if (mine) {
            p.itm.m = c.m;
            p.itm.k = c.k;
            p.itm.pr = c.pr;
            group_decode(c.pr, d.nblk, p.itm.b1, p.itm.b2, p.itm.nbB);
            p.itm.sp = 0;
            const int64_t KT = a.KT;
            p.s_beg = j0 * KT;
            p.s_end = j1 * KT;
            const int first = (int)deal_div(a, t0 * G, a.units);
            const int last = (int)deal_div(a, (t0 + (d.tiles - 1) * w) * G, a.units);
            p.slot = (int)blockIdx.x - first;
            p.nslots = last - first + 1;
        }
        c.ibase += item_units(d.tiles, w);
        if (++c.k == d.C) {
            c.k = 0;
            if (++c.pr == d.npairs) {
                c.pr = 0;
                ++c.m;
            }
        }
        if (mine) return true;
    }
    return false;
}

// Bounded wait with this launch's limit and status word.
template <WaitSem SEM = kAcquireCta>
__device__ __forceinline__ bool wait_bar(uint32_t bar, uint32_t parity, volatile int* abort_word,
                                         const TcArgs& a) {
    return wait_bar_t<SEM>(bar, parity, abort_word, a.timeout_ns, a.status);
}

__device__ __forceinline__ void epi_sync() { asm volatile("bar.sync 1, 256;" ::: "memory"); }


// --------------------------------------------------------------------- kernel

// Stage layout of one item.  A group with its own B slots fills each k-tile's
// atom of the launch's layout.  An item whose A tiles are also its B tiles
// (single block, group on the diagonal) packs them densely: atom = [hi | lo]
// tiles of its mode's box (one block: 2N rows rounded up to 8), as many per
// stage as fit and divide a window.
struct ItemLayout {
    uint32_t atom;      // bytes per k-tile
    uint32_t plo;       // hi -> lo plane within a k-tile
    int at;             // k-tiles per stage
};

__device__ __forceinline__ ItemLayout item_layout(const TcArgs& a, const TcModeArgs& d, bool dense,
                                                  int planes, uint32_t stage_bytes,
                                                  uint32_t atom_bytes, uint32_t plane_off) {
    ItemLayout L;
    if (!dense) {
        L.atom = atom_bytes;
        L.plo = plane_off;
        L.at = a.atoms;
        return L;
    }
    L.atom = (uint32_t)planes * d.box_bytes;
    L.plo = d.box_bytes;
    const int wk = a.W >> a.kt_shift;                 // k-tiles per window
    int at = (int)min((uint32_t)wk, stage_bytes / L.atom);
    while (at > 1 && wk % at) --at;
    L.at = max(at, 1);
    return L;
}

// How far a pair's CTAs came (see WIDE below); rank 0 writes most of it in both.
struct PairEnd {
    int loads[2];       // stage loads of each rank (in rank 0)
    int skipped;        // rank 0's first one, left out by the test hook
    int commits;        // stages and windows whose MMAs rank 0 committed
    int windows;
    int drain;          // rank 0 committed to the drain barrier
    int abort;          // the other rank gave up
};

// Times that n uses of the stages in turn come to stage s.
__device__ __forceinline__ int turns(int n, int s, int stages) {
    return n > s ? (n - 1 - s) / stages + 1 : 0;
}

// One thread of each CTA of a pair, when every role of both has stopped after
// a wait ran out: the copies that either producer started (on rank 0's full
// barriers), and the arrivals of rank 0's commits at this CTA's barriers.
// Waits are bounded.
__device__ __noinline__ void pair_drain(const PairEnd& e, int rank, int stages, uint64_t* full,
                                        uint64_t* empty, uint64_t* accf, uint64_t* drain,
                                        unsigned long long timeout_ns) {
    const unsigned long long until = globaltimer() + timeout_ns;
    auto over = [&](uint64_t* bar, int phases) {      // the last of the barrier's phases
        while (phases > 0 && !mbar_try_wait<kAcquireCluster>(smem_u32(bar), (uint32_t)(phases - 1) & 1u))
            if (globaltimer() > until) break;
    };
    for (int s = 0; s < stages; ++s) {
        if (rank == 0) {
            // a producer is at most one load of a stage ahead of the other:
            // arrive in that one's place
            const int c0 = turns(e.loads[0], s, stages) - (s == 0 ? e.skipped : 0);
            const int c1 = turns(e.loads[1], s, stages);
            if (c0 != c1) mbar_arrive(smem_u32(&full[s]));
            over(&full[s], max(c0, c1));
        }
        over(&empty[s], turns(e.commits, s, stages));
    }
    for (int b = 0; b < 2; ++b) over(&accf[b], turns(e.windows, b, 2));
    over(drain, e.drain);
}

// WIDE: modes of several antenna blocks, worked on by pairs of CTAs (clusters
// of two, tcgen05 cta_group::2).  A pair's MMA is M = 256 (each CTA's 128 A
// rows, one antenna block), N up to 256 (half of the B rows in each CTA's
// shared memory); each CTA's TMEM holds its own 128 rows.  A CTA reads 8 KB
// of operands per K = 16 step of 128 clocks, the shared-memory rate at which
// MMAs are fed (~64 bytes per clock: alone, a CTA's 128 x 256 tile reads 12
// KB per step and ran at 60% of the tensor rate with its loads taken away),
// and loads 8 tiles per channel and k-tile at N = 256, not 12.  A pass of
// 4096 spectra at N = 256, K = 1024: FP32 mode 2033 -> 1402 us, FP16 831 ->
// 527, FP8 371 -> 264 (with the scales and the issue loop below).
// Rank 0 issues the MMAs.  Each CTA loads its own tiles, and both CTAs' copies
// complete on rank 0's full barriers (the loads' .cta_group::2 form), whose
// phases take the two producers' announcements and all the bytes: rank 0 waits,
// with acquire at cluster scope, for what its MMAs read in both CTAs (256
// antennas, K = 1024, 4096 spectra FP16 527 us, 130, K = 2048, 1500 spectra 337,
// not above a relay of each full stage by a warp of the other CTA, 530 and 352,
// which ordered nothing, nor above waits at CTA scope).  Commits arrive at both CTAs'
// barriers; the epilogue warps of both free an accumulator set.
// If a launch gives up, a pair's CTAs exchange how far they came and wait for
// everything still under way to either (pair_drain) before one may end.
template <int MODE, bool WIDE>
__global__ void __launch_bounds__(kTcThreads, 1) xengine_tc_kernel(const __grid_constant__ TcArgs a) {
    extern __shared__ unsigned char smem_raw[];
    unsigned char* smem = reinterpret_cast<unsigned char*>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    constexpr int planes = MODE == 0 ? 2 : 1;
    // Stage layout of a group (WIDE): per k-tile ("atom") the A slot of each
    // plane [hi | lo], then the B half's; a slot has slot_rows = 128 rows.  A
    // single-block item packs its k-tiles densely instead
    // ([hi | lo] of its own 2N-rounded-up-to-8 rows each, item_layout).  The
    // MMA reads 128 rows from a tile (and a single block's concatenated
    // [hi; lo] B operand 2 box rows); rows past the antennas only feed
    // outputs the epilogue ignores, and the ring is followed by enough shared
    // memory for the reads past its last tile.
    const uint32_t slot = (uint32_t)a.slot_rows * (uint32_t)a.row_bytes;
    constexpr int KK = MODE == 2 ? 4 : 2;       // MMA k-steps (32 bytes of a row) per k-tile
    const uint32_t plane_off = slot;                                // A: hi -> lo plane
    const uint32_t bh_off = planes * slot;                          // B half: hi
    const uint32_t bl_off = bh_off + slot;                          // B half: lo (planes == 2)
    const uint32_t atom_bytes = planes * slot * (WIDE ? 2u : 1u);
    constexpr bool single = !WIDE;
    constexpr int CG = WIDE ? 2 : 1;
    const int rank = WIDE ? (int)(blockIdx.x & 1) : 0;              // CTA of the pair
    const uint32_t stage_bytes = atom_bytes * (uint32_t)a.atoms;
    unsigned char* stages = smem;
    float* Gs = reinterpret_cast<float*>(smem + a.stages * stage_bytes);   // <= 128 x 129; WIDE: scales
    // WIDE: each epilogue warp's staging rows for V, [16][kVRow] float2
    float2* vstage = reinterpret_cast<float2*>(Gs + a.gs_floats);
    uint64_t* bars = reinterpret_cast<uint64_t*>(
        (reinterpret_cast<uintptr_t>(vstage + (WIDE ? 8 * 16 * kVRow : 0)) + 15) & ~(uintptr_t)15);
    uint64_t* full = bars;
    uint64_t* empty = full + a.stages;
    uint64_t* accf = empty + a.stages;
    uint64_t* acce = accf + 2;
    uint64_t* drain = acce + 2;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain + 1);
    volatile int* abort_word = reinterpret_cast<volatile int*>(tmem_slot + 1);
    volatile int* epi_last = abort_word + 2;
    PieceCursor* epi_cur = reinterpret_cast<PieceCursor*>(
        (reinterpret_cast<uintptr_t>(epi_last + 2) + 15) & ~(uintptr_t)15);
    Piece* epi_pc = reinterpret_cast<Piece*>(epi_cur + 1);
    volatile int* epi_more = reinterpret_cast<volatile int*>(epi_pc + 2);   // [2], as epi_pc
    volatile int* epi_abort = epi_more + 2;
    PairEnd* pair_end = reinterpret_cast<PairEnd*>(const_cast<int*>(epi_abort + 1));

    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;

    if (threadIdx.x == 0) {
        for (int s = 0; s < a.stages; ++s) {
            mbar_init(smem_u32(&full[s]), WIDE ? 2 : 1);       // one per producer
            mbar_init(smem_u32(&empty[s]), 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(smem_u32(&accf[b]), 1);
            mbar_init(smem_u32(&acce[b]), WIDE ? 16 : 8);      // one arrival per epilogue warp
        }
        mbar_init(smem_u32(drain), 1);
        *abort_word = 0;
        if (WIDE) *pair_end = PairEnd{};
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) {
        if (WIDE) {
            asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                             smem_u32(tmem_slot)),
                         "r"(kTmemCols)
                         : "memory");
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
        } else {
            asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                             smem_u32(tmem_slot)),
                         "r"(kTmemCols)
                         : "memory");
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
        }
    }
    tc_fence_before();
    if (WIDE)
        cluster_sync();
    else
        __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    if (warp == 0) {
        // ------------------------------------------------------ TMA producer
        // (Warps 0 and 1 run their loops whole, with one elected lane issuing:
        // addresses and descriptors then live in uniform registers, which a
        // loop of one lane has to fill again for every instruction.)
        const bool el = elect_one();
        uint32_t st = 0, ph = 0;               // stage slot and its phase parity
        uint32_t armed = 0, armed_ph = 0;      // slots with copies in flight, their parity
        bool ok = true, first = true;
        int loads = 0;
        const uint32_t stage0 = smem_u32(stages);
        const uint32_t full0 = WIDE ? cluster_addr(smem_u32(full), 0) : smem_u32(full);
        PieceCursor cur;
        cursor_init<WIDE>(a, cur);
        Piece pc;
        while (ok && next_piece<WIDE>(a, cur, pc)) {
            const Item& itm = pc.itm;
            const TcModeArgs& d = a.md[itm.m];
            const CUtensorMap* map = &a.tmap[itm.m];
            // one block: A = B, one tile.  Group on the diagonal: A is the
            // CTA's half of B (if both blocks are there)
            const int cols = group_cols(d.N, itm.b2);
            const bool alias = single || (itm.b2 == itm.b1 && cols == 256);
            const int ra = kRows * (itm.b1 + rank);
            const int rb = kRows * itm.b2 + rank * (cols >> 1);
            const uint32_t tile_bytes = planes * d.box_bytes * (alias ? 1u : 2u);
            const ItemLayout lay = item_layout(a, d, alias, planes, stage_bytes, atom_bytes, plane_off);
            const int t_end = (int)(pc.s_end >> a.kt_shift);
            for (int t = (int)(pc.s_beg >> a.kt_shift); t < t_end; t += lay.at) {
                if (!__all_sync(0xffffffffu, wait_bar(smem_u32(&empty[st]), ph ^ 1u, abort_word, a))) {
                    ok = false;
                    break;
                }
                if (!(a.withhold && blockIdx.x == 0 && first)) {      // (test hook)
                    const int n_at = min(lay.at, t_end - t);
                    const uint32_t fb = full0 + 8u * st;
                    uint32_t dst = stage0 + st * stage_bytes;
                    if (el) {
                        if (WIDE)
                            mbar_expect_tx_cluster(fb, (uint32_t)n_at * tile_bytes);
                        else
                            mbar_expect_tx(fb, (uint32_t)n_at * tile_bytes);
                        for (int at = 0; at < n_at; ++at, dst += lay.atom) {
                            tma_load_4d<CG>(dst, map, fb, ra, itm.k, t + at);
                            if (planes == 2)
                                tma_load_4d<CG>(dst + lay.plo, map, fb, ra, itm.k, d.cap_tiles + t + at);
                            if (!alias) {
                                tma_load_4d<CG>(dst + bh_off, map, fb, rb, itm.k, t + at);
                                if (planes == 2)
                                    tma_load_4d<CG>(dst + bl_off, map, fb, rb, itm.k, d.cap_tiles + t + at);
                            }
                        }
                    }
                    armed |= 1u << st;
                    armed_ph = (armed_ph & ~(1u << st)) | (ph << st);
                }
                first = false;
                ++loads;
                if (++st == (uint32_t)a.stages) {
                    st = 0;
                    ph ^= 1u;
                }
            }
        }
        // WIDE: the last commits' arrivals from the other CTA are in
        // (nothing else waits for them before this CTA may end)
        if (WIDE)
            for (int s2 = 0; ok && s2 < a.stages; ++s2)
                if ((armed >> s2) & 1u)
                    ok = __all_sync(0xffffffffu,
                                    wait_bar(smem_u32(&empty[s2]), (armed_ph >> s2) & 1u, abort_word, a));
        if (WIDE && el) {
            st_cluster(cluster_addr(smem_u32(&pair_end->loads[rank]), 0), loads);
            if (a.withhold && blockIdx.x == 0) pair_end->skipped = min(loads, 1);
        }
        if (!WIDE && !ok) {
            // drain: every armed stage's copies must land before teardown
            const unsigned long long d2 = globaltimer() + a.timeout_ns;
            for (int s2 = 0; s2 < a.stages && s2 < 16; ++s2) {
                if (!((armed >> s2) & 1u)) continue;
                while (!mbar_try_wait(smem_u32(&full[s2]), (armed_ph >> s2) & 1u))
                    if (globaltimer() > d2) break;
            }
        }
    } else if (warp == 1) {
        // ------------------------------------------------------- MMA issuer
        // (a pair's other CTA issues none)
        if (rank == 0) {
            const bool el = elect_one();
            uint32_t st = 0, ph = 0;
            int wi = 0;
            bool ok = true;
            bool issued = false;
            int commits = 0, windows = 0;
            // tiles of both CTAs are read; accumulator sets of both overwritten
            constexpr WaitSem kFull = WIDE ? kAcquireCluster : kAcquireCta;
            constexpr WaitSem kFree = WIDE ? kRelaxedCluster : kAcquireCta;
            const uint32_t lo0 = op_desc_lo(smem_u32(stages));
            PieceCursor cur;
            cursor_init<WIDE>(a, cur);
            Piece pc;
            while (ok && next_piece<WIDE>(a, cur, pc)) {
                const Item& itm = pc.itm;
                const TcModeArgs& d = a.md[itm.m];
                // single block: N = 2N rounded up to 16, FP32 mode: B = [hi;
                // lo], the k-tile's two tiles of box_rows rows each, N = 2
                // box_rows, so one MMA forms [Dhh | Dhl] (Dhl from column
                // box_rows)
                const int box_rows = (int)(d.box_bytes / (uint32_t)a.row_bytes);
                const int Nn = !single     ? group_cols(d.N, itm.b2)
                               : MODE == 0 ? 2 * box_rows
                                           : (2 * block_ants(d.N, 0) + 15) & ~15;
                const bool alias = single || (itm.b2 == itm.b1 && Nn == 256);
                // D = F32, A/B = F16 (kind::f16) or E4M3 (kind::f8f6f4), K-major,
                // N>>3 at bits 17-22, M>>4 at bits 24-28
                const uint32_t idesc = (1u << 4) | ((uint32_t)(Nn >> 3) << 17) |
                                       ((CG * kRows >> 4) << 24);
                const ItemLayout lay = item_layout(a, d, alias, planes, stage_bytes, atom_bytes, plane_off);
                // (descriptor addresses count 16 bytes)
                const uint32_t al_o = lay.plo >> 4;                    // A lo
                const uint32_t bh_o = alias ? 0u : bh_off >> 4;        // group: B from its own
                const uint32_t bl_o = alias ? al_o : bl_off >> 4;      // slots, or A's (in both CTAs)
                const uint32_t atom_o = lay.atom >> 4;
                const int wk = a.W >> a.kt_shift;
                const int t_end = (int)(pc.s_end >> a.kt_shift);
                for (int t = (int)(pc.s_beg >> a.kt_shift); ok && t < t_end; ++wi) {
                    const int b = wi & 1;
                    const uint32_t aph = (uint32_t)(wi >> 1) & 1u;
                    if (!__all_sync(0xffffffffu, wait_bar<kFree>(smem_u32(&acce[b]), aph ^ 1u, abort_word, a))) {
                        ok = false;
                        break;
                    }
                    const uint32_t d0 = tmem + (uint32_t)b * 256u;
                    const int tw = min(t_end, t + wk);
                    uint32_t acc = 0;
                    for (; t < tw; t += lay.at) {
                        if (!__all_sync(0xffffffffu, wait_bar<kFull>(smem_u32(&full[st]), ph, abort_word, a))) {
                            ok = false;
                            break;
                        }
                        tc_fence_after();
                        const int n_at = min(lay.at, tw - t);
                        if (el) {
                            uint32_t lo = lo0 + st * (stage_bytes >> 4);
#pragma unroll 2
                            for (int at = 0; at < n_at; ++at, lo += atom_o) {
#pragma unroll
                                for (int kk = 0; kk < KK; ++kk) {
                                    const uint64_t ah = op_desc<MODE>(lo + 2u * kk);
                                    if (single) {
                                        mma<MODE, CG>(d0, ah, ah, idesc, acc);
                                    } else {
                                        const uint64_t bh = op_desc<MODE>(lo + bh_o + 2u * kk);
                                        mma<MODE, CG>(d0, ah, bh, idesc, acc);
                                        if (MODE == 0) {
                                            const uint64_t al = op_desc<MODE>(lo + al_o + 2u * kk);
                                            const uint64_t bl = op_desc<MODE>(lo + bl_o + 2u * kk);
                                            mma<MODE, CG>(d0, ah, bl, idesc, 1u);
                                            mma<MODE, CG>(d0, al, bh, idesc, 1u);
                                        }
                                    }
                                    acc = 1;
                                }
                            }
                            mma_commit<CG>(smem_u32(&empty[st]));
                            if (t + lay.at >= tw) mma_commit<CG>(smem_u32(&accf[b]));
                        }
                        acc = 1;
                        issued = true;
                        ++commits;
                        if (t + lay.at >= tw) ++windows;
                        if (++st == (uint32_t)a.stages) {
                            st = 0;
                            ph ^= 1u;
                        }
                    }
                }
            }
            if (!ok && issued) {
                // drain: wait for every MMA this warp issued before TMEM is freed
                if (el) mma_commit<CG>(smem_u32(drain));
                const unsigned long long d2 = globaltimer() + a.timeout_ns;
                while (!mbar_try_wait(smem_u32(drain), 0u))
                    if (globaltimer() > d2) break;
            }
            if (WIDE && el)
                for (int r = 0; r < 2; ++r) {
                    st_cluster(cluster_addr(smem_u32(&pair_end->commits), r), commits);
                    st_cluster(cluster_addr(smem_u32(&pair_end->windows), r), windows);
                    st_cluster(cluster_addr(smem_u32(&pair_end->drain), r), !ok && issued);
                }
        }
    } else {
        // --------------------------------------------------------- epilogue
        // 8 warps: warp w reads TMEM lane quadrant w % 4 (rows 32q..32q+31)
        // and one half of the Nn accumulator columns.  Each warp waits for a
        // window on its own (lane 0 polls, the warp then loads its slice) and
        // frees the accumulator set by one arrival per warp; the 8 warps meet
        // only at the end of an item.  A warp whose wait fails stops loading
        // but still joins the item-end barriers, after which every warp sees
        // the shared abort word and leaves together.
        const int et = threadIdx.x - 64;            // 0..255
        const int q = warp & 3;
        const int h = (warp - 2) >> 2;
        const int r = 32 * q + lane;
        int wi = 0;
        // one cursor for the 8 warps, in shared memory (registers are scarce here)
        if (et == 0) {
            cursor_init<WIDE>(a, *epi_cur);
            epi_more[0] = next_piece<WIDE>(a, *epi_cur, epi_pc[0]) ? 1 : 0;
        }
        epi_sync();
        for (int pb = 0;; pb ^= 1) {
            if (!epi_more[pb]) break;
            const Piece pc = epi_pc[pb];
            // the piece after it, while this one's windows are on their way
            if (et == 0) epi_more[pb ^ 1] = next_piece<WIDE>(a, *epi_cur, epi_pc[pb ^ 1]) ? 1 : 0;
            const Item& itm = pc.itm;
            const TcModeArgs& d = a.md[itm.m];
            constexpr bool use_t = MODE == 0 && single;
            // antennas of this CTA's A block (a group's second one may not exist)
            const int nb1 = max(0, block_ants(d.N, itm.b1 + rank));
            const int R2 = 2 * nb1;
            // columns per half: one block 2N rounded up to 16, halved (<= 64);
            // a group's columns, halved (<= 128)
            const int NH = single ? ((R2 + 15) & ~15) >> 1 : group_cols(d.N, itm.b2) >> 1;
            const int col0 = h * NH;
            const int64_t s_beg = pc.s_beg;
            const int64_t s_end = pc.s_end;
            // a group's scales, 64 of the rows' and 128 of the columns'
            // antennas, while its windows are on their way (read for each V,
            // from global memory: FP16 at N = 256 655 us a pass, now 589)
            if (!single && et < 192) {
                const int i = et < 64 ? 64 * (itm.b1 + rank) + et : 64 * itm.b2 + et - 64;
                Gs[et] = i >= d.N ? 1.f
                                  : (MODE == 0 ? __ldg(d.split + i)
                                               : __ldg(d.scale + (int64_t)i * d.C + itm.k));
            }
            // window sums: acc[0 .. NH) (single block, FP32 mode: [0, 64) from
            // hi hi^T and [64, 64 + NH) from hi lo^T)
            float acc[128];
#pragma unroll
            for (int j = 0; j < 128; ++j) acc[j] = 0.f;
            bool dead = false;
            for (int64_t w0 = s_beg; w0 < s_end; w0 += a.W, ++wi) {
                if (dead) continue;
                const int b = wi & 1;
                const uint32_t aph = (uint32_t)(wi >> 1) & 1u;
                int ok = 0;
                if (lane == 0) ok = wait_bar(smem_u32(&accf[b]), aph, abort_word, a) ? 1 : 0;
                ok = __shfl_sync(0xffffffffu, ok, 0);
                if (!ok) {
                    dead = true;
                    continue;
                }
                tc_fence_after();
                const uint32_t trow =
                    tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)b * 256u + (uint32_t)col0;
#pragma unroll
                for (int c = 0; c < 16; ++c) {
                    if (8 * c < NH) {
                        uint32_t v[8];
                        tmem_ld8(trow + 8u * c, v);
                        if (c < 8 && use_t) {
                            uint32_t w[8];
                            tmem_ld8(trow + d.box_bytes / (uint32_t)a.row_bytes + 8u * c, w);
                            tmem_ld_wait();
#pragma unroll
                            for (int j = 0; j < 8; ++j) {
                                acc[8 * c + j] += __uint_as_float(v[j]);
                                acc[(64 + 8 * c + j) & 127] += __uint_as_float(w[j]);
                            }
                        } else {
                            tmem_ld_wait();
#pragma unroll
                            for (int j = 0; j < 8; ++j) acc[8 * c + j] += __uint_as_float(v[j]);
                        }
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) {                                  // this warp's slice is free
                    if (rank == 0)
                        mbar_arrive(smem_u32(&acce[b]));
                    else
                        mbar_arrive_cluster(cluster_addr(smem_u32(&acce[b]), 0));
                }
            }
            epi_sync();
            // one reading of the abort word for the 8 warps (the producer and
            // the MMA thread may set it at any time)
            if (et == 0) *epi_abort = *abort_word;
            epi_sync();
            if (*epi_abort) break;
            const int N = d.N, C = d.C, P = d.P;
            const bool direct = pc.nslots == 1;
            if (!single) {
                // Group: rows 2 i' and 2 i' + 1 (Re and Im of antenna i') are
                // adjacent lanes, so V comes from one exchange with the partner
                // lane: for B columns 2 j'' and 2 j'' + 1 the even lane holds
                // G[2i'][..], the odd lane G[2i'+1][..];
                //   Re V = G[2i'][2j''] + G[2i'+1][2j''+1], Im V = G[2i'+1][2j''] - G[2i'][2j''+1].
                // The even lane takes the even column pairs, the odd lane the
                // odd ones, into the warp's staging rows (16 antennas x kVCols
                // baselines per round); the warp then writes each antenna's
                // kVCols baselines, consecutive in the accumulator layout, as
                // one coalesced run of FP32 stores into the item's partial
                // slot.  (FP64 reductions straight into the accumulator, one
                // per word, cost a group pass at N = 256 ~70% more time.)
                const int odd = r & 1;
                float2* vst = vstage + (warp - 2) * 16 * kVRow;
                const int jg0 = col0 >> 1;                  // the warp's first baseline of the group
                float2* pout = d.partial + ((int64_t)pc.slot * C + itm.k) * P;
#pragma unroll
                for (int rho = 0; rho < 64 / kVCols; ++rho) {
                    if (2 * kVCols * rho < NH) {
#pragma unroll
                        for (int kk = 0; kk < kVCols; ++kk) {
                            const int k2 = kVCols * rho + kk;
                            const float v0 = acc[2 * k2], v1 = acc[2 * k2 + 1];
                            const float x0 = __shfl_xor_sync(0xffffffffu, v0, 1);
                            const float x1 = __shfl_xor_sync(0xffffffffu, v1, 1);
                            if ((kk & 1) == odd) {
                                const float av = odd ? x0 : v0, bv = odd ? x1 : v1;
                                const float cv = odd ? v0 : x0, dv = odd ? v1 : x1;
                                vst[(lane >> 1) * kVRow + kk] = make_float2(av + dv, cv - bv);
                            }
                        }
                        __syncwarp();
                        // lane -> baseline jj of the round and one of 32 / kVCols
                        // antennas of each step over the warp's 16
                        constexpr int kRowsPerStep = 32 / kVCols;
                        const int jj = lane % kVCols;
                        const int jg = jg0 + kVCols * rho + jj;
                        const int b2 = itm.b2 + (jg >> 6);
                        const int j_loc = jg & 63;
                        const bool jv = j_loc < block_ants(N, b2);
                        const int j = 64 * b2 + j_loc;
                        const float sj = Gs[64 + jg];
#pragma unroll 1
                        for (int i0 = 0; i0 < 16; i0 += kRowsPerStep) {
                            const int i16 = i0 + lane / kVCols;
                            const int i_loc = 16 * q + i16;
                            if (16 * q + i0 >= nb1) break;
                            const int i = 64 * (itm.b1 + rank) + i_loc;
                            if (i_loc < nb1 && jv && j >= i) {
                                const float f = 1.0f / (Gs[i_loc] * sj);
                                const float2 v = vst[i16 * kVRow + jj];
                                const int p = i * N - i * (i - 1) / 2 + (j - i);
                                pout[p] = make_float2(v.x * f, v.y * f);
                            }
                        }
                        __syncwarp();
                    }
                }
            } else {
            // FP32 mode: G = S + L^T with S = Dhh + Dhl and L = Dhl.  Only the
            // 2 x 2 antenna blocks on and above the diagonal are needed, so
            // the square holds S there and L below it, and L of the diagonal
            // blocks has its own place (Ld): one store per element, and the
            // pair adds the transposed element when it reads.  (Adding L^T in
            // place cost a dependent shared load, add and store per element.)
            const int ldg = R2 + 1;
            float* Ld = Gs + a.gs_floats - 2 * kRows;          // [row][col mod 2]
            if (r < R2) {
                const int dcol = r & ~1;                       // the diagonal block's first column
#pragma unroll
                for (int c = 0; c < 64; ++c) {
                    const int col = col0 + c;
                    if (c < NH && col < R2) {
                        Gs[r * ldg + col] = use_t ? (col < dcol ? acc[64 + c] : acc[c] + acc[64 + c]) : acc[c];
                        if (use_t && (col & ~1) == dcol) Ld[2 * r + (col & 1)] = acc[64 + c];
                    }
                }
            }
            epi_sync();
            const int npl = nb1 * (nb1 + 1) / 2;
            {
                // kVB pairs per thread at a time: their accumulator loads are
                // issued together, so their latencies overlap
                for (int base = et; base < npl; base += kVB * 256) {
                    int pp[kVB];
                    float vre[kVB], vim[kVB];
#pragma unroll
                    for (int u = 0; u < kVB; ++u) {
                        const int pl = base + 256 * u;
                        pp[u] = -1;
                        vre[u] = vim[u] = 0.f;
                        if (pl < npl) {
                            const int li = triangle_row(pl, nb1);
                            const int lj = li + (pl - triangle_start(li, nb1));
                            // block rows 2 i' (Re) and 2 i' + 1 (Im)
                            const float* g0 = Gs + 2 * li * ldg + 2 * lj;
                            float g00 = g0[0], g01 = g0[1], g10 = g0[ldg], g11 = g0[ldg + 1];
                            if (use_t) {
                                const bool dg = li == lj;
                                const float* t = dg ? Ld + 4 * li : Gs + 2 * lj * ldg + 2 * li;
                                const int st = dg ? 2 : ldg;
                                g00 += t[0];
                                g10 += t[1];
                                g01 += t[st];
                                g11 += t[st + 1];
                            }
                            const float re = g00 + g11;
                            const float im = g10 - g01;
                            float f;
                            if (MODE == 0)
                                f = 1.0f / (__ldg(d.split + li) * __ldg(d.split + lj));
                            else
                                f = 1.0f / (__ldg(d.scale + (int64_t)li * C + itm.k) *
                                            __ldg(d.scale + (int64_t)lj * C + itm.k));
                            pp[u] = pl;                    // one block: the pair order itself
                            vre[u] = re * f;
                            vim[u] = im * f;
                        }
                    }
                    if (direct) {
                        double2 old[kVB];
#pragma unroll
                        for (int u = 0; u < kVB; ++u) {
                            old[u] = make_double2(0.0, 0.0);
                            if (pp[u] >= 0 && !d.assign) old[u] = __ldcg(d.acc + (int64_t)itm.k * P + pp[u]);
                        }
#pragma unroll
                        for (int u = 0; u < kVB; ++u)
                            if (pp[u] >= 0)       // sole owner of (k, p) in this launch
                                d.acc[(int64_t)itm.k * P + pp[u]] =
                                    make_double2(old[u].x + (double)vre[u], old[u].y + (double)vim[u]);
                    } else {
#pragma unroll
                        for (int u = 0; u < kVB; ++u)
                            if (pp[u] >= 0)
                                d.partial[((int64_t)pc.slot * C + itm.k) * P + pp[u]] =
                                    make_float2(vre[u], vim[u]);
                    }
                }
            }
            }
            if (single && !direct) {
                // The last of the CTAs sharing this channel to finish adds
                // every partial, in slot order, into the FP64 accumulator:
                // deterministic.  (A group's slots are combined by a launch of
                // their own, launch_combine_ranges.)
                int* const ticket = d.ticket + itm.k;
                __threadfence();
                epi_sync();
                if (et == 0) {
                    const int old = atomicAdd(ticket, 1);
                    *epi_last = old == pc.nslots - 1 ? 1 : 0;
                }
                epi_sync();
                if (*epi_last) {
                    __threadfence();
                    // four pairs per thread at a time, their loads in flight together
                    const int npl_all = nb1 * (nb1 + 1) / 2;
                    constexpr int kCB = 4;
                    for (int base = et; base < npl_all; base += kCB * 256) {
                        int pp[kCB];
                        double re[kCB], im[kCB];
#pragma unroll
                        for (int u = 0; u < kCB; ++u) {
                            const int pl = base + 256 * u;
                            pp[u] = pl < npl_all ? pl : -1;
                            re[u] = im[u] = 0.0;
                        }
                        for (int sp = 0; sp < pc.nslots; ++sp) {
                            float2 v[kCB];
#pragma unroll
                            for (int u = 0; u < kCB; ++u)
                                v[u] = pp[u] >= 0 ? __ldcg(d.partial + ((int64_t)sp * C + itm.k) * P + pp[u])
                                                  : make_float2(0.f, 0.f);
#pragma unroll
                            for (int u = 0; u < kCB; ++u) {
                                re[u] += (double)v[u].x;
                                im[u] += (double)v[u].y;
                            }
                        }
                        double2 old[kCB];
#pragma unroll
                        for (int u = 0; u < kCB; ++u) {
                            old[u] = make_double2(0.0, 0.0);
                            if (pp[u] >= 0 && !d.assign) old[u] = d.acc[(int64_t)itm.k * P + pp[u]];
                        }
#pragma unroll
                        for (int u = 0; u < kCB; ++u)
                            if (pp[u] >= 0)
                                d.acc[(int64_t)itm.k * P + pp[u]] =
                                    make_double2(old[u].x + re[u], old[u].y + im[u]);
                    }
                    if (et == 0) *ticket = 0;
                }
            }
            epi_sync();
        }
    }

    // (a pair's CTAs end together: each may still read the other's tiles, and
    // arrive at its barriers, until here; every wait before this one is bounded)
    tc_fence_before();
    __syncwarp();
    if (WIDE) {
        if (*abort_word && lane == 0) st_cluster(cluster_addr(smem_u32(&pair_end->abort), rank ^ 1), 1);
        cluster_sync();
        if (*abort_word || pair_end->abort) {       // the same in both CTAs
            if (threadIdx.x == 0)
                pair_drain(*pair_end, rank, a.stages, full, empty, accf, drain, a.timeout_ns);
            __syncwarp();
            cluster_sync();
        }
    } else {
        __syncthreads();
    }
    if (warp == 1) {
        __syncwarp();
        tc_fence_after();
        if (WIDE)
            asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                         "r"(kTmemCols)
                         : "memory");
        else
            asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                         "r"(kTmemCols)
                         : "memory");
    }
}

// ----------------------------------------------------------------- host side

constexpr size_t kSmemBudget = 227 * 1024;

}  // namespace

// Ranges per item of each mode of a step, and the busiest worker's load.
struct RangePlan {
    std::vector<int> sp;
    double score = 0;
};

// How a launch deals its work to the CTAs (see next_piece).
struct DealPlan {
    std::vector<int> sp;      // round-robin deal: ranges per item of each mode
    bool balanced = false;    // contiguous deal of weighted k-tiles instead
    int grid = 0;             // CTAs of the balanced deal
    int64_t units = 0;        // its total work units
};

struct TcPlan {
    int N = 0, C = 0, P = 0, nblk = 1, npairs = 1;
    int mode = 0, planes = 1, KT = 32;
    int row_bytes = 64;       // tile row: 32 FP16 values, or 128 FP8
    int num_sms = 0;
    int box_rows = 128;       // TMA box rows: 2N rounded up to 8 for one block, else 128
    CUtensorMap tmap;
    bool have_map = false;
    int64_t cap = 0;
    int max_split = 1;
    int window = 0;           // 0 = per-mode default
    int stages = 0;           // 0 = as many as shared memory allows
    int split = 0;            // 0 = planner's choice
    int atoms = 0;            // k-tiles per stage, 0 = automatic
    unsigned long long timeout_ns = 4000000000ull;
    int withhold = 0;                    // test hook for the next launch
    unsigned long long hook_timeout_ns = 0;
    int* ticket = nullptr;               // [C] arrival counters
    size_t ticket_bytes() const { return (size_t)C * sizeof(int); }
    // decisions already made: ranges, keyed by every mode of the step, and the
    // deal of this plan alone, by its S_pad
    std::vector<std::pair<std::vector<int64_t>, RangePlan>> range_cache;
    std::vector<std::pair<int64_t, DealPlan>> deal_cache;
};

int tc_plan_create(TcPlan** out, int N, int C, int spec_type, std::string& err) {
    *out = nullptr;
    if (!get_encoder()) {
        err = "cuTensorMapEncodeTiled is not available from the driver";
        return CORR_ECUDA;
    }
    TcPlan* p = new TcPlan();
    p->N = N;
    p->C = C;
    p->P = N * (N + 1) / 2;
    p->nblk = (N + 63) / 64;
    p->npairs = groups_of(p->nblk);
    p->mode = spec_type == SPEC_F16X2 ? 0 : (spec_type == SPEC_F16 ? 1 : 2);
    p->planes = p->mode == 0 ? 2 : 1;
    p->KT = p->mode == 2 ? 128 : 32;
    p->row_bytes = p->mode == 2 ? 128 : 64;
    p->box_rows = p->nblk == 1 ? (2 * N + 7) / 8 * 8 : kRows;
    int dev = 0;
    cudaGetDevice(&dev);
    if (cudaDeviceGetAttribute(&p->num_sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
        delete p;
        err = "cudaDeviceGetAttribute failed";
        return CORR_ECUDA;
    }
    const size_t tb = p->ticket_bytes();
    if (dev_malloc((void**)&p->ticket, tb) != cudaSuccess || cudaMemset(p->ticket, 0, tb) != cudaSuccess) {
        cudaGetLastError();
        cudaFree(p->ticket);
        delete p;
        err = "device allocation failed";
        return CORR_ENOMEM;
    }
    *out = p;
    return CORR_OK;
}

int tc_reset(TcPlan* p) {
    // after an aborted launch some arrival counters may be left non-zero
    return cudaMemset(p->ticket, 0, p->ticket_bytes()) == cudaSuccess
               ? CORR_OK
               : CORR_ECUDA;
}

int tc_plan_update(TcPlan* p, void* spec, int64_t cap, int N, int C, int spec_type,
                   std::string& err) {
    (void)N;
    (void)C;
    const int eb = spec_elem_bytes(spec_type);
    const int R2 = 2 * p->N;
    // tile-major workspace: [plane][cap/T tiles][C][2N rows][T frames], T = KT
    const int T = p->row_bytes / eb;
    cuuint64_t dims[4] = {(cuuint64_t)T, (cuuint64_t)R2, (cuuint64_t)p->C,
                          (cuuint64_t)p->planes * (cap / T)};
    cuuint64_t strides[3] = {(cuuint64_t)T * eb, (cuuint64_t)R2 * T * eb,
                             (cuuint64_t)p->C * R2 * T * eb};
    cuuint32_t box[4] = {(cuuint32_t)T, (cuuint32_t)p->box_rows, 1, 1};
    cuuint32_t estr[4] = {1, 1, 1, 1};
    const CUtensorMapDataType dt =
        eb == 2 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16 : CU_TENSOR_MAP_DATA_TYPE_UINT8;
    CUresult r = get_encoder()(&p->tmap, dt, 4, spec, dims, strides, box, estr,
                               CU_TENSOR_MAP_INTERLEAVE_NONE,
                               p->row_bytes == 64 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_128B,
                               CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) {
        char buf[128];
        snprintf(buf, sizeof buf, "cuTensorMapEncodeTiled failed (%d)", (int)r);
        err = buf;
        return CORR_ECUDA;
    }
    p->have_map = true;
    p->cap = cap;
    p->max_split = (int)std::min<int64_t>(8, (cap + 255) / 256);
    p->range_cache.clear();
    p->deal_cache.clear();
    return CORR_OK;
}

int tc_set_tiles(TcPlan* p, int window, int stages, int split, int atoms, std::string& err) {
    if (atoms < 0 || atoms > 8) {
        err = "atoms must be in [0, 8]";
        return CORR_EINVAL;
    }
    if (split < 0 || split > 64) {
        err = "split must be in [0, 64]";
        return CORR_EINVAL;
    }
    if (window != 0 && (window < p->KT || window % p->KT || window > 4096)) {
        err = "window must be a multiple of the k-tile (32 spectra, 128 for FP8) up to 4096";
        return CORR_EINVAL;
    }
    if (stages != 0 && (stages < 2 || stages > 16)) {
        err = "stages must be in [2, 16]";
        return CORR_EINVAL;
    }
    p->window = window;
    p->stages = stages;
    p->split = split;
    p->atoms = atoms;
    p->range_cache.clear();
    p->deal_cache.clear();
    return CORR_OK;
}

namespace {

// Work units per k-tile of work group pr (pair_units()).
int host_pair_units(int pr, int nblk) { return pair_units(pr, nblk); }

struct LaunchShape {
    int wide, gs_floats, stages, W, atoms, slot_rows;
    size_t smem;
};

// lead: the plan whose tile choices hold for the launch.
LaunchShape launch_shape(const TcPlan* lead, TcPlan* const* plans, int n) {
    LaunchShape L{};
    L.wide = plans[0]->nblk > 1;
    // single block: G, and in FP32 mode L of its diagonal blocks; groups: scales
    if (L.wide) {
        L.gs_floats = 64 + 128;
    } else {
        int r2max = 0;
        for (int m = 0; m < n; ++m) r2max = std::max(r2max, 2 * plans[m]->N);
        L.gs_floats = r2max * (r2max + 1) + (plans[0]->mode == 0 ? 2 * kRows : 0);
    }
    L.slot_rows = 8;
    int min_box = kRows;      // the MMA reads 128 rows from a tile: reserve the excess past the ring
    for (int m = 0; m < n; ++m) {
        L.slot_rows = std::max(L.slot_rows, plans[m]->box_rows);
        min_box = std::min(min_box, plans[m]->box_rows);
    }
    const size_t slot = (size_t)L.slot_rows * plans[0]->row_bytes;
    // + the rows an MMA reads past the ring's last slot
    const size_t vstage = L.wide ? (size_t)8 * 16 * kVRow * sizeof(float2) : 0;
    const size_t fixed = 1024 + (size_t)L.gs_floats * 4 + vstage + 16 + 16 + 8 * (2 * 16 + 5) + 256 +
                         (size_t)(kRows - min_box) * plans[0]->row_bytes;
    auto fit = [&](int atoms) {
        const size_t sb = (size_t)plans[0]->planes * atoms * slot * (L.wide ? 2 : 1);
        return std::min<int>(16, (int)((kSmemBudget - fixed) / sb));
    };
    // k-tiles per stage, unless set: as many (up to 256 spectra: 8 k-tiles of
    // 32, or 4 of the FP8 mode's 128) as still leave 3 stages -- each stage
    // handshake costs a fixed latency
    L.atoms = lead->atoms;
    if (!L.atoms) {
        L.atoms = 1;
        for (int at = plans[0]->KT == 32 ? 8 : 4; at > 1; at /= 2)
            if (fit(at) >= 3) {
                L.atoms = at;
                break;
            }
    }
    while (L.atoms > 1 && fit(L.atoms) < 2) L.atoms /= 2;
    const size_t stage_bytes =
        (size_t)plans[0]->planes * L.atoms * slot * (L.wide ? 2 : 1);
    const int smax = fit(L.atoms);
    // default depth: as many stages as fit, up to 8; FP32 mode with one
    // antenna block, which streams its workspace from HBM at the copy rate,
    // takes 3 (at N = 44 a 1 s integration's pass: 0.92 ms against 0.95 with
    // the 4 that fit, 1.03 with 2)
    const int sdef = plans[0]->mode == 0 && !L.wide ? 3 : 8;
    L.stages = lead->stages ? std::min(lead->stages, smax) : std::min(smax, sdef);
    const int step = plans[0]->KT * L.atoms;
    // default window: 256 spectra in FP32 mode (TMEM accumulation bias ~1e-6
    // at full size); 512 for FP16 (its input rounding dominates), 1024 when
    // a mode has several antenna blocks (~10% less time per pass at N = 256;
    // at N = 44 it raised the 1 s FP16 error from 5.7e-6 to 8.1e-6 for no
    // gain); 2048 for FP8 (16 k-tiles of 128 spectra, the MMA steps of a
    // 1024-spectrum FP16 window: 30% less time per pass than 1024 at
    // N = 256, 13% at N = 44, against an input rounding error near 1e-2)
    const int W0 = plans[0]->mode == 0 ? 256 : plans[0]->mode == 2 ? 2048 : (L.wide ? 1024 : 512);
    int W = lead->window ? lead->window : std::max(W0, plans[0]->KT);
    L.W = (W + step - 1) / step * step;   // windows hold whole stages
    L.smem = fixed + (size_t)L.stages * stage_bytes;
    return L;
}

// Ranges into which the passes of n modes are cut, S_pad frames each: the
// counts that minimise the busiest of the SMs in a simulated round-robin deal
// of every mode's items to single CTAs, in units of a k-tile: the tiles, 4
// more for an item's end and 2 when its partial is combined with others.  (A
// group counts there as one A block against two B blocks each, one unit per
// tile loaded and one.)  Ranges are summed in FP32 and combined in FP64, so
// their number also bounds the rounding of a pass, for every deal below: CTA
// pairs would gain by fewer cuts only where a pass is short (100 antennas, K =
// 512, 2048 spectra FP16 60 us whole, 79 and 8 to combine in two; 128, 4096
// spectra FP32 mode 268 against 244 and 11; 200, K = 16, 30000 spectra FP32
// mode 244 against 154 and 10).
RangePlan pass_ranges(TcPlan* const* plans, int n, const int64_t* S_pad) {
    std::vector<int64_t> key;
    for (int m = 0; m < n; ++m) key.insert(key.end(), {S_pad[m], plans[m]->N, plans[m]->C, plans[m]->max_split});
    auto& cache = plans[0]->range_cache;
    for (auto& e : cache)
        if (e.first == key) return e.second;
    const int sms = plans[0]->num_sms;
    int64_t max_tiles = 1;
    for (int m = 0; m < n; ++m) max_tiles = std::max<int64_t>(max_tiles, S_pad[m] / plans[m]->KT);
    std::vector<int> best(n, 1);
    double best_score = 1e300;
    std::vector<double> load(sms);
    for (int64_t T = 1; T <= max_tiles * 2; T *= 2) {
        std::vector<int> sp(n);
        for (int m = 0; m < n; ++m) {
            const int64_t tiles = std::max<int64_t>(1, S_pad[m] / plans[m]->KT);
            int64_t ns = (tiles + T - 1) / T;
            ns = std::min<int64_t>(ns, plans[m]->max_split);
            const int64_t per = (tiles + ns - 1) / ns;
            sp[m] = (int)((tiles + per - 1) / per);
        }
        std::fill(load.begin(), load.end(), 0.0);
        int64_t g = 0;
        for (int m = 0; m < n; ++m) {
            const TcPlan* p = plans[m];
            const int64_t tiles = std::max<int64_t>(1, S_pad[m] / p->KT);
            const int64_t per = (tiles + sp[m] - 1) / sp[m];
            for (int s = 0; s < sp[m]; ++s) {
                const int64_t t = std::min<int64_t>(per, tiles - (int64_t)s * per);
                for (int k = 0; k < p->C; ++k)
                    for (int b1 = 0; b1 < p->nblk; ++b1)
                        for (int b2 = b1; b2 < p->nblk; b2 += 2, ++g) {
                            const int w = p->nblk == 1 ? 2 : std::min(2, p->nblk - b2) + (b2 != b1) + 1;
                            load[g % sms] += (double)t * 0.5 * w + 4.0 + (sp[m] > 1 ? 2.0 : 0.0);
                        }
            }
        }
        const double score = *std::max_element(load.begin(), load.end());
        if (score < best_score - 1e-9) {
            best_score = score;
            best = sp;
        }
    }
    cache.emplace_back(key, RangePlan{best, best_score});
    if (cache.size() > 16) cache.erase(cache.begin());
    return RangePlan{best, best_score};
}

// Work deal of one launch.  Round-robin: items go to the workers in turn, each
// pass cut into `least` ranges (pass_ranges of the step's `total` modes), or,
// single blocks, those of the launch's own modes where they are more.  Balanced
// (a single-block mode alone): contiguous shares of the weighted k-tiles (see
// next_piece), taken when cheaper in pass_ranges' cost model.  At N = 44, K =
// 512 and 8192 frames per pass the round-robin deal leaves 104 CTAs with two
// channels and 48 with one; the balanced deal gives each 1.7 channels.
DealPlan choose_deal(const TcPlan* lead, TcPlan* const* plans, int n, const int64_t* S_pad, int total,
                     const RangePlan& least) {
    DealPlan out;
    out.sp.resize(n);
    if (lead->split > 0) {
        // fixed by corr_set_tiles: round-robin, ranges per channel, at most one per k-tile
        for (int m = 0; m < n; ++m) {
            const int64_t tiles = std::max<int64_t>(1, S_pad[m] / plans[m]->KT);
            out.sp[m] = (int)std::min<int64_t>(std::min(lead->split, plans[m]->max_split), tiles);
        }
        return out;
    }
    if (plans[0]->nblk > 1) {
        out.sp.assign(least.sp.begin(), least.sp.begin() + n);
        return out;
    }
    TcPlan* const p = plans[0];
    if (total == 1)
        for (auto& e : p->deal_cache)
            if (e.first == S_pad[0]) return e.second;
    const RangePlan own = pass_ranges(plans, n, S_pad);
    out.sp = own.sp;
    if (total > 1) {
        for (int m = 0; m < n; ++m) out.sp[m] = std::max(own.sp[m], least.sp[m]);
        return out;
    }
    const int sms = p->num_sms;
    // balanced deal: every CTA gets U/G units; an item then spans at most
    // (tiles - 1) w G / U + 2 CTAs, which must fit the partial slots, and a
    // CTA holds at least 3 units (more than a k-tile's 2), so it owns a k-tile of
    // every item it overlaps and an item's CTAs are consecutive
    // (one mode only: with several, the round-robin deal spreads every mode's
    // items, whose ends differ in cost, evenly over the CTAs -- measured
    // faster on the four-mode batch)
    // (single antenna block only: with several, the round-robin deal hands one
    // channel's block pairs to neighbouring CTAs at once, which then share its
    // tiles through L2; contiguous shares would read them from HBM per pair)
    const int64_t tiles = S_pad[0] / p->KT;
    const int w = host_pair_units(0, 1);
    const int64_t units = item_units(tiles, w) * p->C;
    if (units > 0 && p->max_split >= 3) {
        int64_t G = sms;
        const int64_t span = (tiles - 1) * w;
        if (span > 0)
            G = std::min<int64_t>(G, std::max<int64_t>(1, (int64_t)(p->max_split - 2) * units / span));
        G = std::min<int64_t>(G, std::max<int64_t>(1, units / 3));
        std::vector<double> bl(G, 0.0);
        int64_t ibase = 0;
        for (int k = 0; k < p->C; ++k, ibase += item_units(tiles, w)) {
            const int64_t t0 = ibase + kEndUnits;
            const int64_t first = t0 * G / units;
            const int64_t last = (t0 + span) * G / units;
            for (int64_t j = 0; j < tiles; ++j) bl[(t0 + j * w) * G / units] += 0.5 * w;
            for (int64_t c = first; c <= last; ++c) bl[c] += 4.0 + (last > first ? 2.0 : 0.0);
        }
        if (*std::max_element(bl.begin(), bl.end()) < own.score - 1e-9) {
            out.balanced = true;
            out.grid = (int)G;
            out.units = units;
        }
    }
    p->deal_cache.emplace_back(S_pad[0], out);
    if (p->deal_cache.size() > 16) p->deal_cache.erase(p->deal_cache.begin());
    return out;
}

}  // namespace

namespace {

// One kernel for plans that all have one antenna block, or all several.
int launch_set(TcPlan* lead, TcPlan* const* plans, int n, TcRun* const* runs, int total,
               const RangePlan& least, cudaStream_t st, std::string& err) {
    std::vector<int64_t> S(n);
    for (int m = 0; m < n; ++m) S[m] = runs[m]->S_pad;
    const DealPlan deal = choose_deal(lead, plans, n, S.data(), total, least);
    const std::vector<int>& sp = deal.sp;
    const LaunchShape L = launch_shape(lead, plans, n);
    TcArgs a;
    memset(&a, 0, sizeof a);
    a.n_modes = n;
    a.stages = L.stages;
    a.KT = plans[0]->KT;
    a.kt_shift = a.KT == 128 ? 7 : 5;
    a.row_bytes = plans[0]->row_bytes;
    a.W = L.W;
    a.atoms = L.atoms;
    a.gs_floats = L.gs_floats;
    a.slot_rows = L.slot_rows;
    a.status = runs[0]->status;
    a.timeout_ns = lead->timeout_ns;
    if (lead->withhold) {
        a.withhold = 1;
        a.timeout_ns = lead->hook_timeout_ns;
        lead->withhold = 0;
    }
    int base = 0;
    int64_t units = 0;
    for (int m = 0; m < n; ++m) {
        const TcPlan* p = plans[m];
        a.tmap[m] = p->tmap;
        TcModeArgs& d = a.md[m];
        d.N = p->N;
        d.C = p->C;
        d.P = p->P;
        d.nblk = p->nblk;
        d.npairs = p->npairs;
        d.S_pad = runs[m]->S_pad;
        const int64_t tiles = std::max<int64_t>(1, d.S_pad / p->KT);
        const int64_t per = (tiles + sp[m] - 1) / sp[m];
        d.S_item = per * p->KT;
        d.n_split = d.S_pad > 0 ? (int)((d.S_pad + d.S_item - 1) / d.S_item) : 0;
        d.item_base = base;
        d.n_items = d.n_split * p->npairs * p->C;
        base += d.n_items;
        d.partial = runs[m]->partial;
        d.acc = runs[m]->acc;
        d.ticket = plans[m]->ticket;
        d.scale = runs[m]->scale;
        d.split = runs[m]->split;
        d.assign = runs[m]->assign;
        d.tiles = d.S_pad / p->KT;
        d.cap_tiles = (int)(p->cap / p->KT);
        d.box_bytes = (uint32_t)p->box_rows * p->row_bytes;
        d.unit_base = units;
        for (int pr = 0; pr < p->npairs; ++pr)
            units += item_units(d.tiles, host_pair_units(pr, p->nblk)) * p->C;
        // single block: ranges are combined inside the kernel, into acc;
        // several blocks: each range lands in its partial slot (coalesced FP32
        // stores), and one reduction launch combines them
        runs[m]->direct = p->nblk == 1;
        runs[m]->n_split = d.n_split;
    }
    a.total_items = base;
    // (largest dividend of the deal: units x CTAs plus a divisor)
    a.u32 = (units + 1) * (plans[0]->num_sms + 1) < ((int64_t)1 << 32);
    if (base == 0) return CORR_OK;
    int grid = L.wide ? 2 * std::min(base, plans[0]->num_sms / 2) : std::min(base, plans[0]->num_sms);
    if (deal.balanced) {
        a.balanced = 1;
        a.units = units;
        grid = deal.grid;
    }
    cudaError_t e;
    auto go = [&](auto kern) {
        cudaError_t r = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)L.smem);
        if (r != cudaSuccess) return r;
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute pair[1];
        pair[0].id = cudaLaunchAttributeClusterDimension;
        pair[0].val.clusterDim.x = 2;
        pair[0].val.clusterDim.y = pair[0].val.clusterDim.z = 1;
        cfg.gridDim = dim3(grid);
        cfg.blockDim = dim3(kTcThreads);
        cfg.dynamicSmemBytes = L.smem;
        cfg.stream = st;
        cfg.attrs = pair;
        cfg.numAttrs = L.wide ? 1 : 0;
        return cudaLaunchKernelEx(&cfg, kern, a);
    };
    if (plans[0]->mode == 0)
        e = L.wide ? go(xengine_tc_kernel<0, true>) : go(xengine_tc_kernel<0, false>);
    else if (plans[0]->mode == 1)
        e = L.wide ? go(xengine_tc_kernel<1, true>) : go(xengine_tc_kernel<1, false>);
    else
        e = L.wide ? go(xengine_tc_kernel<2, true>) : go(xengine_tc_kernel<2, false>);
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e != cudaSuccess) {
        err = std::string("tensor-core X-engine launch: ") + cudaGetErrorString(e);
        return CORR_ECUDA;
    }
    return CORR_OK;
}

}  // namespace

int tc_launch(TcPlan* const* plans, int n, TcRun* runs, cudaStream_t st, std::string& err, int* launches) {
    if (launches) *launches = 0;
    if (n < 1 || n > kMaxTcModes) {
        err = "between 1 and 4 modes per tensor-core launch";
        return CORR_EINVAL;
    }
    for (int m = 0; m < n; ++m) {
        if (!plans[m]->have_map) {
            err = "tensor-core plan has no workspace";
            return CORR_ESTATE;
        }
        if (plans[m]->mode != plans[0]->mode) {
            err = "modes of one tensor-core launch must share the X-engine precision";
            return CORR_EINVAL;
        }
    }
    // Modes of one antenna block and modes of several take a kernel each (CTA
    // pairs share their MMAs, and one kernel's tcgen05 code is of one
    // cta_group).  The lead's set goes first: a test hook on it fires there.
    TcPlan* set[kMaxTcModes];
    TcRun* srun[kMaxTcModes];
    int64_t S[kMaxTcModes];
    for (int m = 0; m < n; ++m) S[m] = runs[m].S_pad;
    RangePlan all;                     // (a lone single-block mode has its deal at hand)
    if (plans[0]->split == 0 && (n > 1 || plans[0]->nblk > 1)) all = pass_ranges(plans, n, S);
    const bool wide0 = plans[0]->nblk > 1;
    for (int pass = 0; pass < 2; ++pass) {
        int ns = 0;
        RangePlan least;
        for (int m = 0; m < n; ++m)
            if ((plans[m]->nblk > 1) == (wide0 == (pass == 0))) {
                if (!all.sp.empty()) least.sp.push_back(all.sp[m]);
                set[ns] = plans[m];
                srun[ns++] = &runs[m];
            }
        if (!ns) continue;
        const int rc = launch_set(plans[0], set, ns, srun, n, least, st, err);
        if (rc != CORR_OK) return rc;
        if (launches) ++*launches;
    }
    return CORR_OK;
}

int tc_test_withhold(TcPlan* p, double wait_limit_s, std::string& err) {
    if (!(wait_limit_s >= 0.001 && wait_limit_s <= 10.0)) {
        err = "wait limit must be in [0.001, 10] s";
        return CORR_EINVAL;
    }
    p->withhold = 1;
    p->hook_timeout_ns = (unsigned long long)(wait_limit_s * 1e9);
    return CORR_OK;
}

void tc_plan_destroy(TcPlan* p) {
    if (!p) return;
    cudaFree(p->ticket);
    delete p;
}

}  // namespace gbcorr
