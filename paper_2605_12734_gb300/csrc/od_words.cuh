// od_words.cuh -- the tile sweep over a field of fixed-point words
// (od_arith.cuh), what the default arithmetic runs: fused, persistent and
// per-chare launches, 3D 7-point and 2D 5-point.
//
// The words make the update a chain of integer adds and roundings, about half
// the instructions of the sweep over doubles (od_tile.cuh), so what held that
// sweep back next -- a CTA barrier on every plane, and one warp delayed each
// plane by issuing copies and patching the x halo -- would bound this one.
// Here the CTA is specialised by warp instead: NT compute threads and one
// producer warp.  The producer takes tiles (by ticket where its CTA has several),
// waits for their dependencies, issues the bulk copies of their planes into
// the ring, patches each landed plane's x halo, and hands the plane over; the
// compute warps release a slot when they have read it.  No barrier joins the
// compute warps, so they drift apart by up to the ring, and the producer runs
// ahead into the next tile while the current one is computed: the ticket, the
// dependency wait, the table reads and the first copies of a tile are hidden.
//
// Barriers (mbarriers in shared memory, S ring slots):
//   full[s]    the slot's bulk copies have landed (transaction bytes); the
//              producer waits on it
//   ready[s]   the slot holds its plane with its x halo (one arrival, the
//              producer's); the compute warps wait on it
//   empty[s]   every compute warp has read the slot; the producer waits
//   told[i]    the tile record i (of two) is written; the compute warps wait
//   taken[i]   every compute warp has finished that tile; the producer waits
// Measured at 512^3 in 4096 chares (128 x 4, persistent), ms a step: 0.640 the
// sweep over doubles, 0.565 that sweep over words, 0.597 this one with a
// producer that alternates strictly between issuing and finishing planes,
// 0.541 event-driven, 0.524 with one 256-byte record per tile instead of five
// dependent table reads, 0.489 with 6 ring slots (0.456 with the roundings left
// out), 0.460 with rows of whole sectors (od_plan.cpp), 0.443 with 256 x 4, 0.441 with
// conversions that select (od_arith.cuh).  Two-dimensional,
// 16384^2: 0.76 to 0.65.  What bounds it: at 32^3 chares the traffic (2.39 GB a
// step, 0.79 of the copy bandwidth) and the ALU pipe (62 % busy, issue 67 %)
// together; in two dimensions the copy bandwidth (0.99 of it).  A fused step on
// the same case: 0.553 with a fixed stride of tiles per CTA, 0.480 by ticket.
// Tried and slower: each thread's own cells of three planes kept in registers
// (80 registers, five CTAs), publishing a tile from the producer (its fence
// waits for the whole SM's stores), a full fence after the dependency wait
// (+6000 cycles a tile), nanosleep in the producer's loop, taking the next
// ticket earlier than the last plane's issue.
//
// Every wait is bounded, and no lane leaves its warp alone.  Whoever runs into
// a limit on a phase raises `stop`, which ends every other such wait of the
// CTA, and its warp records the error; a dependency wait that runs out records
// the error and ends the CTA's tiles.  Copies in flight are left to no
// one: the producer waits, bounded, for them before it leaves.
#pragma once
#include "od_plan.h"
#include "od_tile.cuh"

namespace od {
namespace tile {

// fx_round (od_arith.cuh) of two sums: the four binary32 operations as two
// packed ones, which take half the issue slots.
__device__ __forceinline__ void fx_round_pair(uint64_t &F0, uint64_t &F1, uint32_t &z0, uint32_t &z1) {
    const uint32_t c0 = mad_lo(top_bit((uint32_t)(F0 >> 32)), 1u << 23, 0u - (19u << 23));
    const uint32_t c1 = mad_lo(top_bit((uint32_t)(F1 >> 32)), 1u << 23, 0u - (19u << 23));
    asm("{\n\t.reg .b64 x, c;\n\t"
        "mov.b64 x, {%2, %3};\n\t"
        "mov.b64 c, {%4, %5};\n\t"
        "add.rn.f32x2 x, x, c;\n\t"
        "sub.rn.f32x2 x, x, c;\n\t"
        "mov.b64 {%0, %1}, x;\n\t}\n"
        : "=r"(z0), "=r"(z1)
        : "r"((uint32_t)F0 & 0x007FFFFFu), "r"((uint32_t)F1 & 0x007FFFFFu), "r"(c0), "r"(c1));
    F0 &= ~(uint64_t)0x007FFFFFu;
    F1 &= ~(uint64_t)0x007FFFFFu;
}

// fx_div6's quotient and the position of its high word's top bit (20..27 in
// the window, 0xFFFFFFFF for a zero quotient).
__device__ __forceinline__ uint64_t fx_div6_top(uint64_t F, uint32_t &t) {
    uint32_t qh;
    const uint64_t q = fx_div6(F, qh);
    t = top_bit(qh);  // the one fx_div6 computed
    return q;
}

constexpr int kMaxStages = 8;

struct WordsShared {
    uint64_t full[kMaxStages], ready[kMaxStages], empty[kMaxStages], told[2], taken[2];
    struct Tile {
        double *dst;     // cell slot offsets count from here in each destination plane
        int32_t plane;   // doubles from one destination plane to the next
        int32_t pitch;   // doubles from one row to the next
        int32_t bx, n;   // cells of a row, cells of a plane of the tile
        int32_t cell0;   // slot offset of a row's first cell
        int32_t nk;      // planes to compute
        int32_t tile;    // -1: no more tiles
        int32_t done;    // what its step counter says when it is done (persistent)
    } t[2];
    uint32_t finished[2];  // compute warps that have finished the tile (persistent)
    TileRec rec[2];      // the producer's: its tile's record and the next one's
    uint32_t stop;
};
static_assert(sizeof(WordsShared) <= words_static_smem(128), "the planner's figure for it");

// Wait for a phase of `bar`, until it is there, the limit runs out or the CTA
// stops.  The hardware suspends a try for a while by itself; the clock and the
// stop word are looked at only between groups of tries, because reading the
// clock takes longer than most waits.
// A lane tries, reads the clock and reads the stop word for itself, so lanes of
// one warp may differ in why they came back.  None acts on that alone: the one
// that ran into the limit raises the stop word and goes on with its warp, which
// asks `stopped` together before anything relies on the wait.
__device__ __forceinline__ void wait_phase(uint64_t *bar, uint32_t parity, uint32_t *stop, uint64_t limit_ns) {
    if (mbar_try_wait(bar, parity)) return;
    uint64_t t0 = 0;
    for (;;) {
#pragma unroll 1
        for (int k = 0; k < 32; ++k)
            if (mbar_try_wait(bar, parity)) return;
        if (*(volatile uint32_t *)stop != 0u) return;
        const uint64_t t = now_ns();
        if (t0 == 0) t0 = t;
        if (t - t0 > limit_ns) {
            *(volatile uint32_t *)stop = 1u;
            return;
        }
    }
}

// Whether the CTA stops: one answer for a whole warp (all lanes together).
__device__ __forceinline__ bool stopped(const uint32_t *stop) {
    return __any_sync(0xFFFFFFFFu, *(const volatile uint32_t *)stop != 0u);
}

__device__ __forceinline__ bool mbar_test(uint64_t *bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}\n"
        : "=r"(ok)
        : "r"(smem_addr(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

__device__ __forceinline__ void mbar_arrive(uint64_t *bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(bar)) : "memory");
}

// Adds 1 to a counter in shared memory; what the other warps wrote before
// their counts is then visible here.
__device__ __forceinline__ uint32_t count_acq_rel(uint32_t *p) {
    uint32_t old;
    asm volatile("atom.acq_rel.cta.shared::cta.add.u32 %0, [%1], 1;" : "=r"(old) : "r"(smem_addr(p)) : "memory");
    return old;
}

// ---------------------------------------------------------------- compute warps

// The cells of a warp's plane that have an operand or a quotient outside the
// window (`rare`: this lane may have some), with IEEE operations: they are
// numbered over the warp and dealt to its lanes, so that a few scattered ones
// take one call instead of one for each of a thread's cells (the first step
// from a uniform random field, 2 % of the cells, 512^3 in 64^3 chares: 1.31 ms
// without, 1.07 with it; 40 steps from a cold 200^3 field 3.88 and 3.48).
// Out of line: 64^3 chares in 256 x 4 0.427 ms a step, inlined 0.433.
constexpr int kRedoWarps = 16;  // of a CTA of up to 512 compute threads
static_assert(kRedoWarps * 32 * 4 <= words_static_smem(256) - words_static_smem(128), "the planner's figure for it");

// This warp's list: one array for every N that a kernel calls words_redo with.
__device__ __forceinline__ int32_t *redo_list() {
    __shared__ int32_t lists[kRedoWarps][32];
    return lists[threadIdx.x >> 5];
}

template <int N>
struct Offsets {
    int r[N];
};

template <int ST, int N>
static __device__ __noinline__ void words_redo(const double *sd, const double *sc, const double *su, double *dpl,
                                               Offsets<N> rf, int pitch, uint32_t e0, bool rare) {
    constexpr bool k3D = ST == OD_STENCIL_3D7;
    int32_t *list = redo_list();
    const uint32_t lane = threadIdx.x & 31u, below = (1u << lane) - 1u;
    uint32_t number[N], total = 0;
#pragma unroll
    for (int m = 0; m < N; ++m) {
        const int r = rf.r[m];
        bool bad = rare;
        if (bad && e0 != 0u) {
            const uint64_t w = f64_bits(sc[r - 1]), e = f64_bits(sc[r + 1]), d = f64_bits(sd[r]), u = f64_bits(su[r]);
            uint64_t x = w | e | d | u, sum = w + e + d + u;
            if (k3D) {
                const uint64_t v = f64_bits(sc[r - pitch]), n = f64_bits(sc[r + pitch]);
                x |= v | n;
                sum += v + n;
            }
            // a quotient below 2^52 needs a sum below that times the divisor;
            // the margin covers the roundings on the way (a cell redone in
            // vain gets the same bits)
            bad = (uint32_t)(x >> 32) >= kFxEnd || (sum != 0u && sum < ((k3D ? 6ull : 4ull) << 52) + 4096u);
        }
        const uint32_t mask = __ballot_sync(0xFFFFFFFFu, bad);
        number[m] = bad ? total + (uint32_t)__popc(mask & below) : 0xFFFFFFFFu;
        total += (uint32_t)__popc(mask);
    }
#pragma unroll 1
    for (uint32_t base = 0; base < total; base += 32u) {
#pragma unroll
        for (int m = 0; m < N; ++m)
            if (number[m] - base < 32u) list[number[m] - base] = rf.r[m];
        __syncwarp();
        if (base + lane < total) {
            const int r = list[lane];
            dpl[r] = k3D ? update_slow_fx(sd + r, sc + r, su + r, pitch, e0) : update2d_slow_fx(sd + r, sc + r, su + r, e0);
        }
        __syncwarp();
    }
}

// One thread's cells of plane k, whose planes below, of and above it lie in the
// ring slots sd, sc and su: cell m is q = tid + m*NT of the tile's plane,
// row-major, at slot offset rf[m] (a cell past the end repeats cell 0: the
// same value to the same place).  Cells are worked on in pairs, whose roundings
// share packed binary32 operations.  The window is checked once for all of
// them; the cells of a plane that fails it are redone with IEEE operations, out
// of line.  All lanes of a warp call it together.
// N: how many of the CPT cells to do, the first ones.  DEAL: redo through
// words_redo (otherwise each lane its own cells).
template <int CPT, int ST, bool DEAL, int N = CPT>
__device__ __forceinline__ void words_plane(const double *sd, const double *sc, const double *su, double *dpl,
                                            const int (&rf)[CPT], int pitch, uint32_t e0) {
    constexpr bool k3D = ST == OD_STENCIL_3D7;
    constexpr int W = N == 1 ? 1 : 2;
    // bits of every operand's high word, and the lowest top bit of a quotient
    uint32_t any = e0 == 0u ? kFxEnd : 0u, low = 0xFFFFFFFFu;
#pragma unroll
    for (int m = 0; m < N; m += W) {
        uint64_t F[2], b[2][4];
        uint32_t z[2];
#pragma unroll
        for (int u = 0; u < W; ++u) {
            const int r = rf[m + u];
            const uint64_t w = f64_bits(sc[r - 1]), e = f64_bits(sc[r + 1]);
            any |= (uint32_t)((w | e) >> 32);
            if (k3D) {
                b[u][0] = f64_bits(sc[r - pitch]);
                b[u][1] = f64_bits(sc[r + pitch]);
                any |= (uint32_t)((b[u][0] | b[u][1]) >> 32);
            }
            b[u][k3D ? 2 : 0] = f64_bits(sd[r]);
            b[u][k3D ? 3 : 1] = f64_bits(su[r]);
            any |= (uint32_t)((b[u][k3D ? 2 : 0] | b[u][k3D ? 3 : 1]) >> 32);
            F[u] = w + e;
        }
        constexpr int kAdds = k3D ? 4 : 2;  // adds after W + E
#pragma unroll
        for (int t = 0; t <= kAdds; ++t) {
            if constexpr (W == 2) {
                fx_round_pair(F[0], F[1], z[0], z[1]);
            } else {
                const FxRounded r = fx_round(F[0]);
                F[0] = r.a;
                z[0] = r.z;
            }
#pragma unroll
            for (int u = 0; u < W; ++u) F[u] = t < kAdds ? F[u] + z[u] + b[u][t < kAdds ? t : 0] : F[u] + z[u];
        }
#pragma unroll
        for (int u = 0; u < W; ++u) {
            uint32_t top;
            uint64_t q;
            if (k3D) {
                q = fx_div6_top(F[u], top);
            } else {
                q = F[u] >> 2;
                top = top_bit((uint32_t)(q >> 32));
            }
            dpl[rf[m + u]] = f64_from(q);
            low = top < low ? top : low;
        }
    }
    const bool rare = any >= kFxEnd || low < 20u;
    if constexpr (DEAL) {
        if (__any_sync(0xFFFFFFFFu, rare)) {
            Offsets<N> o;
#pragma unroll
            for (int m = 0; m < N; ++m) o.r[m] = rf[m];
            words_redo<ST, N>(sd, sc, su, dpl, o, pitch, e0, rare);
        }
    } else if (rare) {
#pragma unroll
        for (int m = 0; m < N; ++m) {
            const int r = rf[m];
            uint64_t x = f64_bits(sc[r - 1]) | f64_bits(sc[r + 1]) | f64_bits(sd[r]) | f64_bits(su[r]);
            if (k3D) x |= f64_bits(sc[r - pitch]) | f64_bits(sc[r + pitch]);
            const uint32_t q = (uint32_t)(f64_bits(dpl[r]) >> 32);
            if (e0 == 0u || (uint32_t)(x >> 32) >= kFxEnd || q - 1u < (1u << 20) - 1u)
                dpl[r] = k3D ? update_slow_fx(sd + r, sc + r, su + r, pitch, e0) : update2d_slow_fx(sd + r, sc + r, su + r, e0);
        }
    }
}

template <int NT, int CPT, int ST, bool PUBLISH>
__device__ __forceinline__ void words_compute(const KArgs &a, WordsShared &sh, const double *ring) {
    // dealing needs a few registers, which only the larger CTAs have to spare
    // (128 x 4 spills with it: 32^3 chares 0.481 instead of 0.460 ms a step)
    constexpr bool kDeal = NT >= 256;
    const int tid = threadIdx.x, lane = tid & 31;
    const int S = a.stages, SD = a.stage_doubles;
    const uint32_t e0 = a.fmt->base;
    const uint64_t limit = 4u * a.spin_ns;  // the producer's own waits come first
    uint32_t sl = 0, ph = 0;                // the next plane's slot and phase
    auto advance = [&]() {
        if (++sl == (uint32_t)S) {
            sl = 0;
            ph ^= 1u;
        }
    };
    for (uint32_t n = 0;; ++n) {
        const uint32_t i = n & 1u;
        wait_phase(&sh.told[i], (n >> 1) & 1u, &sh.stop, limit);
        if (stopped(&sh.stop)) {
            if (lane == 0) record_err(a.err, OD_ERR_TMA_TIMEOUT, -1, -1);  // (the first error stays)
            break;
        }
        const int tile = sh.t[i].tile;
        if (tile < 0) break;
        const int pitch = sh.t[i].pitch, plane = sh.t[i].plane;
        int rf[CPT];
        int busy = 2;  // two cells a thread: how many cells a lane has that are not past the tile's end in the whole warp
        {
            const int bx = sh.t[i].bx, nc = sh.t[i].n, cell0 = sh.t[i].cell0;
#pragma unroll
            for (int m = 0; m < CPT; ++m) {
                const int q0 = tid + m * NT;
                const int q = q0 < nc ? q0 : 0;
                if (ST == OD_STENCIL_3D7) {
                    const int j = q / bx;
                    rf[m] = (j + 1) * pitch + cell0 + (q - j * bx);
                } else {
                    rf[m] = cell0 + q;
                }
            }
            if (CPT == 2) busy = (nc - (tid & ~31) + NT - 1) / NT;
        }
        // the planes below the first computed one and that one
        uint64_t *held_d = &sh.empty[sl];  // the slots of planes k-1 and k
        const double *sd = ring + (size_t)sl * SD;
        wait_phase(&sh.ready[sl], ph, &sh.stop, limit);
        advance();
        uint64_t *held_c = &sh.empty[sl];
        const double *sc = ring + (size_t)sl * SD;
        wait_phase(&sh.ready[sl], ph, &sh.stop, limit);
        double *dpl = sh.t[i].dst;
        // A warp whose wait ends without its phase goes on to the tile's end:
        // it reads slots that may be half filled and stores into the tile's own
        // cells of a context that has failed, and the tile is not published.
        // (A vote on every wait instead: 512^3 in 32^3 chares 0.448 ms a step,
        // 0.443 with this.)
        for (int left = sh.t[i].nk; left > 0; --left) {
            advance();
            const double *su = ring + (size_t)sl * SD;
            wait_phase(&sh.ready[sl], ph, &sh.stop, limit);
            // In the shapes of two cells a thread, which narrow planes get, a
            // warp past the plane's end has nothing to do and one in its last
            // part one cell (5195 x 7129 in 83-cell rows: 0.392 / 0.318 ms a
            // step).  With four cells the second form spills: 32^3 chares ran
            // 0.60 instead of 0.48 ms.
            if (CPT != 2 || busy > 1) words_plane<CPT, ST, kDeal>(sd, sc, su, dpl, rf, pitch, e0);
            else if (busy > 0) words_plane<CPT, ST, kDeal, CPT == 2 ? 1 : CPT>(sd, sc, su, dpl, rf, pitch, e0);
            __syncwarp();
            if (lane == 0) mbar_arrive(held_d);
            held_d = held_c;
            held_c = &sh.empty[sl];
            sd = sc;
            sc = su;
            dpl += plane;
        }
        if (stopped(&sh.stop)) {
            if (lane == 0) record_err(a.err, OD_ERR_TMA_TIMEOUT, tile, -1);
            break;
        }
        if (lane == 0) {
            mbar_arrive(held_d);
            mbar_arrive(held_c);
        }
        advance();
        if (lane == 0) {
            // The last warp to finish publishes the tile: the warps' stores
            // come before their counts, those before its own (acquire), and
            // the release puts them before the step counter for every CTA.
            if (PUBLISH && count_acq_rel(&sh.finished[i]) == NT / 32 - 1) {
                sh.finished[i] = 0u;
                if ((int64_t)tile != a.stall_tile) st_release(a.epoch + tile, sh.t[i].done);
            }
            mbar_arrive(&sh.taken[i]);
        }
    }
}

// ---------------------------------------------------------------- producer warp

// An x-halo item of a computed plane: its ring-slot offset and the source
// pointer of plane -1 (the neighbour's boundary column), null at a domain face.
struct HaloItem {
    const double *src;
    int32_t plane;  // doubles from one plane of the source to the next
    int32_t off;
};

template <int ST, bool FUSED>
__device__ __forceinline__ HaloItem halo_item(const TileRec &R, int sp, int t) {
    HaloItem h = {nullptr, 0, 0};
    if (!FUSED || t >= 2 * R.rows) return h;
    const bool hi = t >= R.rows;
    const int j = hi ? t - R.rows : t;
    const double *base = hi ? R.xhi[sp] : R.xlo[sp];
    h.plane = hi ? R.xhi_plane : R.xlo_plane;
    if (base) h.src = base + (int64_t)j * (hi ? R.xhi_pitch : R.xlo_pitch);
    h.off = ST == OD_STENCIL_3D7 ? (j + 1) * R.pitch + R.cell0 + (hi ? R.bx : -1) : R.cell0 + (hi ? R.cells : -1);
    return h;
}

template <int NT, int CPT, int ST, bool FUSED, bool PERSIST>
__device__ __forceinline__ void words_produce(const KArgs &a, WordsShared &sh, double *ring) {
    const int lane = threadIdx.x & 31;
    const int S = a.stages, SD = a.stage_doubles;
    uint32_t si = 0, pe = 1;  // next slot to issue; phase of its release (1: the first use waits for none)
    uint32_t sf = 0, pf = 0;  // next slot to finish; phase of its copies
    int in_flight = 0;        // planes issued and not finished
    int err = 0, etile = -1, estep = -1;
    // The next tile is looked up while the current one is handed over, in
    // stages of one memory latency each: 1 its ticket, 2 its record (8 bytes
    // per lane), 3 the step counters it depends on, 4 all of them far enough
    // (5: not yet).
    int stage = 0, ticket = 0;
    int tile = -1, step = -1, sp = a.parity, r = 0;  // the tile at hand: index, step, source parity, step of the launch
    int ntile = -1, nr = 0;                          // the next one
    uint64_t word = 0;
    int32_t seen = 0;
    auto look_up = [&](uint32_t n) {  // one stage for tile number n of this CTA
        if (stage == 0) {
            // Tickets: on the persistent path every tile of every step; in a
            // fused step those past the grid's, whose CTAs take their own
            // first (a step of few tiles then waits for no counter).  Each CTA
            // draws until one is past the end, so the last draw's number is
            // known, and it leaves the counter at zero for the next launch.
            if (lane == 0 && (PERSIST || (FUSED && n > 0u && a.tile_count > (int)gridDim.x))) {
                ticket = atomicAdd(a.queue, 1);
                if (ticket == (PERSIST ? a.iters * a.ntiles + (int)gridDim.x : a.tile_count) - 1) *a.queue = 0;
            }
            stage = 1;
        } else if (stage == 1) {
            ntile = -1;
            if (PERSIST) {
                const uint32_t tk = (uint32_t)__shfl_sync(0xFFFFFFFFu, ticket, 0);  // below 2^31
                if (tk < (uint32_t)a.iters * (uint32_t)a.ntiles) {
                    nr = (int)(tk / (uint32_t)a.ntiles);
                    int pos = (int)(tk - (uint32_t)nr * (uint32_t)a.ntiles);
                    if (a.order_mode == 1 && (nr & 1)) pos = a.ntiles - 1 - pos;
                    ntile = a.order ? a.order[pos] : pos;
                }
            } else {
                int64_t tk = (int64_t)blockIdx.x + (int64_t)n * gridDim.x;
                if (FUSED && n > 0u && a.tile_count > (int)gridDim.x)
                    tk = (int64_t)gridDim.x + __shfl_sync(0xFFFFFFFFu, ticket, 0);
                if (tk < a.tile_count) ntile = a.tile_begin + (int)tk;
            }
            if (ntile >= 0) word = reinterpret_cast<const uint64_t *>(a.rec + ntile)[lane];
            stage = ntile >= 0 ? 2 : 4;
        } else if (stage == 2) {
            reinterpret_cast<uint64_t *>(&sh.rec[n & 1u])[lane] = word;
            __syncwarp();
            const TileRec &N = sh.rec[n & 1u];
            stage = 4;
            if (PERSIST) {
                if (N.ndep <= 19) seen = lane < N.ndep ? ld_acquire(a.epoch + N.dep[lane]) : INT32_MAX;
                stage = 3;
            }
        } else if (stage == 3) {
            // once only: further looks wait until the tile's turn, so that
            // they do not hold up the planes of the current one
            stage = sh.rec[n & 1u].ndep <= 19 && __all_sync(0xFFFFFFFFu, seen >= nr) ? 4 : 5;
        }
    };
    for (uint32_t n = 0;; ++n) {
        const uint32_t i = n & 1u;
        while (stage < (PERSIST ? 3 : 4)) look_up(n);
        tile = ntile;
        r = nr;
        const TileRec &R = sh.rec[i];
        if (PERSIST && tile >= 0) {
            step = a.t0 + r;
            sp = step & 1;
            // Wait until every tile this one reads has finished step r-1, each
            // lane watching its share of the list (a tile of this CTA is
            // published by its compute warps).
            if (stage != 4) {
                const int nd = R.ndep;
                const int32_t *more = nd > 19 ? a.dep_idx + R.dep[0] : nullptr;
                int q = lane;
                uint64_t t0 = 0;
                for (uint32_t k = 1;; ++k) {
                    while (q < nd && ld_acquire(a.epoch + (more ? more[q] : R.dep[q])) >= r) q += 32;
                    if (__all_sync(0xFFFFFFFFu, q >= nd)) break;
                    if (k % 16u == 0u) {
                        const uint64_t t = now_ns();
                        if (t0 == 0) t0 = t;
                        const bool late = t - t0 > a.spin_ns;
                        if (__any_sync(0xFFFFFFFFu, late)) {
                            if (lane == 0) record_err(a.err, OD_ERR_DEP_TIMEOUT, tile, step);
                            tile = -1;
                            break;
                        }
                        if (__any_sync(0xFFFFFFFFu, ld_relaxed(&a.err->code) != 0)) {
                            tile = -1;
                            break;
                        }
                    }
                    __nanosleep(32);
                }
            }
            // Each lane has acquired the counters it watched, and a vote orders
            // no memory: the barrier puts every lane's acquire before lane 0's
            // copies and the other lanes' halo loads.
            __syncwarp();
            // data written by other CTAs (generic proxy) is next read by bulk
            // copies (async proxy)
            asm volatile("fence.proxy.async.global;" ::: "memory");
        }
        stage = 0;
        if (n >= 2) wait_phase(&sh.taken[i], ((n >> 1) - 1u) & 1u, &sh.stop, 2u * a.spin_ns);
        if (stopped(&sh.stop)) {
            err = OD_ERR_TMA_TIMEOUT;
            break;
        }
        if (tile < 0) {  // no more tiles (or an error somewhere): the compute warps leave too
            if (lane == 0) {
                sh.t[i].tile = -1;
                mbar_arrive(&sh.told[i]);
            }
            break;
        }
        etile = tile;
        estep = step;
        const int plane = R.plane;
        const int kf = R.k0, kb = kf - 1, ke = kf + R.nk;  // planes kb..ke are copied, kf..ke-1 computed
        if (lane == 0) {
            WordsShared::Tile &t = sh.t[i];
            t.dst = R.own[sp ^ 1] + (int64_t)(kf + 1) * plane;
            t.plane = plane;
            t.pitch = R.pitch;
            t.bx = R.bx;
            t.cell0 = R.cell0;
            t.n = R.cells;
            t.nk = R.nk;
            t.tile = tile;
            t.done = r + 1;
            mbar_arrive(&sh.told[i]);
        }
        const uint32_t row_bytes = (uint32_t)R.pitch * 8u, run_bytes = (uint32_t)R.run;
        // (lane 0) the copies of plane p into slot s
        auto issue = [&](int p, uint32_t s) {
            uint64_t *bar = &sh.full[s];
            double *to = ring + (size_t)s * SD;
            mbar_expect_tx(bar, run_bytes);
            if (FUSED && p < 0 && R.zlo[sp]) {  // the z- neighbour's top plane
                bulk_g2s(to, R.zlo[sp], run_bytes, bar);
                return;
            }
            if (FUSED && p >= R.bz && R.zhi[sp]) {  // the z+ neighbour's bottom plane
                bulk_g2s(to, R.zhi[sp], run_bytes, bar);
                return;
            }
            const double *row0 = R.own[sp] + (int64_t)(p + 1) * plane;
            if (ST == OD_STENCIL_3D7) {
                // a computed plane's y-ghost rows come from the y neighbours
                const bool computed = p >= kf && p < ke;
                const double *ylo = R.ylo[sp], *yhi = R.yhi[sp];
                uint32_t bytes = run_bytes;
                double *at = to;
                if (FUSED && computed && ylo) {
                    bulk_g2s(to, ylo + (int64_t)(p + 1) * R.ylo_plane, row_bytes, bar);
                    at += R.pitch;
                    row0 += R.pitch;
                    bytes -= row_bytes;
                }
                if (FUSED && computed && yhi) {
                    // (with the ghosts apart, its first two words hold the
                    // last row's x+ ghost, this chare's)
                    const uint32_t lead = R.cell0 == 4 ? 2u : 0u;
                    bulk_g2s(to + (size_t)(R.rows + 1) * R.pitch + lead, yhi + (int64_t)(p + 1) * R.yhi_plane + lead,
                             row_bytes - 8u * lead, bar);
                    bytes -= row_bytes - 8u * lead;
                }
                bulk_g2s(at, row0, bytes, bar);
            } else {
                bulk_g2s(to, row0, run_bytes, bar);
            }
        };
        // this lane's first two x-halo items, their values loaded a plane ahead
        // (from L2: other SMs wrote them); tiles of more than 32 rows load the
        // rest when they need them
        const int nhalo = FUSED ? 2 * R.rows : 0;
        const HaloItem h0 = halo_item<ST, FUSED>(R, sp, lane), h1 = halo_item<ST, FUSED>(R, sp, lane + 32);
        double x0 = 0.0, x1 = 0.0;
        auto fetch = [&](int p) {
            if (p < kf || p >= ke) return;
            if (h0.src) x0 = __ldcg(h0.src + (int64_t)(p + 1) * h0.plane);
            if (h1.src) x1 = __ldcg(h1.src + (int64_t)(p + 1) * h1.plane);
        };
        // issue a plane whenever its slot is free, finish the oldest issued one
        // whenever it has landed, whichever can be done
        int pnew = kb, pold = kb;  // next plane to issue, to finish
        uint64_t t0 = 0;
        uint32_t idle = 0;
        fetch(kf);
        while (pold <= ke) {
            bool moved = false;
            if (pnew <= ke && __all_sync(0xFFFFFFFFu, mbar_test(&sh.empty[si], pe))) {
                if (lane == 0) {
                    fence_proxy_async_smem();  // after the halo's generic stores into the slot
                    issue(pnew, si);
                }
                ++pnew;
                ++in_flight;
                if (++si == (uint32_t)S) {
                    si = 0;
                    pe ^= 1u;
                }
                moved = true;
            }
            if (in_flight > 0 && __all_sync(0xFFFFFFFFu, mbar_test(&sh.full[sf], pf))) {
                --in_flight;
                if (FUSED && pold >= kf && pold < ke) {
                    double *to = ring + (size_t)sf * SD;
                    if (h0.src) to[h0.off] = x0;
                    if (h1.src) to[h1.off] = x1;
                    for (int t = lane + 64; t < nhalo; t += 32) {
                        const HaloItem h = halo_item<ST, FUSED>(R, sp, t);
                        if (h.src) to[h.off] = __ldcg(h.src + (int64_t)(pold + 1) * h.plane);
                    }
                    __syncwarp();
                    fetch(pold + 1);
                }
                if (lane == 0) mbar_arrive(&sh.ready[sf]);
                ++pold;
                if (++sf == (uint32_t)S) {
                    sf = 0;
                    pf ^= 1u;
                }
                moved = true;
            }
            if (pnew > ke && stage < 4) {
                look_up(n + 1u);
                continue;
            }
            if (moved) {
                idle = 0;
                t0 = 0;
                continue;
            }
            // nothing to do: let the hardware suspend the warp for a while
            if (in_flight > 0) mbar_try_wait(&sh.full[sf], pf);
            else mbar_try_wait(&sh.empty[si], pe);
            if (++idle == 64u) {  // look at the clock now and then
                idle = 0;
                const uint64_t t = now_ns();
                if (t0 == 0) t0 = t;
                const bool late = t - t0 > 2u * a.spin_ns || *(volatile uint32_t *)&sh.stop != 0u;
                if (__any_sync(0xFFFFFFFFu, late)) {
                    err = OD_ERR_TMA_TIMEOUT;
                    break;
                }
            }
        }
        if (err) break;
    }
    if (err) {
        if (lane == 0) {
            record_err(a.err, err, etile, estep);
            *(volatile uint32_t *)&sh.stop = 1u;
        }
        // copies still in flight land before the CTA's shared memory is given up
        for (; in_flight > 0; --in_flight) {
            mbar_wait_bounded(&sh.full[sf], pf, drain_limit(a.spin_ns));
            if (++sf == (uint32_t)S) {
                sf = 0;
                pf ^= 1u;
            }
        }
    }
}

// ---------------------------------------------------------------- kernels

// NT compute threads and the producer warp (the last one).  FUSED: faces read
// from the neighbours' arrays; PERSIST: all steps in one launch, tiles by
// ticket (see k_persistent).  FUSED alone draws one step's tiles by ticket too;
// a per-chare launch has its tiles in turn, gridDim.x apart.  The registers
// allow words_ctas CTAs per SM (od_plan.h).
template <int NT, int CPT, bool FUSED, bool PERSIST, int ST>
__global__ void __launch_bounds__(NT + 32, words_ctas(NT, CPT, ST == OD_STENCIL_3D7)) k_words(const KArgs a) {
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ WordsShared sh;
    if (blockDim.x != NT + 32 || a.stages < 3 || a.stages > kMaxStages) {
        if (threadIdx.x == 0) record_err(a.err, OD_ERR_BAD_LAUNCH, -1, -1);
        return;
    }
    double *ring = reinterpret_cast<double *>(smem + kSmemRing);
    if (threadIdx.x == 0) {
        for (int s = 0; s < kMaxStages; ++s) {
            mbar_init(&sh.full[s], 1);
            mbar_init(&sh.ready[s], 1);
            mbar_init(&sh.empty[s], NT / 32);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(&sh.told[i], 1);
            mbar_init(&sh.taken[i], NT / 32);
            sh.finished[i] = 0u;
        }
        sh.stop = 0u;
        mbar_init_fence();
    }
    __syncthreads();
    if (threadIdx.x >= NT)
        words_produce<NT, CPT, ST, FUSED, PERSIST>(a, sh, ring);
    else
        words_compute<NT, CPT, ST, PERSIST>(a, sh, ring);
}

}  // namespace tile
}  // namespace od
