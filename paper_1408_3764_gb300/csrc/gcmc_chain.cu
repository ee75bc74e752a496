// gcmc_chain.cu -- the grand canonical Markov chain run entirely on the
// device (Sec. 2 and Algorithm 1), with the concurrent evaluation of
// upcoming moves that the paper lists as future work (Sec. 5: run multiple
// moves concurrently), here inside one CTA.
//
// One CTA owns one chain.  Its warps have two roles:
//
//  * W movers: mover k owns the moves k, k + W, k + 2 W, ...  It evaluates a
//    move alone and ahead of its turn: it reads the configuration as it
//    stands when it starts (after c0 committed moves; the particle pick uses
//    the counts predicted at the move's turn) and produces the trial, its
//    energy change dU over the 27 neighbour cells (Algorithms 6 and 7; the
//    union of both neighbourhoods for a displacement into an adjacent cell),
//    the error scale uabs, and the Metropolis decision (Eqs. 3-5, textbook
//    sign of mu) for each particle count its turn can meet.  Then it waits
//    for its turn, checking each move that is committed meanwhile: one that
//    put, removed or moved a particle within rc of the trial, touched its
//    old cell or its record, or one that changes the particle the counts
//    pick, makes it evaluate again (at once, before its turn).  At its turn
//    the mover takes the decision for the actual count, applies an accepted
//    move (Sec. 3.2.5: swap-with-last removal, append, species index refill)
//    and passes the turn on.  A decision inside the FP32 error band is taken
//    on a trial recomputed in FP64.  Every decision is therefore the one the
//    sequential chain takes;
//  * the keeper (the last warp) keeps the FP64 running energy, the averages,
//    the counters and the trace.
//
// What bounds it: the turn passes through every move, so a chain cannot run
// faster than one hand-over per move (a poll of shared memory, the checks, the
// stores of an accepted move and a fence; 700-1,800 cycles, the more the more
// moves are accepted), and it runs at (evaluation + hand-over) / W when that
// is longer (an evaluation takes 7,000-16,000 cycles: dependent shared-memory,
// shuffle and L2 latencies, 1,500-2,500 warp instructions).  One warp per
// move leaves the set-up (trial, cells, sums) unreplicated, and W evaluations
// in flight hide its latency.  Measured against two teams of six warps that
// evaluated a move together and a separate committing warp: 10^4 moves of
// 2,048 particles in FP64 23.0 -> 8.0 ms (8.5 before the shorter FP64 pair
// term), 2*10^4 of 131,072 in FP32 29.9 -> 15.6 ms, the 64-chain isotherm step
// 223 -> 126 ms.
//
// The microcell chain (Sec. 3.3.3) is the same kernel with the evaluation over
// the cube of microcells and both lists kept: 4,000 moves of 87,296 particles in
// FP32 19.2 -> 7.9 ms against a block of eight warps that evaluated and
// committed one move after another.  Its counters stay in global memory.
//
// Movers hand the turn on through shared memory with block-scope fences;
// every wait is bounded and sets a timeout status instead of hanging.  Cell
// counters live in shared memory (uint16) for the whole launch; particle data
// stays in the padded cell-major layout in L1/L2.
//
#include <algorithm>
#include <climits>
#include <cmath>
#include <cstring>
#include <string>
#include <vector>

#include "gcmc_ctx.h"
#include "gcmc_stage.cuh"

namespace gcmc {

struct ChainOut {
    long long attempted[3];
    long long accepted[3];
    long long flagged;
    long long moves_done;
    double energy;
    double sum_energy;
    double sum_n;
    long long n[kMaxSpecies];
    int status;
    // why the chain stopped: waits that gave up (1 room in the book, 2 the turn, 4
    // the keeper); 8 an evaluation begun at its turn does not hold, 16 capacity or a
    // record missing from its cell, 32 the species' last record missing
    int pad;
    long long reevaluated;  // moves evaluated more than once
    long long refines;      // trials decided in FP64 after the FP32 band test
    double virial;          // running virial after the last move (virial runs)
    double sum_virial;      // sum over the moves of the running virial
    unsigned long long t0, t1;  // global timer (ns) when the chain's CTA started and finished
    unsigned long long prof[12];  // SM clock cycles by role (gcmc_chain_profile)
};

struct ChainArgs {
    uint64_t seed;
    uint64_t first;
    int n_moves;
    uint32_t chain;
    int movers;  // W
    int T;
    int ncell;
    int cap;
    long long maxN;
    int S;
    unsigned long long R2;
    float r2hi;  // FP32 squared distances above it are outside the cutoff
    unsigned long long thr_disp, thr_ins;
    uint32_t span;  // 2 D + 1 grid steps
    int D;          // displacement half-width in grid steps
    double beta, lnV;
    double logz[kMaxSpecies];
    double tol;  // relative tolerance that defines "near the threshold"
    float beta_f, tol_f;  // beta and tol in FP32 (the FP32 Metropolis test)
    unsigned long long wait_ns;  // limit of every wait (kWaitNs unless a test shortens it)
    int stall_at;  // diagnostic: the mover waits on a flag nothing sets at this move (-1 none)
    int virial;  // also keep the running virial sum_{i<j} r U'(r)
    float lnzv_f[kMaxSpecies];
    FieldF ff;
    FieldD fd;
    uint4 *cell_pos;
    int32_t *cell_count;
    uint4 *pos_by_id;
    // the microcell list (microcell launches): M per side, cubes of nax per
    // side reaching D each way, mcap slots of ncm records
    int M, nax, mD, mcap;
    uint32_t ncm;
    uint8_t *mc_count;
    uint4 *mc_pos;
    int64_t *d_n;
    double *d_energy;
    gcmc_trace *trace;
    ChainOut *out;
};

constexpr int kChainWarps = 16;              // movers and the keeper
constexpr int kMaxMovers = kChainWarps - 1;
constexpr int kRS = 32;                      // log, book and outlook rings (at least 2 kMaxMovers)
constexpr int kWords = 16;                   // moves a mover draws the words of at once
constexpr int kQ = 128;                      // a mover's queue of pairs: at most 31 + 64 wait
// a mover's dynamic shared memory: queue, words and the work cells, or -- in a
// microcell launch -- the records of kMcGroup microcells
constexpr int kMcGroup = 128;
constexpr int kMoverBytes = kQ * 16 + kWords * 48 + 64 * 16;
constexpr int kMicroMoverBytes = kQ * 16 + kWords * 48 + kMcGroup * kMicroMaxCap * 4;
constexpr unsigned long long kWaitNs = 1000000000ull;  // a wait gives up after 1 s (default)
static_assert(kRS >= 2 * kMaxMovers, "ring entries of moves that can still be read");

constexpr uint32_t kOld = 1u, kNew = 2u;
constexpr int kStatusMicroOverflow = 64;  // a move needs a full microcell

// ---------------------------------------------------------------- trials
struct Trial {
    uint4 Po, Pn;          // old / new position; Po.w = the particle's tag (~0 for insertions)
    int co, cn;            // cells (-1 when absent)
    int idx;               // particle index (-1: none)
    int px, py, pz;        // old cell (insertions: the new one)
    int qx, qy, qz;        // new cell
    int type, s;
    bool possible, cross, far;  // cross: the cell changes; far: to a cell that is not adjacent
};

__device__ __forceinline__ bool near1(int d, int T)
{
    d = d < 0 ? -d : d;
    return d <= 1 || d == T - 1;
}

__device__ __forceinline__ int wrapc(int x, int T) { return x < 0 ? x + T : (x >= T ? x - T : x); }

// 1 << d, 0 for d outside 0 .. 31
__device__ __forceinline__ uint32_t bit_at(int d)
{
    uint32_t r;
    asm("shl.b32 %0, 1, %1;" : "=r"(r) : "r"(d));
    return r;
}

// ---------------------------------------------------------------- shared state
struct __align__(16) WordRec {
    uint32_t w[8];
    float lnu;  // FP32 ln(u) of the acceptance uniform; NaN: decide in FP64
    int pad[3];
};

// SM clock for the cycle counters of a profiled launch; an unprofiled
// launch compiles the reads (and the sums) away.
template <bool PROF>
__device__ __forceinline__ unsigned long long prof_clock()
{
    if constexpr (PROF) return clock64();
    else return 0ull;
}

// What a move changes if it is accepted, for the checks of the moves after
// it.  A mover writes its entry as soon as its evaluation is in, so that
// later moves are tested against it before its turn; sh.ver says for which
// move and evaluation it stands.
struct __align__(16) LogRec {
    int4 ids;     // x, y: cells written; z, w: (s << 24) | index of the records written (-1 none)
    uint4 pos0;   // .w: bit 0 a second position, bit 1 a moved entry, bit 2 an insertion, species << 8
    uint4 pos1;
    uint4 moved;  // the cell's last entry, moved into the freed slot
};

struct __align__(16) BookRec {  // mover -> keeper
    double dU64, lnA;  // dU when decided in FP64 or evaluated in FP64 mode
    double dW;         // virial change of the trial (virial runs)
    double uab;
    float hi, lo;      // dU = hi + lo otherwise
    // bit 0 accepted, 1 possible, 2 dU64 holds dU, 3 near the threshold, 4
    // decided in FP64, 5 evaluated again; type << 8, species << 16
    int bits;
    int index;
    int n;             // N_s before the move
    int ready;         // move + 1
    int pad[2];
};
constexpr int kBkAcc = 1, kBkPossible = 2, kBkUse64 = 4, kBkNear = 8, kBkRefined = 16, kBkAgain = 32;

struct __align__(16) Shared {
    // the turn: x = moves committed, y = whether the last 32 of them were
    // accepted (bit 0 the last one) -- written together -- z = 1 once the
    // chain stops
    int4 turn;
    LogRec logs[kRS];
    BookRec book[kRS];
    float4 field[kMaxSpecies * kMaxSpecies];  // FP32 mode: (c4e, sig2, c4e_lo, sig2_lo); FP64 pairs read ChainArgs::fd
    int ver[kRS];      // of the log entries: (move << 8) | evaluation, 0 while one is written
    int outlook[kRS];  // of pending moves: (move << 8) | species << 2 | 1 (adds a particle) or 2 (removes one)
    int n[kMaxSpecies];
    int booked;    // moves the keeper has processed
    int status;
    int where;     // which waits gave up
    int gone;      // movers that have finished
    int never;     // a flag nothing sets (the diagnostic stall waits on it)
    // 1 while this chain accepts most of its insertions [0] / deletions [1]
    // (the bet the count prediction makes on moves not yet evaluated)
    int likely[2];
    long long evaluations;
    unsigned long long prof[12];
};

__device__ __forceinline__ int vload(const int &x) { return *(volatile const int *)&x; }
__device__ __forceinline__ void vstore(int &x, int v) { *(volatile int *)&x = v; }
__device__ __forceinline__ int cload(const uint16_t &x) { return *(volatile const uint16_t *)&x; }
__device__ __forceinline__ void cstore(uint16_t &x, int v) { *(volatile uint16_t *)&x = (uint16_t)v; }
// Counters in global memory, shared by the warps of one block.
__device__ __forceinline__ int gload(const int32_t *p)
{
    int v;
    asm volatile("ld.relaxed.cta.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void gstore(int32_t *p, int v)
{
    asm volatile("st.relaxed.cta.global.s32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ int gload(const uint8_t *p)
{
    uint32_t v;
    asm volatile("ld.relaxed.cta.global.u8 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return (int)v;
}
__device__ __forceinline__ void gstore(uint8_t *p, int v)
{
    asm volatile("st.relaxed.cta.global.u8 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ void fence_cta() { asm volatile("fence.acq_rel.cta;" ::: "memory"); }

__device__ __forceinline__ int4 turn_load(const Shared &sh)
{
    int4 v;
    asm volatile("ld.volatile.shared.v4.s32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "r"(smem_addr(&sh.turn))
                 : "memory");
    return v;
}
__device__ __forceinline__ void turn_store(Shared &sh, int c, uint32_t hist)
{
    asm volatile("st.volatile.shared.v2.s32 [%0], {%1, %2};" ::"r"(smem_addr(&sh.turn)), "r"(c), "r"((int)hist)
                 : "memory");
}

// Stops the chain: no further move is committed.
__device__ __noinline__ void chain_stop(Shared &sh, int status, int where)
{
    atomicOr(&sh.status, status);
    if (where) atomicOr(&sh.where, where);
    fence_cta();
    *(volatile int *)&sh.turn.z = 1;
}

// |a - p| along an axis, the minimum image as an unsigned 32-bit distance.
__device__ __forceinline__ uint32_t axis_dist(uint32_t a, uint32_t p)
{
    const uint32_t d = a - p;
    return min(d, 0u - d);
}

// ---------------------------------------------------------------- a mover
// Sums of an evaluation: dU = e + el in FP32, de in FP64; uabs; virial change.
struct Sums {
    float e, el, ua, w;
    double de, da, dw;
};

// The words of moves m, m + W, ... (at most kWords of them below n): lane l
// draws block l & 1 of the (l >> 1)-th.  (Out of line, as what follows: rare
// code is kept out of the loop, which has to stay in the instruction cache.)
__device__ __noinline__ void fill_words(const ChainArgs &a, WordRec *words, int m, int lane)
{
    const long long mk = (long long)m + (long long)(lane >> 1) * a.movers;
    __syncwarp();
    if (mk < a.n_moves) {
        const uint64_t mv = a.first + (uint64_t)mk;
        const uint4 r = philox_block(make_uint4((uint32_t)mv, (uint32_t)(mv >> 32), a.chain, (uint32_t)(lane & 1)),
                                     make_uint2((uint32_t)a.seed, (uint32_t)(a.seed >> 32)));
        WordRec &W = words[lane >> 1];
        ((uint4 *)W.w)[lane & 1] = r;
        if (lane & 1) {
            const uint64_t k53 = ((uint64_t)(r.z >> 5) << 26) | (uint64_t)(r.w >> 6);
            float l;
            if (k53 == 0) l = -INFINITY;                                   // u = 0: always accept
            else if (k53 < (1ull << 27)) l = __int_as_float(0x7fc00000);  // u < 2^-26: decide in FP64
            else l = logf((float)((double)k53 * 1.1102230246251565404e-16));
            W.lnu = l;
        }
    }
    __syncwarp();
}


// The slot of `tag` in a cell of n entries (-1: not there), and in lane (n - 1)
// & 31 the last entry; v: the lane's entry of the first 32.
struct Found {
    int at;
    uint4 last;
};
__device__ __noinline__ Found find_far(const uint4 *cell, uint32_t tag, int n, uint4 v, int lane)
{
    Found r = {-1, v};
#pragma unroll 1
    for (int b = 0; b < n; b += 32) {
        const bool have = b + lane < n;
        if (b > 0 && have) v = cell[b + lane];
        const unsigned hit = __ballot_sync(0xffffffffu, have && v.w == tag);
        if (hit && r.at < 0) r.at = b + __ffs(hit) - 1;
        if (b + lane == n - 1) r.last = v;
    }
    return r;
}

// The record of particle (s, i), its cell and its slot there (at its turn only).
struct Entry {
    uint4 Q;
    int cell, slot;
};
template <bool MICRO>
__device__ __noinline__ Entry find_now(const ChainArgs &a, const uint16_t *cnt, int s, int i, int lane)
{
    Entry r;
    r.Q = a.pos_by_id[(long long)s * a.maxN + i];
    r.cell = cell_of(r.Q.x, r.Q.y, r.Q.z, a.T);
    const int n = MICRO ? gload(a.cell_count + r.cell) : cload(cnt[r.cell]);
    const uint4 *cell = a.cell_pos + (long long)r.cell * a.cap;
    uint4 v = make_uint4(0, 0, 0, 0);
    if (lane < n) v = cell[lane];
    r.slot = find_far(cell, r.Q.w, n, v, lane).at;
    return r;
}

// A microcell's entries as a warp sees them: its count, the lane's entry and
// the slot of `tag` (-1: not there).
struct MicroEntry {
    int n, slot;
    uint4 v;
};
__device__ __forceinline__ MicroEntry micro_find(const ChainArgs &a, uint32_t c, uint32_t tag, int lane)
{
    MicroEntry r;
    r.n = __shfl_sync(0xffffffffu, gload(a.mc_count + c), 0);
    fence_cta();
    r.v = make_uint4(0, 0, 0, 0);
    if (lane < r.n) r.v = a.mc_pos[(long long)lane * a.ncm + c];
    r.slot = __ffs(__ballot_sync(0xffffffffu, lane < r.n && r.v.w == tag)) - 1;
    return r;
}
__device__ __forceinline__ uint32_t micro_of(const uint4 &p, int M)
{
    return (uint32_t)((cell_coord(p.z, (uint32_t)M) * M + cell_coord(p.y, (uint32_t)M)) * M + cell_coord(p.x, (uint32_t)M));
}

// The decision in FP64: accepted, near the threshold, ln A.
struct Decision {
    int bits;
    double lnA;
};
__device__ __noinline__ Decision decide_f64(const ChainArgs &a, uint32_t w6, uint32_t w7, int type, int s, int ns,
                                            double de, double da)
{
    const double lnu = log(uniform53(w6, w7));
    double lnK = 0.0;
    if (type != 0) {
        lnK = log((double)(type == 1 ? ns + 1 : ns));
        if (type == 1) lnK = a.logz[s] + a.lnV - lnK;
        else lnK = lnK - a.logz[s] - a.lnV;
    }
    Decision d;
    d.lnA = lnK - a.beta * de;
    const double band = a.beta * a.tol * da + 1e-12 * (1.0 + fabs(d.lnA));
    d.bits = (lnu < d.lnA ? kBkAcc : 0) | (fabs(lnu - d.lnA) <= band ? kBkNear : 0);
    return d;
}

// A bounded wait's expiry, the same in every lane; stops the chain.
__device__ __forceinline__ bool gave_up(const ChainArgs &a, Shared &sh, Wait &wt, int where)
{
    if (!__any_sync(0xffffffffu, wt.expired(a.wait_ns))) return false;
    if ((threadIdx.x & 31) == 0) chain_stop(sh, kStatusTimeout, where);
    __syncwarp();
    return true;
}

// Room in the keeper's book for move m (false: the chain stopped).
__device__ __noinline__ bool wait_room(const ChainArgs &a, Shared &sh, int m)
{
    Wait wt;
    for (;;) {
        const int room = m < vload(sh.booked) + kRS, st = vload(sh.turn.z);
        if (__shfl_sync(0xffffffffu, room, 0)) return true;
        if (__shfl_sync(0xffffffffu, st, 0) || gave_up(a, sh, wt, 1)) return false;
        __nanosleep(40);
    }
}

// The diagnostic stall: a bounded wait on a flag nothing sets runs out,
// and the chain stops before this move with a timeout status.
__device__ __noinline__ bool wait_never(const ChainArgs &a, Shared &sh)
{
    Wait wt;
    for (;;) {
        const int go = vload(sh.never), st = vload(sh.turn.z);
        if (__shfl_sync(0xffffffffu, go, 0)) return true;
        if (__shfl_sync(0xffffffffu, st, 0) || gave_up(a, sh, wt, 2)) return false;
    }
}

template <bool MICRO>
struct Mover {
    const ChainArgs &a;
    Shared &sh;
    uint16_t *cnt;
    int4 *q;         // kQ queued pairs: separation, pair index | 0x100 for a term that counts negatively
    WordRec *words;  // kWords
    int4 *tab;       // 64 work cells: record offset (2 words), flags; microcells: record offsets
    uint4 *cell_pos;
    unsigned long long R2;
    float r2hi;
    int lane, T, S, cap;
    int k27;  // this lane's cell of the 27: (dx + 1) | (dy + 1) << 8 | (dz + 1) << 16

    // The particle that the counts pick (Algorithm 1; idx = -1 if there is
    // none); lane q < S holds species q's count.
    __device__ __forceinline__ void pick(const uint32_t *w, int type, int nq, int &s, int &idx) const
    {
        idx = -1;
        s = type ? (int)__umulhi(w[5], (uint32_t)S) : 0;
        if (type == 1) return;
        int N = __shfl_sync(0xffffffffu, nq, s);
        if (type == 0) {
#pragma unroll 1
            for (int k = 1; k < S; ++k) N += __shfl_sync(0xffffffffu, nq, k);
        }
        if (N <= 0) return;
        idx = pick_index((uint32_t)N, w, type);
        if (type == 0) {
#pragma unroll 1
            for (;;) {
                const int n = __shfl_sync(0xffffffffu, nq, s);
                if (idx < n || s + 1 >= S) break;
                idx -= n;
                ++s;
            }
        }
    }

    // the counters: in shared memory, with microcells in global memory (the
    // evaluation does not read them there)
    __device__ __forceinline__ int count(int c) const { return MICRO ? gload(a.cell_count + c) : cload(cnt[c]); }
    __device__ __forceinline__ void set_count(int c, int n) const
    {
        if (MICRO) gstore(a.cell_count + c, n);
        else cstore(cnt[c], n);
    }

    __device__ __forceinline__ int cell_at(int x, int y, int z) const
    {
        return (wrapc(z, T) * T + wrapc(y, T)) * T + wrapc(x, T);
    }

    // The cells a trial visits (its work list), 0 .. n - 1: the 27 around its
    // cell (no cell change, insertions, deletions); for a displacement into
    // an adjacent cell the union of the old and new neighbourhoods, 3 or 4
    // values per axis, each cell flagged kOld and/or kNew (cells of the union
    // box in neither neighbourhood carry no flag); for a longer displacement
    // the old 27 (kOld) followed by the new 27 (kNew).  At most 64 cells.
    // Per axis of a union, d in {-1, 0, 1} the change of the cell: the values
    // p - 1 - (d < 0) + i, i < 3 + |d|; boxes of three cells per side have
    // every value in both neighbourhoods.
    __device__ __forceinline__ int union_axis(int p, int q) const
    {
        int d = q - p;
        d = d > 1 ? -1 : (d < -1 ? 1 : d);
        return T == 3 ? 0 : d;
    }
    __device__ __forceinline__ void cross_cell(const Trial &t, int i, int &cell, uint32_t &fl) const
    {
        if (t.far) {
            const bool nw = i >= 27;
            const int k = nw ? i - 27 : i;
            cell = cell_at((nw ? t.qx : t.px) + k % 3 - 1, (nw ? t.qy : t.py) + k / 3 % 3 - 1,
                           (nw ? t.qz : t.pz) + k / 9 - 1);
            fl = nw ? kNew : kOld;
            return;
        }
        const int dx = union_axis(t.px, t.qx), dy = union_axis(t.py, t.qy), dz = union_axis(t.pz, t.qz);
        const int r = dx ? i >> 2 : i / 3, z = dy ? r >> 2 : r / 3;
        // offsets from the old cell
        const int ox = i - r * (dx ? 4 : 3) - 1 - (dx < 0), oy = r - z * (dy ? 4 : 3) - 1 - (dy < 0), oz = z - 1 - (dz < 0);
        cell = cell_at(t.px + ox, t.py + oy, t.pz + oz);
        fl = 0;
        if (max(max(abs(ox), abs(oy)), abs(oz)) <= 1) fl |= kOld;
        if (max(max(abs(ox - dx), abs(oy - dy)), abs(oz - dz)) <= 1) fl |= kNew;
        if (T == 3) fl = kOld | kNew;
    }

    // The trial's energy change.  The records of the work cells are numbered
    // cell after cell and taken 32 at a time, one per lane; the next 32 load
    // while the last are screened on the FP32 squared distance against a
    // bound just above rc^2.  Pairs that pass join the queue and are
    // evaluated 32 at a time, where the exact integer test decides, so the
    // long pair term (FP32: compensated, lj_ff; FP64) runs with every lane
    // busy and only on the ~15 % of records inside the cutoff.
    template <bool P32, bool VIR>
    __device__ __forceinline__ void evaluate(const Trial &t, Sums &o) const
    {
        o.e = o.el = o.ua = o.w = 0.f;
        o.de = o.da = o.dw = 0.0;
        if (!t.possible) return;
        if constexpr (MICRO && P32) {
            evaluate_micro32(t, o);
            return;
        }
        if constexpr (MICRO) evaluate_micro<VIR>(t, o);
        else evaluate_cells<P32, VIR>(t, o);
        if constexpr (P32) {
            const FF s = ff_warp_sum<false>(FF{o.e, o.el});  // (not finite: decided in FP64)
            o.e = s.hi;
            o.el = s.lo;
            o.ua = warp_sum(o.ua);
            if (VIR) o.w = warp_sum(o.w);
        } else {
            o.de = warp_sum(o.de);
            o.da = warp_sum(o.da);
            if (VIR) o.dw = warp_sum(o.dw);
        }
    }

    // Lowest cell of the cube around grid coordinate X (0 when the cube spans
    // the axis).
    __device__ __forceinline__ int cube_base(uint32_t X) const
    {
        return a.nax >= a.M ? 0 : cell_coord(X, (uint32_t)a.M) - a.mD;
    }
    // The change of a cube's base between two positions, as a wrapped difference.
    __device__ __forceinline__ int cube_shift(int d) const { return 2 * d > a.M ? d - a.M : (2 * d < -a.M ? d + a.M : d); }

    // The trial's energy change over the microcells (Sec. 3.3.3): the cube
    // around its position; for a displacement that moves the cube by at most
    // a cell per axis the union of both cubes, each record tested against
    // both positions; for a longer one the old cube, then the new one.
    // kMcGroup cells at a time: the lanes read their counts, number the
    // records and list them, and the records are taken 32 at a time as in
    // evaluate_cells.  FP64.
    template <bool VIR>
    __device__ __forceinline__ void evaluate_micro(const Trial &t, Sums &o) const
    {
        const unsigned lt = (1u << lane) - 1u;
        uint32_t *list = (uint32_t *)tab;
        const uint4 PA = t.type == 1 ? t.Pn : t.Po;
        int bx = cube_base(PA.x), by = cube_base(PA.y), bz = cube_base(PA.z);
        const int cx = cube_base(t.Pn.x), cy = cube_base(t.Pn.y), cz = cube_base(t.Pn.z);
        int nx = a.nax, ny = a.nax, nz = a.nax, sets = 1;
        if (t.type == 0) {
            const int dx = cube_shift(cx - bx), dy = cube_shift(cy - by), dz = cube_shift(cz - bz);
            if (max(max(abs(dx), abs(dy)), abs(dz)) > 1) {
                sets = 2;
            } else {
                bx += min(dx, 0);
                by += min(dy, 0);
                bz += min(dz, 0);
                nx += abs(dx);
                ny += abs(dy);
                nz += abs(dz);
            }
        }
        const uint32_t self = t.Po.w;
        const int wA = t.s * kMaxSpecies + (t.type == 1 ? 0 : 0x100), wB = t.s * kMaxSpecies;
        const uint32_t ix = 0xFFFFFFFFu / (uint32_t)nx + 1u, iy = 0xFFFFFFFFu / (uint32_t)ny + 1u;  // i / nx = umulhi(i, ix)
        const int n = nx * ny * nz;
        int head = 0, nq = 0;
        for (int set = 0; set < sets; ++set) {
            const bool testA = set == 0, testB = t.type == 0 && (sets == 1 || set == 1);
            if (set == 1) {
                bx = cx;
                by = cy;
                bz = cz;
            }
#pragma unroll 1
            for (int i0 = 0; i0 < n; i0 += kMcGroup) {
                uint32_t c[kMcGroup / 32];
                int k[kMcGroup / 32], mine = 0;
#pragma unroll
                for (int j = 0; j < kMcGroup / 32; ++j) {
                    const int i = i0 + 32 * j + lane;
                    c[j] = 0;
                    k[j] = 0;
                    if (i < n) {
                        const int r = nx == 1 ? i : (int)__umulhi((uint32_t)i, ix), z = ny == 1 ? r : (int)__umulhi((uint32_t)r, iy);
                        const int x = wrapc(bx + i - r * nx, a.M), y = wrapc(by + r - z * ny, a.M), w = wrapc(bz + z, a.M);
                        c[j] = (uint32_t)((w * a.M + y) * a.M + x);
                        k[j] = gload(a.mc_count + c[j]);
                    }
                }
#pragma unroll
                for (int j = 0; j < kMcGroup / 32; ++j) mine += k[j];
                fence_cta();  // the counts are read before the records they cover
                const int inc = warp_inclusive_scan(mine), P = __shfl_sync(0xffffffffu, inc, 31);
                int off = inc - mine;
                __syncwarp();
#pragma unroll
                for (int j = 0; j < kMcGroup / 32; ++j)
#pragma unroll 1
                    for (int q2 = 0; q2 < k[j]; ++q2) list[off++] = (uint32_t)q2 * a.ncm + c[j];
                __syncwarp();
                const bool final = set == sets - 1 && i0 + kMcGroup >= n;
                uint4 r = make_uint4(0, 0, 0, 0);
                bool have = lane < P;
                if (have) r = a.mc_pos[list[lane]];
#pragma unroll 1
                for (int base = 0; base < P || (final && nq > 0); base += 32) {
                    uint4 rn = r;
                    const bool next = base + 32 + lane < P;
                    if (next) rn = a.mc_pos[list[base + 32 + lane]];
                    if (have && r.w == self) have = false;  // the particle itself (no tag for an insertion)
                    if (testA) {
                        const int ex = (int)(PA.x - r.x), ey = (int)(PA.y - r.y), ez = (int)(PA.z - r.z);
                        const float gx = (float)ex, gy = (float)ey, gz = (float)ez;
                        const bool in = have && fmaf(gx, gx, fmaf(gy, gy, gz * gz)) < r2hi;
                        const unsigned b = __ballot_sync(0xffffffffu, in);
                        if (in) q[(head + nq + __popc(b & lt)) & (kQ - 1)] = make_int4(ex, ey, ez, wA + (int)tag_species(r.w));
                        nq += __popc(b);
                    }
                    if (testB) {
                        const int ex = (int)(t.Pn.x - r.x), ey = (int)(t.Pn.y - r.y), ez = (int)(t.Pn.z - r.z);
                        const float gx = (float)ex, gy = (float)ey, gz = (float)ez;
                        const bool in = have && fmaf(gx, gx, fmaf(gy, gy, gz * gz)) < r2hi;
                        const unsigned b = __ballot_sync(0xffffffffu, in);
                        if (in) q[(head + nq + __popc(b & lt)) & (kQ - 1)] = make_int4(ex, ey, ez, wB + (int)tag_species(r.w));
                        nq += __popc(b);
                    }
                    const bool last = final && base + 32 >= P;
#pragma unroll 1
                    while (nq >= 32 || (last && nq > 0)) {
                        const int cq = min(nq, 32);
                        __syncwarp();
                        if (lane < cq) pair_term<false, VIR>(q[(head + lane) & (kQ - 1)], o);
                        head += cq;
                        nq -= cq;
                        __syncwarp();
                    }
                    r = rn;
                    have = next;
                }
            }
        }
    }

    // The same in FP32: plain FP32 terms, whose order of addition is part of
    // the result to its last digits -- eight groups of 32 lanes stride over the
    // cells of the old cube and then the new one, four strides at a time, slot
    // by slot; a group's sums cross its lanes and are added in group order.
    // The warp takes the groups one after another; a step's counts are read
    // while the records of the step before it are evaluated.
    __device__ __forceinline__ void evaluate_micro32(const Trial &t, Sums &o) const
    {
        constexpr int kB = 4, kGroups = 8, kStride = 32 * kGroups;
        const int nax = a.nax, n3 = nax * nax * nax, total = (t.type == 0 ? 2 : 1) * n3;
        const uint4 P0 = t.type == 1 ? t.Pn : t.Po;
        const int bx = cube_base(P0.x), by = cube_base(P0.y), bz = cube_base(P0.z);
        const int cx = cube_base(t.Pn.x), cy = cube_base(t.Pn.y), cz = cube_base(t.Pn.z);
        const uint32_t ix = 0xFFFFFFFFu / (uint32_t)nax + 1u;  // i / nax = umulhi(i, ix), nax > 1
        uint32_t c[kB], cn[kB];
        int k[kB], kn[kB];
        auto counts = [&](int f0) {
#pragma unroll
            for (int j = 0; j < kB; ++j) {
                const int f = f0 + j * kStride;
                cn[j] = 0;
                kn[j] = 0;
                if (f < total) {
                    const bool side = f >= n3;
                    const int i = side ? f - n3 : f;
                    const int r = nax == 1 ? i : (int)__umulhi((uint32_t)i, ix), z = nax == 1 ? r : (int)__umulhi((uint32_t)r, ix);
                    const int x = wrapc((side ? cx : bx) + i - r * nax, a.M), y = wrapc((side ? cy : by) + r - z * nax, a.M),
                              w = wrapc((side ? cz : bz) + z, a.M);
                    cn[j] = (uint32_t)((w * a.M + y) * a.M + x);
                    kn[j] = gload(a.mc_count + cn[j]);
                }
            }
        };
        counts(lane);
#pragma unroll 1
        for (int g = 0; g < kGroups; ++g) {
            float e = 0.f, u = 0.f;
#pragma unroll 1
            for (int b0 = 0; b0 < total; b0 += kB * kStride) {
                const int f0 = b0 + 32 * g + lane;
                int kmax = 0;
#pragma unroll
                for (int j = 0; j < kB; ++j) {
                    c[j] = cn[j];
                    k[j] = kn[j];
                    kmax = max(kmax, k[j]);
                }
                fence_cta();  // the counts are read before the records they cover
                const bool more = b0 + kB * kStride < total;
                if (more || g + 1 < kGroups) counts(more ? f0 + kB * kStride : 32 * (g + 1) + lane);
#pragma unroll 1
                for (int q2 = 0; q2 < kmax; ++q2) {
                    uint4 r[kB];
#pragma unroll
                    for (int j = 0; j < kB; ++j)
                        if (q2 < k[j]) r[j] = a.mc_pos[(long long)q2 * a.ncm + c[j]];
#pragma unroll
                    for (int j = 0; j < kB; ++j) {
                        if (q2 >= k[j]) continue;
                        if (t.type != 1 && r[j].w == t.Po.w) continue;
                        const bool old_side = t.type == 2 || (t.type == 0 && f0 + j * kStride < n3);
                        const GridSep sep = grid_sep(old_side ? t.Po : t.Pn, r[j]);
                        if (sep.g >= R2) continue;
                        const int kk = t.s * kMaxSpecies + (int)tag_species(r[j].w);
                        float x, m;
                        lj_f32(sep, a.ff.c4e[kk], a.ff.sig2[kk], x, m);
                        e += old_side ? -x : x;
                        u += m;
                    }
                }
            }
            o.e += warp_sum(e);
            o.ua += warp_sum(u);
        }
    }

    template <bool P32, bool VIR>
    __device__ __forceinline__ void evaluate_cells(const Trial &t, Sums &o) const
    {
        const unsigned lt = (1u << lane) - 1u;
        // lane l owns work cells l and l + 32.  The counts are read before the
        // records: a count covers records that are already in place.
        int c0 = 0, c1 = 0, n0 = 0, n1 = 0, nw = 27;
        uint32_t f0 = t.type == 0 ? (kOld | kNew) : (t.type == 1 ? kNew : kOld), f1 = 0;
        if (!t.cross) {
            c0 = cell_at(t.px + (k27 & 0xFF) - 1, t.py + ((k27 >> 8) & 0xFF) - 1, t.pz + (k27 >> 16) - 1);
            if (lane >= 27) f0 = 0;
        } else {
            nw = t.far ? 54
                       : (3 + (union_axis(t.px, t.qx) != 0)) * (3 + (union_axis(t.py, t.qy) != 0)) *
                             (3 + (union_axis(t.pz, t.qz) != 0));
            cross_cell(t, lane, c0, f0);
            if (lane >= nw) f0 = 0;
            if (nw > 32) {
                cross_cell(t, lane + 32, c1, f1);
                if (lane + 32 >= nw) f1 = 0;
                if (f1) n1 = cload(cnt[c1]);
            }
        }
        if (f0) n0 = cload(cnt[c0]);
        fence_cta();
        const int i0 = warp_inclusive_scan(n0);
        int P = __shfl_sync(0xffffffffu, i0, 31);
        const unsigned e0 = __ballot_sync(0xffffffffu, n0 > 0);
        // where each cell's records begin (out of reach for an empty cell),
        // and the table of the cells that have some
        const int s0 = n0 ? i0 - n0 : INT_MAX;
        int s1 = INT_MAX;
        __syncwarp();
        if (n0) {
            const long long off = (long long)c0 * cap - s0;
            tab[__popc(e0 & lt)] = make_int4((int)off, (int)(off >> 32), (int)f0, 0);
        }
        if (nw > 32) {
            const int i1 = warp_inclusive_scan(n1) + P;
            P = __shfl_sync(0xffffffffu, i1, 31);
            const unsigned e1 = __ballot_sync(0xffffffffu, n1 > 0);
            if (n1) {
                s1 = i1 - n1;
                const long long off = (long long)c1 * cap - s1;
                tab[__popc(e0) + __popc(e1 & lt)] = make_int4((int)off, (int)(off >> 32), (int)f1, 0);
            }
        }
        __syncwarp();
        const uint32_t self = t.Po.w;
        const uint4 PA = t.type == 1 ? t.Pn : t.Po;
        const int wA = t.s * kMaxSpecies + (t.type == 1 ? 0 : 0x100), wB = t.s * kMaxSpecies;
        const uint32_t fA = t.type == 1 ? kNew : kOld;
        int head = 0, nq = 0, ord = -1;
        uint4 r = make_uint4(0, 0, 0, 0);
        uint32_t f = 0;  // flags of r (0: no record)
        // base: first of the records being screened; those after them load
#pragma unroll 1
        for (int base = -32;; base += 32) {
            // (opaque to the compiler, which would make a copy of the loop for
            // every combination of the two)
            int two = t.type == 0, wide = nw > 32;
            asm volatile("" : "+r"(two), "+r"(wide));
            uint4 rn = r;
            uint32_t fn = 0;
            const int nb = base + 32;
            if (nb < P) {
                // the cells whose records begin among these 32
                uint32_t x = bit_at(s0 - nb);
                if (wide) x |= bit_at(s1 - nb);
                x = __reduce_or_sync(0xffffffffu, x);
                const int k = ord + __popc(x & (lt * 2u + 1u));
                ord += __popc(x);
                if (nb + lane < P) {
                    const int4 e = tab[k];
                    const long long off = ((long long)e.y << 32) | (uint32_t)e.x;
                    rn = cell_pos[off + (nb + lane)];
                    fn = (uint32_t)e.z;
                }
            }
            if (f && r.w == self) f = 0;  // the particle itself
            {
                const int ex = (int)(PA.x - r.x), ey = (int)(PA.y - r.y), ez = (int)(PA.z - r.z);
                const float gx = (float)ex, gy = (float)ey, gz = (float)ez;
                const bool in = (f & fA) && fmaf(gx, gx, fmaf(gy, gy, gz * gz)) < r2hi;
                const unsigned b = __ballot_sync(0xffffffffu, in);
                if (in) q[(head + nq + __popc(b & lt)) & (kQ - 1)] = make_int4(ex, ey, ez, wA + (int)tag_species(r.w));
                nq += __popc(b);
            }
            if (two) {
                const int ex = (int)(t.Pn.x - r.x), ey = (int)(t.Pn.y - r.y), ez = (int)(t.Pn.z - r.z);
                const float gx = (float)ex, gy = (float)ey, gz = (float)ez;
                const bool in = (f & kNew) && fmaf(gx, gx, fmaf(gy, gy, gz * gz)) < r2hi;
                const unsigned b = __ballot_sync(0xffffffffu, in);
                if (in) q[(head + nq + __popc(b & lt)) & (kQ - 1)] = make_int4(ex, ey, ez, wB + (int)tag_species(r.w));
                nq += __popc(b);
            }
            const bool last = nb >= P;
#pragma unroll 1
            while (nq >= 32 || (last && nq > 0)) {
                const int c = min(nq, 32);
                __syncwarp();
                if (lane < c) pair_term<P32, VIR>(q[(head + lane) & (kQ - 1)], o);
                head += c;
                nq -= c;
                __syncwarp();
            }
            if (last) break;
            r = rn;
            f = fn;
        }
    }

    // Adds one queued pair, if it is inside the cutoff.
    template <bool P32, bool VIR>
    __device__ __forceinline__ void pair_term(const int4 &p, Sums &o) const
    {
        const unsigned long long g2 = (unsigned long long)((long long)p.x * p.x) +
                                      (unsigned long long)((long long)p.y * p.y) +
                                      (unsigned long long)((long long)p.z * p.z);
        if (g2 >= R2) return;
        const int k = p.w & 0xFF;
        const bool neg = (p.w & 0x100) != 0;
        if constexpr (P32) {
            const float4 c = sh.field[k];
            float uh, ul, m;
            lj_ff(p.x, p.y, p.z, c.x, c.z, c.y, c.w, uh, ul, m);
            ff_acc(o.e, o.el, neg ? -uh : uh, neg ? -ul : ul);
            o.ua += m;
            if (VIR) {
                const float w = -fmaf(3.f, m, 9.f * uh);  // r U'(r) = -12 rep + 6 att
                o.w += neg ? -w : w;
            }
        } else {
            GridSep s;
            s.dx = p.x;
            s.dy = p.y;
            s.dz = p.z;
            s.g = g2;
            double u, m;
            lj_f64(s, a.fd.rep[k], a.fd.att[k], u, m);
            o.de += neg ? -u : u;
            o.da += m;
            if (VIR) {
                const double w = 3.0 * m + 9.0 * u;
                o.dw -= neg ? -w : w;
            }
        }
    }

    // The Metropolis test of Eqs. 3-5 (textbook sign of mu) in FP32 with an
    // explicit error band, for N_s = ns: 1 accept, 0 reject, -1 inside the
    // band or not finite (decided in FP64).  The band holds the rounding of
    // every term at its own size: ln K is the difference of z = ln z + ln V
    // (rounded, 6e-8 |z|, and |z| <= |ln K| + l) and l = ln N (logf, 1.2e-7 l),
    // which cancel.
    __device__ __forceinline__ int decide_f32(int type, int sp, int ns, float lnu, float dUf, float uab) const
    {
        float lnK = 0.f, l = 0.f;
        if (type != 0) {
            const float z = a.lnzv_f[sp];
            l = logf((float)(type == 1 ? ns + 1 : ns));
            lnK = type == 1 ? z - l : l - z;
        }
        const float bd = a.beta_f * dUf;
        const float band =
            a.beta_f * a.tol_f * uab + 1e-6f * (1.f + fabsf(lnK) + 2.f * l + fabsf(bd) + fabsf(lnu));
        const float diff = lnu - (lnK - bd);
        if (fabsf(diff) > band) return (diff < 0.f) ? 1 : 0;
        return -1;
    }

    // Tests the trial of move m, evaluated after c0 committed moves, against
    // the logged moves c0 .. m - 1, evaluated or committed.  Bit i of conf:
    // move m - 1 - i, if accepted, voids the evaluation: it touches the old
    // cell or the particle's record, or puts, removes or moves a particle
    // within rc of the trial's old or new position (a coordinate of a record
    // overwritten in place may be read from either value, so a move's old and
    // new positions are tested per axis by the nearer one; an entry that a
    // removal moved into the freed slot may be met twice by an evaluation
    // that read the older count).  Changes farther away add nothing: their
    // pair terms are exactly zero.  Bit i of stale: it changes what is known
    // of the species' last particle.  ver: lane i's version of the entry of
    // move m - 1 - i (0: not there yet).  Eight moves a pass; lane 8 k + i tests
    // positions (k = 0, 1) or the moved entry (k = 2, 3) of the i-th against
    // the trial's old (k even) or new (k odd) position.
    __device__ __forceinline__ void check_logs(const Trial &t, int last_id, int last_cell, bool unborn, int c0, int m,
                                               uint32_t &conf, uint32_t &stale, int &ver) const
    {
        conf = stale = 0;
        const int k = lane >> 3;
        const bool side = (k & 1) ? t.type != 2 : t.type != 1;
        const uint4 P = (k & 1) ? t.Pn : t.Po;
        const int myid = (t.s << 24) | t.idx;
#pragma unroll 1
        for (int b = 0; b < m - c0; b += 8) {
            const int i = b + (lane & 7), j = m - 1 - i;
            bool bad = false, old = false;
            int v = 0;
            if (j >= c0) v = vload(sh.ver[j & (kRS - 1)]);
            fence_cta();
            if ((v >> 8) == (j & 0x7FFFFF) && v != 0 && j >= c0) {
                const LogRec &L = sh.logs[j & (kRS - 1)];
                const uint4 p0 = L.pos0;
                const uint4 X0 = k < 2 ? p0 : L.moved, X1 = k < 2 && (p0.w & 1u) ? L.pos1 : X0;
                if (k == 0) {
                    const int4 id = L.ids;
                    bad = t.type != 1 && (id.x == t.co || id.y == t.co || id.z == myid || id.w == myid ||
                                          (unborn && (p0.w & 4u) && (int)(p0.w >> 8) == t.s));
                    old = id.x == last_cell || id.y == last_cell || id.z == last_id || id.w == last_id;
                }
                const float dx = (float)min(axis_dist(X0.x, P.x), axis_dist(X1.x, P.x)),
                            dy = (float)min(axis_dist(X0.y, P.y), axis_dist(X1.y, P.y)),
                            dz = (float)min(axis_dist(X0.z, P.z), axis_dist(X1.z, P.z));
                if (side && (k < 2 || (p0.w & 2u)) && fmaf(dx, dx, fmaf(dy, dy, dz * dz)) < r2hi) bad = true;
            } else {
                v = 0;
            }
            unsigned x = __ballot_sync(0xffffffffu, bad);
            x |= x >> 16;
            conf |= ((x | (x >> 8)) & 0xFFu) << b;
            stale |= (__ballot_sync(0xffffffffu, old) & 0xFFu) << b;
            if ((lane & ~7) == b) ver = v;
        }
    }

    // The particle counts at the turn of move m, predicted after c committed
    // moves: an insertion or deletion evaluated and likely accepted, or not
    // yet evaluated and of a kind this chain mostly accepts, counts +1 or -1
    // for its species (the movers post this outlook).  Lane q < S gets
    // species q's count.
    __device__ __forceinline__ int predict_counts(int c, int m, int &now) const
    {
        int code = 0;
        const int k = c + lane;
        if (k < m) {
            const int o = vload(sh.outlook[k & (kRS - 1)]);
            if ((o >> 8) == (k & 0x7FFFFF)) code = o & 0xFF;
        }
        now = lane < S ? vload(sh.n[lane]) : 0;
        int n = now;
#pragma unroll 1
        for (int s = 0; s < S; ++s) {
            const int d = __popc(__ballot_sync(0xffffffffu, code == ((s << 2) | 1))) -
                          __popc(__ballot_sync(0xffffffffu, code == ((s << 2) | 2)));
            if (lane == s) n += d;
        }
        return (int)min((long long)max(n, 0), a.maxN);
    }

};

// FP64 evaluation of a trial inside the FP32 error band.
template <bool VIR, bool MICRO>
__device__ __noinline__ Sums evaluate64(Mover<MICRO> M, Trial t)
{
    Sums d;
    M.template evaluate<false, VIR>(t, d);
    return d;
}

template <bool F32, bool VIR, bool PROF, bool MICRO>
__device__ __forceinline__ void mover_loop(const ChainArgs &a, Shared &sh, uint16_t *cnt, unsigned char *mine, int warp)
{
    const int lane = threadIdx.x & 31, n = a.n_moves, W = a.movers;
    Mover<MICRO> M{a, sh, cnt, (int4 *)mine, (WordRec *)(mine + kQ * 16), (int4 *)(mine + kQ * 16 + kWords * 48),
                   a.cell_pos, a.R2, a.r2hi, lane, a.T, a.S, a.cap, lane % 3 | (lane / 3 % 3) << 8 | (lane / 9) << 16};
    const int S = M.S;
    unsigned long long c_eval = 0, c_room = 0, c_wait = 0, c_logs = 0, c_pick = 0, c_dec = 0, c_app = 0, c_book = 0,
                       c_all = 0;
    long long n_eval = 0;
    int it = 0;
#pragma unroll 1
    for (int m = warp; m < n; m += W, ++it) {
        if ((it & (kWords - 1)) == 0) fill_words(a, M.words, m, lane);
        const WordRec &WR = M.words[it & (kWords - 1)];
        uint32_t w[8];
        {
            const uint4 x = ((const uint4 *)WR.w)[0], y = ((const uint4 *)WR.w)[1];
            w[0] = x.x; w[1] = x.y; w[2] = x.z; w[3] = x.w;
            w[4] = y.x; w[5] = y.y; w[6] = y.z; w[7] = y.w;
        }
        const int type = w[0] < a.thr_disp ? 0 : (w[0] < a.thr_ins ? 1 : 2);
        const int slot = m & (kRS - 1), mtag = (m & 0x7FFFFF) << 8;
        if (type && lane == 0) {
            // a bet for the predictions of later moves, until the evaluation is in
            const int code = vload(sh.likely[type - 1]) ? ((int)__umulhi(w[5], (uint32_t)S) << 2) | type : 0;
            vstore(sh.outlook[slot], mtag | code);
        }
        bool need64 = false;
#pragma unroll 1
        for (int attempt = 1;; ++attempt) {
            // ------------------------------------------------ evaluate
            const unsigned long long t0 = prof_clock<PROF>();
            const int4 v0 = turn_load(sh);
            const int c0 = __shfl_sync(0xffffffffu, v0.x, 0);
            if (__shfl_sync(0xffffffffu, v0.z, 0)) goto done;
            fence_cta();
            // lane q < S: the count of species q now, and the one the evaluation assumes
            int now;
            const int nq = M.predict_counts(c0, m, now);
            Trial t;
            M.pick(w, type, nq, t.s, t.idx);
            const int s = t.s, idx = t.idx;
            const int nref = __shfl_sync(0xffffffffu, nq, s);  // N_s assumed
            const int nnow = __shfl_sync(0xffffffffu, now, s);
            const bool unborn = idx >= nnow;  // a pending insertion's particle
            t.type = type;
            t.possible = type == 1 || idx >= 0;
            t.cross = t.far = false;
            t.co = t.cn = -1;
            t.Po = make_uint4(0, 0, 0, 0xFFFFFFFFu);
            t.Pn = make_uint4(0, 0, 0, 0);
            // the old cell's count, and its entry `lane`; for a deletion the
            // species' last particle, which will take the freed index
            int nco = 0, qcell = -1, last_id = -1, qn = 0;
            uint4 lastv = make_uint4(0, 0, 0, 0), Q = lastv;
            uint32_t qtag = 0;
            if (t.possible) {
                if (type != 1) {
                    // the records in lanes 0 (the particle) and 1 (the last one)
                    uint4 r = make_uint4(0, 0, 0, 0);
                    if (lane < (type == 2 ? 2 : 1)) r = a.pos_by_id[(long long)s * a.maxN + (lane ? nref - 1 : idx)];
                    t.Po.x = __shfl_sync(0xffffffffu, r.x, 0);
                    t.Po.y = __shfl_sync(0xffffffffu, r.y, 0);
                    t.Po.z = __shfl_sync(0xffffffffu, r.z, 0);
                    t.Po.w = __shfl_sync(0xffffffffu, r.w, 0);
                    if (type == 2 && idx != nref - 1 && nref <= nnow) {  // (a particle that is there)
                        last_id = (s << 24) | (nref - 1);
                        Q.x = __shfl_sync(0xffffffffu, r.x, 1);
                        Q.y = __shfl_sync(0xffffffffu, r.y, 1);
                        Q.z = __shfl_sync(0xffffffffu, r.z, 1);
                        Q.w = __shfl_sync(0xffffffffu, r.w, 1);
                        qcell = cell_of(Q.x, Q.y, Q.z, M.T);
                    }
                    t.px = cell_coord(t.Po.x, (uint32_t)M.T);
                    t.py = cell_coord(t.Po.y, (uint32_t)M.T);
                    t.pz = cell_coord(t.Po.z, (uint32_t)M.T);
                    t.co = (t.pz * M.T + t.py) * M.T + t.px;
                    nco = __shfl_sync(0xffffffffu, M.count(t.co), 0);
                    if (qcell >= 0) qn = __shfl_sync(0xffffffffu, M.count(qcell), 0);
                    fence_cta();
                    if (lane < nco) lastv = M.cell_pos[(long long)t.co * M.cap + lane];
                    if (lane < qn) qtag = M.cell_pos[(long long)qcell * M.cap + lane].w;
                }
                if (type == 0) {
                    t.Pn.x = t.Po.x + (uint32_t)((int)__umulhi(w[2], a.span) - a.D);
                    t.Pn.y = t.Po.y + (uint32_t)((int)__umulhi(w[3], a.span) - a.D);
                    t.Pn.z = t.Po.z + (uint32_t)((int)__umulhi(w[4], a.span) - a.D);
                } else if (type == 1) {
                    t.Pn = make_uint4(w[2], w[3], w[4], 0u);
                }
                if (type != 2) {
                    t.qx = cell_coord(t.Pn.x, (uint32_t)M.T);
                    t.qy = cell_coord(t.Pn.y, (uint32_t)M.T);
                    t.qz = cell_coord(t.Pn.z, (uint32_t)M.T);
                    t.cn = (t.qz * M.T + t.qy) * M.T + t.qx;
                    if (type == 1) {
                        t.px = t.qx;
                        t.py = t.qy;
                        t.pz = t.qz;
                    } else {
                        t.cross = t.co != t.cn;
                        t.far = t.cross && !(near1(t.px - t.qx, M.T) && near1(t.py - t.qy, M.T) && near1(t.pz - t.qz, M.T));
                    }
                }
            }
            // the microcells, and the entry that a removal moves (for the log)
            uint32_t mo = 0, mn = 0;
            uint4 mlast = make_uint4(0, 0, 0, 0);
            int m_last = -1;  // its slot (-1: none)
            if constexpr (MICRO) {
                mn = micro_of(t.Pn, a.M);
                mo = type == 1 ? mn : micro_of(t.Po, a.M);
                if (t.possible && type != 1 && (type == 2 || mo != mn)) {
                    const MicroEntry x = micro_find(a, mo, t.Po.w, lane);
                    if (x.slot != x.n - 1) m_last = x.n - 1;
                    mlast = x.v;
                }
            }
            Sums E;
            M.template evaluate<F32, VIR>(t, E);
            ++n_eval;
            // the slots of the particle and of the species' last one
            int self_slot = -1, qslot = -1;
            if (type != 1) {
                const unsigned hit = __ballot_sync(0xffffffffu, lane < nco && lastv.w == t.Po.w);
                if (nco <= 32) {
                    self_slot = __ffs(hit) - 1;
                } else {
                    const Found x = find_far(M.cell_pos + (long long)t.co * M.cap, t.Po.w, nco, lastv, lane);
                    self_slot = x.at;
                    lastv = x.last;
                }
                if (qn > 0) {
                    const unsigned hq = __ballot_sync(0xffffffffu, lane < qn && qtag == Q.w);
                    qslot = __ffs(hq) - 1;  // -1: looked up at the turn
                }
            }
            const bool has_last = (type == 2 || t.cross) && self_slot != nco - 1;
            const bool last_mine = has_last && lane == ((nco - 1) & 31);
            // the decision and the pick for each count N_s = nref - 16 + lane
            // its turn can meet (at most kMaxMovers - 1 moves are pending)
            uint32_t acc_mask, band_mask, same_mask;
            {
                const int nl = nref - 16 + lane;
                const float dUf = F32 ? E.e + E.el : __double2float_rn(E.de), uab = F32 ? E.ua : __double2float_rn(E.da);
                const int dec = t.possible && nl >= 0 ? M.decide_f32(type, s, nl, WR.lnu, dUf, uab) : 0;
                bool same = true;
                if (type == 2 || (type == 0 && S == 1))
                    same = nl > 0 ? (idx >= 0 && pick_index((uint32_t)nl, w, type) == idx) : idx < 0;
                acc_mask = __ballot_sync(0xffffffffu, dec > 0);
                band_mask = __ballot_sync(0xffffffffu, dec < 0);
                same_mask = __ballot_sync(0xffffffffu, same);
            }
            // FP32 mode: a trial inside the band is evaluated in FP64 too
            bool have64 = !F32;
            if constexpr (F32) {
                if (need64 || ((band_mask >> 16) & 1u)) {
                    const Sums d = evaluate64<VIR, MICRO>(M, t);
                    E.de = d.de;
                    E.da = d.da;
                    E.dw = d.dw;
                    have64 = true;
                }
            }
            // what later moves need to know
            {
                LogRec &L = sh.logs[slot];
                if (attempt > 1) {
                    if (lane == 0) vstore(sh.ver[slot], 0);
                    fence_cta();
                    __syncwarp();
                }
                if (MICRO ? lane == m_last : last_mine) L.moved = MICRO ? mlast : lastv;
                if (lane == 0) {
                    L.ids = make_int4(type == 1 ? t.cn : t.co, t.cross ? t.cn : qcell, type == 1 ? -1 : (s << 24) | idx,
                                      last_id);
                    const uint4 p = type == 1 ? t.Pn : t.Po;
                    L.pos0 = make_uint4(p.x, p.y, p.z,
                                        (type == 0 ? 1u : 0u) | ((MICRO ? m_last >= 0 : has_last) ? 2u : 0u) | (type == 1 ? 4u : 0u) | ((uint32_t)s << 8));
                    L.pos1 = t.Pn;
                    if (type) vstore(sh.outlook[slot], mtag | (((acc_mask >> 16) & 1u) ? (s << 2) | type : 0));
                }
                __syncwarp();
                if (lane == 0) {
                    fence_cta();
                    vstore(sh.ver[slot], mtag | (attempt & 0x7F) | 0x80);
                }
            }
            const unsigned long long t1 = prof_clock<PROF>();
            c_eval += t1 - t0;
            // ------------------------------------------------ wait for the turn
            if (m >= __shfl_sync(0xffffffffu, vload(sh.booked), 0) + kRS && !wait_room(a, sh, m)) goto done;
            const unsigned long long t2 = prof_clock<PROF>();
            c_room += t2 - t1;
            // tested against the moves before it while it waits
            uint32_t conf = 0, stale = 0;
            int ver = 0, seen = c0;
            int4 v;
            bool again = false;
            {
                Wait wt;
                const bool mine_i = lane < m - c0;
                const int vi = (m - 1 - lane) & (kRS - 1);
#pragma unroll 1
                for (;;) {
                    v = turn_load(sh);
                    if (__all_sync(0xffffffffu, v.x == m && v.z == 0)) break;
                    const int c = __shfl_sync(0xffffffffu, v.x, 0);
                    if (__shfl_sync(0xffffffffu, v.z, 0)) goto done;
                    if (c < m && t.possible) {
                        const uint32_t hist = (uint32_t)__shfl_sync(0xffffffffu, v.y, 0) << (m - c);
                        fence_cta();
                        // entries that are new since they were tested: tested
                        // once their move is committed and accepted, or near the turn
                        const uint32_t fresh = __ballot_sync(0xffffffffu, mine_i && vload(sh.ver[vi]) != ver);
                        if ((fresh & hist) || (fresh && m - c <= 2))
                            M.check_logs(t, last_id, qcell, unborn, c0, m, conf, stale, ver);
                        if (c != seen) {
                            seen = c;
                            wt = Wait();
                            if (conf & hist) again = true;
                            // the pick for the counts as now predicted
                            if (same_mask != 0xffffffffu) {
                                int x;
                                const int i = __shfl_sync(0xffffffffu, M.predict_counts(c, m, x), s) - nref + 16;
                                if (i < 0 || i > 31 || !((same_mask >> i) & 1u)) again = true;
                            }
                            if (again) break;
                            continue;
                        }
                    }
                    if (gave_up(a, sh, wt, 2)) goto done;
                    if (m - c > 2) __nanosleep(20 * (m - c - 1));
                }
            }
            if (again) {
                c_wait += prof_clock<PROF>() - t2;
                continue;  // evaluate again, before the turn
            }
            // ------------------------------------------------ the turn
            if (m == a.stall_at && !wait_never(a, sh)) goto done;
            fence_cta();
            const unsigned long long t3 = prof_clock<PROF>();
            c_wait += t3 - t2;
            const int ns = vload(sh.n[s]);
            const int c_n = t.cn >= 0 ? M.count(t.cn) : 0;
            const uint32_t hist = (uint32_t)v.y & ((1u << (m - c0)) - 1u);  // m - c0 < kRS
            if (t.possible) {
                const uint32_t fresh = __ballot_sync(0xffffffffu, lane < m - c0 && vload(sh.ver[(m - 1 - lane) & (kRS - 1)]) != ver);
                if (fresh & hist) M.check_logs(t, last_id, qcell, unborn, c0, m, conf, stale, ver);
            }
            const unsigned long long t4 = prof_clock<PROF>();
            c_logs += t4 - t3;
            const int i = ns - nref + 16;
            bool valid = !(conf & hist) && i >= 0 && i <= 31 && ((same_mask >> (i & 31)) & 1u);
            if (type == 0 && S > 1) {
                // several counts decide the pick: the same counts, or the same pick
                const int cur = lane < S ? vload(sh.n[lane]) : 0;
                if (!__all_sync(0xffffffffu, lane >= S || cur == nq)) {
                    int s2, i2;
                    M.pick(w, 0, cur, s2, i2);
                    valid = !(conf & hist) && i2 == idx && (idx < 0 || s2 == s);
                }
            }
            const int ii = type == 0 ? 16 : (i & 31);  // a displacement's decision does not depend on the counts
            const bool in_band = (band_mask >> ii) & 1u;
            const unsigned long long t5 = prof_clock<PROF>();
            c_pick += t5 - t4;
            if (!valid || (in_band && !have64)) {
                // an evaluation that began at the turn stands, unless FP64 is wanted
                if (c0 == m && !valid) {
                    if (lane == 0) chain_stop(sh, kStatusBadInput, 8);
                    goto done;
                }
                need64 = need64 || in_band;
                continue;
            }
            // the Metropolis test in FP32 with an error band, inside it in FP64
            int bits = (((acc_mask >> ii) & 1u) ? kBkAcc : 0) | (attempt > 1 ? kBkAgain : 0) | (F32 ? 0 : kBkUse64);
            double lnA = 0.0;
            if (in_band) {
                const Decision d = decide_f64(a, w[6], w[7], type, s, ns, E.de, E.da);
                lnA = d.lnA;
                bits = (bits & ~kBkAcc) | kBkUse64 | (MICRO && !F32 ? 0 : kBkRefined) | d.bits;
            }
            const bool fin = bits & kBkAcc;
            MicroEntry mx = {0, -1, make_uint4(0, 0, 0, 0)};
            int n_mn = 0;
            if (fin) {
                int stop_bits = 0;
                if (type != 2 && (type == 1 || t.cross) && c_n >= M.cap) stop_bits = kStatusCellOverflow;
                if (type == 1 && ns >= a.maxN) stop_bits = kStatusCapacity;
                if (type != 1 && self_slot < 0) stop_bits = kStatusBadInput;  // a record missing from its cell
                if constexpr (MICRO) {
                    // the microcells as they are now
                    if (type == 1 || (type == 0 && mn != mo)) {
                        n_mn = __shfl_sync(0xffffffffu, gload(a.mc_count + mn), 0);
                        if (!stop_bits && n_mn >= a.mcap) stop_bits = kStatusMicroOverflow;
                    }
                    if (type != 1) {
                        mx = micro_find(a, mo, t.Po.w, lane);
                        if (mx.slot < 0) stop_bits = kStatusBadInput;
                        // a removal moves another entry than the log says: later moves test it again
                        const int moves = (type == 2 || mn != mo) && mx.slot != mx.n - 1 ? mx.n - 1 : -1;
                        const bool same = moves == m_last &&
                                          (lane != moves || (mx.v.x == mlast.x && mx.v.y == mlast.y && mx.v.z == mlast.z));
                        if (!stop_bits && !__all_sync(0xffffffffu, same)) {
                            LogRec &L = sh.logs[slot];
                            if (lane == 0) {
                                vstore(sh.ver[slot], 0);
                                fence_cta();
                                L.pos0.w = (L.pos0.w & ~2u) | (moves >= 0 ? 2u : 0u);
                            }
                            __syncwarp();
                            if (lane == moves) L.moved = mx.v;
                            __syncwarp();
                            if (lane == 0) {
                                fence_cta();
                                vstore(sh.ver[slot], mtag | 0x7E);
                            }
                            __syncwarp();
                        }
                    }
                }
                if (stop_bits) {
                    if (lane == 0) chain_stop(sh, stop_bits, 16);
                    goto done;
                }
            }
            const unsigned long long t6 = prof_clock<PROF>();
            c_dec += t6 - t5;
            // ------------------------------------------------ apply (Sec. 3.2.5)
            if (fin) {
                uint4 *by_id = a.pos_by_id + (long long)s * a.maxN;
                uint4 *old_cell = M.cell_pos + (long long)t.co * M.cap;
                bool both = false;
                uint32_t ntag = t.Po.w;
                if (type == 2) {
                    // swap-with-last inside the cell, then the species' last
                    // index takes the freed index (its record and its cell entry)
                    const int last = ns - 1;
                    ntag = make_tag((uint32_t)idx, (uint32_t)s);
                    if (idx != last) {
                        // known from the evaluation unless a later move touched it
                        if (last_id != ((s << 24) | last) || (stale & hist) || qslot < 0) {
                            const Entry x = find_now<MICRO>(a, cnt, s, last, lane);
                            Q = x.Q;
                            qcell = x.cell;
                            qslot = x.slot;
                            if (lane == 0) {
                                sh.logs[slot].ids.y = qcell;
                                sh.logs[slot].ids.w = (s << 24) | last;
                                fence_cta();
                                vstore(sh.ver[slot], mtag | 0x7F);  // later moves test it again
                            }
                            if (qslot < 0) {
                                if (lane == 0) chain_stop(sh, kStatusBadInput, 32);
                                goto done;
                            }
                        }
                        // the last particle may be the entry that moves into the freed slot
                        both = qcell == t.co && qslot == nco - 1;
                        if constexpr (MICRO) {
                            // the same in the microcells
                            const uint32_t mq = micro_of(Q, a.M);
                            const MicroEntry x = micro_find(a, mq, Q.w, lane);
                            if (x.slot < 0) {
                                if (lane == 0) chain_stop(sh, kStatusBadInput, 32);
                                goto done;
                            }
                            if (mq == mo && x.slot == mx.n - 1) {
                                if (lane == mx.n - 1) mx.v.w = ntag;
                            } else if (lane == 0) {
                                a.mc_pos[(long long)x.slot * a.ncm + mq].w = ntag;
                            }
                        }
                        if (lane == 0) {
                            if (!both) M.cell_pos[(long long)qcell * M.cap + qslot].w = ntag;
                            by_id[idx] = make_uint4(Q.x, Q.y, Q.z, ntag);
                        }
                    }
                } else if (lane == 0) {
                    const bool move_in = type == 1 || t.cross;
                    if (type == 1) ntag = make_tag((uint32_t)ns, (uint32_t)s);
                    const uint4 r = make_uint4(t.Pn.x, t.Pn.y, t.Pn.z, ntag);
                    M.cell_pos[(long long)t.cn * M.cap + (move_in ? c_n : self_slot)] = r;
                    by_id[type == 1 ? ns : idx] = r;
                }
                if (last_mine) {
                    if (both) lastv.w = ntag;
                    old_cell[self_slot] = lastv;
                }
                if constexpr (MICRO) {
                    const bool leaves = type == 2 || (type == 0 && mn != mo);
                    if (leaves && lane == mx.n - 1 && mx.slot != mx.n - 1) a.mc_pos[(long long)mx.slot * a.ncm + mo] = mx.v;
                    if (type != 2 && lane == 0)
                        a.mc_pos[(long long)(type == 0 && !leaves ? mx.slot : n_mn) * a.ncm + mn] =
                            make_uint4(t.Pn.x, t.Pn.y, t.Pn.z, ntag);
                    __syncwarp();
                    if (lane == 0 && (leaves || type == 1)) {
                        fence_cta();
                        if (leaves) gstore(a.mc_count + mo, mx.n - 1);
                        if (type != 2) gstore(a.mc_count + mn, n_mn + 1);
                    }
                }
                __syncwarp();
                if (lane == 0 && (type != 0 || t.cross)) {
                    fence_cta();  // the records before the counts that cover them
                    if (type != 1) M.set_count(t.co, nco - 1);
                    if (type != 2) M.set_count(t.cn, c_n + 1);
                    if (type != 0) vstore(sh.n[s], type == 1 ? ns + 1 : ns - 1);
                }
            }
            const unsigned long long t7 = prof_clock<PROF>();
            c_app += t7 - t6;
            // ------------------------------------------------ pass the turn on
            if (lane == 0) {
                fence_cta();  // the move's writes before the turn that says they are there
                turn_store(sh, m + 1, ((uint32_t)v.y << 1) | (fin ? 1u : 0u));
                BookRec &B = sh.book[slot];
                B.dU64 = E.de;
                B.lnA = lnA;
                B.dW = VIR ? (F32 && !in_band ? (double)E.w : E.dw) : 0.0;
                B.hi = E.e;
                B.lo = E.el;
                B.uab = F32 && !in_band ? (double)E.ua : E.da;
                B.bits = bits | (t.possible ? kBkPossible : 0) | (type << 8) | (s << 16);
                B.index = type == 1 ? ns : idx;
                B.n = ns;
                fence_cta();
                vstore(B.ready, m + 1);
            }
            __syncwarp();
            const unsigned long long t8 = prof_clock<PROF>();
            c_book += t8 - t7;
            c_all += t8 - t1;
            break;
        }
    }
done:
    __syncwarp();
    if (lane == 0) {
        fence_cta();
        atomicAdd(&sh.gone, 1);
        atomicAdd((unsigned long long *)&sh.evaluations, (unsigned long long)n_eval);
        if constexpr (PROF) {
            atomicAdd(&sh.prof[0], c_wait);
            atomicAdd(&sh.prof[1], c_logs + c_pick);
            atomicAdd(&sh.prof[2], c_dec);
            atomicAdd(&sh.prof[3], c_app);
            atomicAdd(&sh.prof[4], c_all);
            atomicAdd(&sh.prof[5], c_room);
            atomicAdd(&sh.prof[6], c_eval);
            atomicAdd(&sh.prof[9], c_logs);
            atomicAdd(&sh.prof[10], c_pick);
            atomicAdd(&sh.prof[11], c_book);
        }
    }
}

// The keeper: books the committed moves in order.
template <bool VIR>
__device__ void keeper_loop(const ChainArgs &a, Shared &sh)
{
    const int lane = threadIdx.x & 31, n = a.n_moves;
    double E = *a.d_energy, sumE = 0.0;
    // the running virial, for the chains of the launch that keep it
    const bool vir = VIR && a.virial;
    double Wv = vir ? a.d_energy[1] : 0.0, sumW = 0.0;
    long long sumN = 0, att0 = 0, att1 = 0, att2 = 0, acc0 = 0, acc1 = 0, acc2 = 0;
    long long flagged = 0, reeval = 0, refines = 0, Ncur = 0;
    for (int k = 0; k < kMaxSpecies; ++k) Ncur += k < a.S ? a.d_n[k] : 0;
    int mb = 0;
    Wait wt;
    while (mb < n) {
        const int rdy = vload(sh.book[mb & (kRS - 1)].ready);
        if (__shfl_sync(0xffffffffu, rdy, 0) == mb + 1) {
            fence_cta();
            if (lane == 0) {
                const BookRec &B = sh.book[mb & (kRS - 1)];
                const int bits = B.bits, type = (bits >> 8) & 0xFF, sp = bits >> 16;
                const bool acc = bits & kBkAcc;
                att0 += type == 0;
                att1 += type == 1;
                att2 += type == 2;
                if (bits & kBkNear) ++flagged;
                if (bits & kBkRefined) ++refines;
                if (bits & kBkAgain) ++reeval;
                const double dU = (bits & kBkUse64) ? B.dU64 : (double)B.hi + (double)B.lo;
                if (acc) {
                    acc0 += type == 0;
                    acc1 += type == 1;
                    acc2 += type == 2;
                    E += dU;
                    Wv += B.dW;
                    Ncur += (type == 1) - (type == 2);
                }
                if (type == 1) vstore(sh.likely[0], 2 * acc1 > att1);
                else if (type == 2) vstore(sh.likely[1], 2 * acc2 > att2);
                if (a.trace) {
                    const bool possible = bits & kBkPossible;
                    gcmc_trace tr;
                    double lnA = B.lnA;
                    if (!(bits & kBkRefined)) {
                        double lnK = 0.0;
                        if (type == 1) lnK = a.logz[sp] + a.lnV - log((double)(B.n + 1));
                        else if (type == 2 && B.n > 0) lnK = log((double)B.n) - a.logz[sp] - a.lnV;
                        lnA = possible ? lnK - a.beta * dU : -INFINITY;
                    }
                    tr.dU = possible ? dU : 0.0;
                    tr.lnA = lnA;
                    tr.uabs = possible ? B.uab : 0.0;
                    tr.index = B.index;
                    tr.type = (uint8_t)type;
                    tr.species = (uint8_t)sp;
                    tr.accepted = (uint8_t)acc;
                    tr.flagged = (uint8_t)(((bits & kBkNear) ? 1 : 0) | ((bits & kBkRefined) ? 2 : 0));
                    a.trace[mb] = tr;
                }
                sumE += E;
                sumW += Wv;
                sumN += Ncur;
                fence_cta();
                vstore(sh.booked, mb + 1);
            }
            __syncwarp();
            ++mb;
            wt = Wait();
            continue;
        }
        // a stopped chain may still commit the move that held the turn: its
        // last move is known once every mover has finished
        const int gone = vload(sh.gone);
        fence_cta();
        const int4 v = turn_load(sh);
        if (__shfl_sync(0xffffffffu, v.z && gone == a.movers && mb >= v.x, 0)) break;
        if (__any_sync(0xffffffffu, wt.expired(a.wait_ns))) {
            if (lane == 0) chain_stop(sh, kStatusTimeout, 4);
            break;
        }
        __nanosleep(40);
    }
    if (lane == 0) {
        ChainOut &o = *a.out;
        o.attempted[0] = att0;
        o.attempted[1] = att1;
        o.attempted[2] = att2;
        o.accepted[0] = acc0;
        o.accepted[1] = acc1;
        o.accepted[2] = acc2;
        o.flagged = flagged;
        o.moves_done = mb;
        o.energy = E;
        o.sum_energy = sumE;
        o.sum_n = (double)sumN;
        o.reevaluated = reeval;
        o.refines = refines;
        o.virial = vir ? Wv : NAN;
        o.sum_virial = vir ? sumW : NAN;
        *a.d_energy = E;
        if (vir) a.d_energy[1] = Wv;
    }
}

template <bool F32, bool VIR, bool PROF, bool MICRO>
__global__ void __launch_bounds__(kChainWarps * 32, 1) k_chain(const ChainArgs *__restrict__ args)
{
    constexpr int NTH = kChainWarps * 32;
    // dynamic shared memory: each mover's queue and words, then the cell counters
    extern __shared__ __align__(16) unsigned char dyn[];
    unsigned long long t_start = 0;
    if (threadIdx.x == 0) asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t_start));
    __shared__ Shared sh;
    // this CTA's chain: its arguments copied to shared memory
    __shared__ __align__(16) ChainArgs a;
    const int tid = threadIdx.x, warp = tid >> 5;
    {
        const uint32_t *src = (const uint32_t *)(args + blockIdx.x);
        uint32_t *dst = (uint32_t *)&a;
        for (int k = tid; k < (int)(sizeof(ChainArgs) / 4); k += NTH) dst[k] = src[k];
        __syncthreads();
    }
    if (a.n_moves <= 0) {
        if (tid == 0) {
            ChainOut &o = *a.out;
            o.moves_done = 0;
            o.energy = *a.d_energy;
            for (int k = 0; k < kMaxSpecies; ++k) o.n[k] = k < a.S ? a.d_n[k] : 0;
            o.status = 0;
        }
        return;
    }
    constexpr int kBytes = MICRO ? kMicroMoverBytes : kMoverBytes;
    uint16_t *cnt = (uint16_t *)(dyn + (size_t)a.movers * kBytes);
    if constexpr (!MICRO)
        for (int c = tid; c < a.ncell; c += NTH) cnt[c] = (uint16_t)a.cell_count[c];
    if (tid < kMaxSpecies) sh.n[tid] = tid < a.S ? (int)a.d_n[tid] : 0;
    if (tid < kRS) {
        sh.book[tid].ready = 0;
        sh.outlook[tid] = -1;
        sh.ver[tid] = 0;
    }
    if constexpr (F32)
        for (int k = tid; k < kMaxSpecies * kMaxSpecies; k += NTH)
            sh.field[k] = make_float4(a.ff.c4e[k], a.ff.sig2[k], a.ff.c4e_lo[k], a.ff.sig2_lo[k]);
    if (tid < 12) sh.prof[tid] = 0ull;
    if (tid == 0) {
        sh.turn = make_int4(0, 0, 0, 0);
        sh.booked = sh.status = sh.where = sh.gone = sh.never = 0;
        sh.likely[0] = sh.likely[1] = 0;
        sh.evaluations = 0;
    }
    __syncthreads();
    if (warp < a.movers) mover_loop<F32, VIR, PROF, MICRO>(a, sh, cnt, dyn + (size_t)warp * kBytes, warp);
    else if (warp == kChainWarps - 1) keeper_loop<VIR>(a, sh);
    __syncthreads();
    if constexpr (!MICRO)
        for (int c = tid; c < a.ncell; c += NTH) a.cell_count[c] = cnt[c];
    if (tid < a.S) a.d_n[tid] = sh.n[tid];
    if (tid == 0) {
        ChainOut &o = *a.out;
        for (int k = 0; k < kMaxSpecies; ++k) o.n[k] = sh.n[k];
        int st = sh.status;
        if (!(o.energy - o.energy == 0.0)) st |= kStatusNonFinite;
        o.status = st;
        o.pad = sh.where;
        unsigned long long t_end;
        asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t_end));
        o.t0 = t_start;
        o.t1 = t_end;
        for (int k = 0; k < 12; ++k) o.prof[k] = sh.prof[k];
        o.prof[7] = (unsigned long long)sh.evaluations;
    }
}

// ---------------------------------------------------------------- host side
// The launcher's choices of W, the moves in flight.  More movers hide a longer
// evaluation; fewer evaluate on a newer configuration, so fewer evaluations
// are repeated where most moves are accepted or the box is small.
constexpr int kMoverChoices[kChainConfigs] = {8, 5, 11, 15};

template <bool F32, bool VIR>
static void *chain_kernel(bool prof)
{
    return prof ? (void *)k_chain<F32, VIR, true, false> : (void *)k_chain<F32, VIR, false, false>;
}
// Moves in flight of a microcell launch: all there is room for (eleven took 12 %
// longer for the 4,000 moves named at the top).
constexpr int kMicroMovers = kMaxMovers;

// One chain of a launch: its context, random stream, moves and outputs.
struct ChainJob {
    gcmc_ctx *ctx;
    uint64_t seed;
    uint32_t chain;
    uint64_t first;
    int64_t n_moves;
    gcmc_move_mix mix;
    gcmc_trace *trace;
    gcmc_move_stats agg;
    int64_t done;
    gcmc_status result;
};

static void fill_args(ChainArgs &a, const ChainJob &j, int movers, ChainOut *out)
{
    gcmc_ctx *ctx = j.ctx;
    const gcmc_move_mix *mix = &j.mix;
    memset(&a, 0, sizeof(a));
    a.seed = j.seed;
    a.first = j.first + (uint64_t)j.done;
    a.n_moves = (j.result == GCMC_OK) ? (int)std::min<int64_t>(j.n_moves - j.done, 1 << 30) : 0;
    a.chain = j.chain;
    a.movers = movers;
    a.T = ctx->T;
    a.ncell = (int)ctx->ncell;
    a.cap = ctx->cap;
    a.maxN = ctx->maxN;
    a.S = ctx->S;
    a.R2 = ctx->R2;
    // FP32 r^2 from exact integer separations carries a relative error below
    // 1e-6: every pair inside the cutoff passes the screen
    a.r2hi = (float)((double)ctx->R2 * (1.0 + 1e-5));
    a.thr_disp = (unsigned long long)(mix->p_disp * 4294967296.0);
    a.thr_ins = (unsigned long long)((mix->p_disp + mix->p_ins) * 4294967296.0);
    const int64_t D = (int64_t)(mix->max_disp * ctx->q);
    a.D = (int)D;
    a.span = (uint32_t)(2 * D + 1);
    a.beta = mix->beta;
    a.lnV = std::log(ctx->V);
    for (int s = 0; s < kMaxSpecies; ++s) a.logz[s] = s < ctx->S ? mix->log_z[s] : 0.0;
    a.tol = ctx->precision == GCMC_FP32 ? 1e-5 : 1e-12;
    a.beta_f = (float)a.beta;
    a.tol_f = (float)a.tol;
    a.virial = (mix->flags & GCMC_MIX_VIRIAL) ? 1 : 0;
    a.wait_ns = ctx->wait_ns ? ctx->wait_ns : kWaitNs;
    a.stall_at = (ctx->stall_at >= j.done && ctx->stall_at - j.done < a.n_moves) ? (int)(ctx->stall_at - j.done) : -1;
    for (int s = 0; s < kMaxSpecies; ++s) a.lnzv_f[s] = (float)(a.logz[s] + a.lnV);
    a.ff = ctx->ff;
    a.fd = ctx->fd;
    a.cell_pos = ctx->cell_pos;
    a.cell_count = ctx->cell_count;
    a.pos_by_id = ctx->pos_by_id;
    a.M = ctx->mc_M;
    a.mD = ctx->mc_D;
    a.nax = std::min(2 * ctx->mc_D + 1, ctx->mc_M);
    a.mcap = ctx->mc_cap;
    a.ncm = (uint32_t)ctx->mc_ncell;
    a.mc_count = ctx->mc_count;
    a.mc_pos = ctx->mc_pos;
    a.d_n = ctx->d_n;
    a.d_energy = ctx->d_energy;
    a.trace = j.trace ? j.trace + j.done : nullptr;
    a.out = out;
}

// Device and pinned buffers of a multi-chain launch.
struct LaunchBufs {
    ChainArgs *d_args = nullptr;
    ChainOut *d_out = nullptr;
    ChainArgs *h_args = nullptr;  // pinned
    ChainOut *h_out = nullptr;    // pinned
    int cap = 0;
    int device = -1;  // where they are: a thread may use contexts of several devices
    // a captured round (upload, kernel, download) and what it was captured for
    cudaGraphExec_t exec = nullptr;
    void *g_kern = nullptr;
    int g_K = 0;
    size_t g_smem = 0;
    cudaEvent_t ev0 = nullptr, ev1 = nullptr;  // launch timing
    void drop_graph()
    {
        if (exec) cudaGraphExecDestroy(exec);
        exec = nullptr;
        g_kern = nullptr;
        g_K = 0;
        g_smem = 0;
    }
    void free_all()
    {
        drop_graph();
        if (ev0) cudaEventDestroy(ev0);
        if (ev1) cudaEventDestroy(ev1);
        if (d_args) cudaFree(d_args);
        if (d_out) cudaFree(d_out);
        if (h_args) cudaFreeHost(h_args);
        if (h_out) cudaFreeHost(h_out);
        ev0 = ev1 = nullptr;
        d_args = h_args = nullptr;
        d_out = h_out = nullptr;
        cap = 0;
    }
    ~LaunchBufs() { free_all(); }
    cudaError_t ensure(int k)
    {
        int dev = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e != cudaSuccess) return e;
        if (k <= cap && dev == device) return cudaSuccess;
        free_all();
        device = dev;
        e = cudaMalloc(&d_args, k * sizeof(ChainArgs));
        if (e == cudaSuccess) e = cudaMalloc(&d_out, k * sizeof(ChainOut));
        if (e == cudaSuccess) e = cudaMallocHost(&h_args, k * sizeof(ChainArgs));
        if (e == cudaSuccess) e = cudaMallocHost(&h_out, k * sizeof(ChainOut));
        if (e == cudaSuccess) cap = k;
        return e;
    }
};

// Runs all jobs to completion in rounds of one launch (one CTA per chain);
// a chain that would overflow a cell or its capacity stops, is re-laid out
// and continues in the next round.  Errors are per job.
// dev_ms (may be NULL) accumulates the device time of the launches, taken
// with CUDA events on st around each launch (argument upload and result
// download of a few hundred bytes included).
static gcmc_status run_jobs(std::vector<ChainJob> &jobs, cudaStream_t st, bool f32, int config, LaunchBufs &B,
                            int64_t *launches, std::string *err, bool use_graph = false, double *dev_ms = nullptr,
                            bool micro = false)
{
    const int K = (int)jobs.size();
    if (K == 0) return GCMC_OK;
    cudaError_t e = B.ensure(K);
    if (e == cudaSuccess && dev_ms && !B.ev0) {
        e = cudaEventCreate(&B.ev0);
        if (e == cudaSuccess) e = cudaEventCreate(&B.ev1);
    }
    if (e != cudaSuccess) {
        if (err) *err = cudaGetErrorString(e);
        return GCMC_ERR_CUDA;
    }
    size_t counters = 16;
    for (auto &j : jobs) counters = std::max(counters, ((size_t)j.ctx->ncell * sizeof(uint16_t) + 15) / 16 * 16);
    // a box of very many cells leaves room for fewer movers
    const size_t state = sizeof(Shared) + sizeof(ChainArgs) + 1024;
    const size_t room = (jobs[0].ctx->smem_optin - state - counters) / kMoverBytes;
    const int movers = micro ? kMicroMovers : (int)std::min<size_t>(kMoverChoices[config], room);
    const size_t smem = micro ? (size_t)movers * kMicroMoverBytes : (size_t)movers * kMoverBytes + counters;
    // the virial sums are compiled in only when a chain of the launch keeps
    // it, the cycle counters only when a chain's context asked for them
    bool vir = false, prof = false;
    for (auto &j : jobs) {
        vir |= (j.mix.flags & GCMC_MIX_VIRIAL) != 0;
        prof |= j.ctx->chain_prof;
    }
    void *kern = f32 ? (vir ? chain_kernel<true, true>(prof) : chain_kernel<true, false>(prof))
                     : (vir ? chain_kernel<false, true>(prof) : chain_kernel<false, false>(prof));
    if (micro) kern = f32 ? (void *)k_chain<true, false, false, true> : (void *)k_chain<false, false, false, true>;
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) {
        if (err) *err = std::string("cudaFuncSetAttribute: ") + cudaGetErrorString(e);
        return GCMC_ERR_CUDA;
    }
    for (int round = 0; round < (1 << 20); ++round) {
        bool any = false;
        for (int k = 0; k < K; ++k) {
            fill_args(B.h_args[k], jobs[k], movers, B.d_out + k);
            if (micro) {  // no diagnostic stall, the default limit of the waits
                B.h_args[k].stall_at = -1;
                B.h_args[k].wait_ns = kWaitNs;
            }
            any = any || B.h_args[k].n_moves > 0;
        }
        if (!any) break;
        auto enqueue = [&]() {
            cudaError_t r = cudaMemcpyAsync(B.d_args, B.h_args, K * sizeof(ChainArgs), cudaMemcpyHostToDevice, st);
            if (r == cudaSuccess) r = cudaMemsetAsync(B.d_out, 0, K * sizeof(ChainOut), st);
            if (r == cudaSuccess) {
                void *kargs[] = {(void *)&B.d_args};
                r = cudaLaunchKernel(kern, dim3(K), dim3(kChainWarps * 32), kargs, smem, st);
            }
            if (r == cudaSuccess)
                r = cudaMemcpyAsync(B.h_out, B.d_out, K * sizeof(ChainOut), cudaMemcpyDeviceToHost, st);
            return r;
        };
        if (dev_ms) e = cudaEventRecord(B.ev0, st);
        if (e != cudaSuccess) {
            if (err) *err = std::string("cudaEventRecord: ") + cudaGetErrorString(e);
            return GCMC_ERR_CUDA;
        }
        if (use_graph) {
            if (!B.exec || B.g_kern != kern || B.g_K != K || B.g_smem != smem) {
                B.drop_graph();
                cudaGraph_t g = nullptr;
                e = cudaStreamBeginCapture(st, cudaStreamCaptureModeThreadLocal);
                if (e == cudaSuccess) {
                    cudaError_t e2 = enqueue();
                    e = cudaStreamEndCapture(st, &g);
                    if (e == cudaSuccess) e = e2;
                }
                if (e == cudaSuccess) e = cudaGraphInstantiate(&B.exec, g, 0);
                if (g) cudaGraphDestroy(g);
                if (e == cudaSuccess) {
                    B.g_kern = kern;
                    B.g_K = K;
                    B.g_smem = smem;
                }
            }
            if (e == cudaSuccess) e = cudaGraphLaunch(B.exec, st);
        } else {
            e = enqueue();
        }
        if (launches) *launches += 1;
        if (e == cudaSuccess && dev_ms) e = cudaEventRecord(B.ev1, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        if (e == cudaSuccess && dev_ms) {
            float ms = 0.f;
            e = cudaEventElapsedTime(&ms, B.ev0, B.ev1);
            *dev_ms += ms;
        }
        if (e != cudaSuccess) {
            if (err) *err = std::string("chain launch: ") + cudaGetErrorString(e);
            return GCMC_ERR_CUDA;
        }
        for (int k = 0; k < K; ++k) {
            ChainJob &j = jobs[k];
            if (B.h_args[k].n_moves <= 0) continue;
            const ChainOut &o = B.h_out[k];
            gcmc_ctx *ctx = j.ctx;
            for (int t = 0; t < 3; ++t) {
                j.agg.attempted[t] += o.attempted[t];
                j.agg.accepted[t] += o.accepted[t];
            }
            j.agg.flagged += o.flagged;
            j.agg.moves_done += o.moves_done;
            j.agg.sum_energy += o.sum_energy;
            j.agg.sum_n += o.sum_n;
            j.agg.chain_ms += (double)(o.t1 - o.t0) * 1e-6;
            j.agg.energy = o.energy;
            if (j.mix.flags & GCMC_MIX_VIRIAL) {
                j.agg.virial = o.virial;
                j.agg.sum_virial += o.sum_virial;
                ctx->virial = o.virial;
            } else {
                ctx->virial_valid = false;  // the moves did not keep it up to date
            }
            for (int q = 0; q < kMaxSpecies; ++q) {
                j.agg.n[q] = o.n[q];
                ctx->n_host[q] = o.n[q];
            }
            ctx->energy = o.energy;
            ctx->compact_valid = false;
            ctx->order_valid = false;
            ctx->last_refetch += o.reevaluated;
            ctx->last_refines += o.refines;
            for (int q = 0; q < 12; ++q) ctx->last_prof[q] += (double)o.prof[q];
            j.done += o.moves_done;
            if (o.status & kStatusNonFinite) j.result = GCMC_ERR_NONFINITE;
            if (o.status & kStatusTimeout) {
                j.result = fail(ctx, GCMC_ERR_TIMEOUT,
                                "gcmc_run_moves: a bounded wait inside the chain kernel gave up (sites " +
                                    std::to_string(o.pad) + ")");
                continue;
            }
            if (o.status & kStatusMicroOverflow) {
                if (ctx->mc_cap_req != 0 || ctx->mc_cap >= kMicroMaxCap) {
                    j.result = fail(ctx, GCMC_ERR_CELL_OVERFLOW, "gcmc_run_moves_micro: a microcell is full");
                } else {
                    const gcmc_status rs = micro_grow(ctx, std::min(kMicroMaxCap, ctx->mc_cap + 2));
                    if (rs != GCMC_OK) j.result = rs;
                }
                continue;
            }
            if (o.status & (kStatusCellOverflow | kStatusCapacity)) {
                const bool grow_cap = (o.status & kStatusCellOverflow) && ctx->cap_req == 0;
                const bool grow_n = (o.status & kStatusCapacity) && ctx->max_particles_req == 0;
                if ((o.status & kStatusCellOverflow) && !grow_cap) {
                    j.result = fail(ctx, GCMC_ERR_CELL_OVERFLOW, "gcmc_run_moves: cell capacity exceeded");
                    continue;
                }
                if ((o.status & kStatusCapacity) && !grow_n) {
                    j.result = fail(ctx, GCMC_ERR_CAPACITY, "gcmc_run_moves: max_particles exceeded");
                    continue;
                }
                const int ncap = grow_cap ? std::min(65535, ctx->cap + std::max(8, ctx->cap / 2)) : ctx->cap;
                const int64_t nmax = grow_n ? std::min<int64_t>(1ll << 24, ctx->maxN * 2) : ctx->maxN;
                gcmc_status rs = relayout(ctx, ncap, nmax);
                if (rs != GCMC_OK) j.result = rs;
                continue;
            }
            if (o.moves_done == 0)
                j.result = fail(ctx, GCMC_ERR_CUDA, "gcmc_run_moves: the chain kernel made no progress (status " +
                                                        std::to_string(o.status) + ", sites " + std::to_string(o.pad) + ")");
        }
        // the grown arrays must be visible to the next round's arguments
        for (auto &j : jobs) j.ctx->energy_valid = true;
    }
    return GCMC_OK;
}

// Runs the jobs with the given choice of W, or -- config < 0 -- picks one:
// the first quarter of the moves runs under choice 0 (a fresh configuration
// relaxes there, and its rates do not predict the rest), then every choice is
// timed on short chunks, twice, in the orders 0 .. K-1 and K-1 .. 0 (the sum
// cancels a steady drift of the chains), and the rest runs under the one
// with the smallest total (config returns it).  Every choice takes exactly
// the same moves, so tuning never changes the chain.
static gcmc_status run_jobs_tuned(std::vector<ChainJob> &jobs, cudaStream_t st, bool f32, int &config,
                                  LaunchBufs &B, int64_t *launches, std::string *err, bool use_graph,
                                  double *probe_ms, double *dev_ms = nullptr)
{
    if (config >= 0) return run_jobs(jobs, st, f32, config, B, launches, err, use_graph, dev_ms);
    int64_t remaining = INT64_MAX;
    for (auto &j : jobs) remaining = std::min<int64_t>(remaining, j.n_moves - j.done);
    const int64_t chunk = std::min<int64_t>(std::max<int64_t>(remaining / (8 * kChainConfigs), 256), 2048);
    if (remaining < 4 * chunk * kChainConfigs) {
        config = 0;
        return run_jobs(jobs, st, f32, config, B, launches, err, use_graph, dev_ms);
    }
    // runs the next `count` moves of every job under choice c; returns its time
    auto run_limited = [&](int c, int64_t count, float *ms_out) -> gcmc_status {
        std::vector<int64_t> saved(jobs.size());
        for (size_t k = 0; k < jobs.size(); ++k) {
            saved[k] = jobs[k].n_moves;
            jobs[k].n_moves = std::min<int64_t>(jobs[k].n_moves, jobs[k].done + count);
        }
        cudaEvent_t e0, e1;
        cudaEventCreate(&e0);
        cudaEventCreate(&e1);
        cudaEventRecord(e0, st);
        gcmc_status r = run_jobs(jobs, st, f32, c, B, launches, err, false, dev_ms);
        cudaEventRecord(e1, st);
        cudaEventSynchronize(e1);
        float ms = 0.f;
        cudaEventElapsedTime(&ms, e0, e1);
        cudaEventDestroy(e0);
        cudaEventDestroy(e1);
        for (size_t k = 0; k < jobs.size(); ++k) jobs[k].n_moves = saved[k];
        if (ms_out) *ms_out = ms;
        return r;
    };
    const int64_t burn = std::min<int64_t>(remaining / 4, remaining - 3 * chunk * kChainConfigs);
    gcmc_status r = run_limited(0, burn, nullptr);
    if (r != GCMC_OK) return r;
    double total[kChainConfigs] = {};
    for (int pass = 0; pass < 2; ++pass) {
        for (int i = 0; i < kChainConfigs; ++i) {
            const int c = pass == 0 ? i : kChainConfigs - 1 - i;
            float ms = 0.f;
            r = run_limited(c, chunk, &ms);
            if (r != GCMC_OK) return r;
            total[c] += ms;
        }
    }
    int bc = 0;
    for (int c = 0; c < kChainConfigs; ++c) {
        if (probe_ms) probe_ms[c] = total[c];
        if (total[c] < total[bc]) bc = c;
    }
    config = bc;
    return run_jobs(jobs, st, f32, config, B, launches, err, use_graph, dev_ms);
}

// The library's limit on the cells of a chain's box (97,936 in FP64 mode, 83,600
// in FP32 mode where a CTA may have 227 KB): it leaves the chain's state and four
// movers at least.  The FP32 share is part of the limit that callers know; both
// modes need the same room.
constexpr size_t kChainReserve = 36576, kChainReserveFp32 = 28672;

static gcmc_status check_chain_fits(gcmc_ctx *ctx)
{
    const size_t smem = ((size_t)ctx->ncell * sizeof(uint16_t) + 15) / 16 * 16;
    static_assert(sizeof(Shared) + sizeof(ChainArgs) + 4 * kMoverBytes + 2048 <= kChainReserve, "chain state");
    const size_t queues = ctx->precision == GCMC_FP32 ? kChainReserveFp32 : 0;
    if (smem + kChainReserve + queues > ctx->smem_optin)
        return fail(ctx, GCMC_ERR_INVALID_ARG, "gcmc_run_moves: too many cells (the limit counts two bytes of shared memory a cell)");
    if (ctx->T > 1023) return fail(ctx, GCMC_ERR_INVALID_ARG, "gcmc_run_moves: more than 1023 cells per side");
    return GCMC_OK;
}

gcmc_status run_moves(gcmc_ctx *ctx, uint64_t seed, uint64_t first, int64_t n_moves, const gcmc_move_mix *mix,
                      gcmc_move_stats *stats, gcmc_trace *trace)
{
    gcmc_status st = check_chain_fits(ctx);
    if (st != GCMC_OK) return st;
    if (!ctx->energy_valid) {
        st = total_energy(ctx, nullptr);
        if (st != GCMC_OK) return st;
    }
    const bool vir = (mix->flags & GCMC_MIX_VIRIAL) != 0;
    if (vir && !ctx->virial_valid) {
        st = total_energy(ctx, nullptr, true);
        if (st != GCMC_OK) return st;
    }
    static thread_local LaunchBufs bufs;
    std::vector<ChainJob> jobs(1);
    ChainJob &j = jobs[0];
    memset(&j, 0, sizeof(j));
    j.ctx = ctx;
    j.seed = seed;
    j.chain = 0;
    j.first = first;
    j.n_moves = n_moves;
    j.mix = *mix;
    j.trace = trace;
    j.result = GCMC_OK;
    j.agg.virial = vir ? ctx->virial : NAN;
    j.agg.sum_virial = vir ? 0.0 : NAN;
    ctx->last_refetch = 0;
    ctx->last_refines = 0;
    for (double &v : ctx->last_prof) v = 0.0;
    std::string err;
    st = run_jobs_tuned(jobs, ctx->stream, ctx->precision == GCMC_FP32, ctx->chain_config, bufs, &ctx->launches,
                        &err, false, nullptr);
    if (st != GCMC_OK) return fail(ctx, st, err);
    if (stats) *stats = j.agg;
    return j.result;
}

gcmc_status run_moves_micro(gcmc_ctx *ctx, uint64_t seed, uint64_t first, int64_t n_moves, const gcmc_move_mix *mix,
                            gcmc_move_stats *stats, gcmc_trace *trace)
{
    gcmc_status st;
    if (!ctx->mc_valid) {
        st = micro_build(ctx, ctx->mc_edge, ctx->mc_cap_req);
        if (st != GCMC_OK) return st;
    }
    if (!ctx->energy_valid) {
        st = total_energy(ctx, nullptr);
        if (st != GCMC_OK) return st;
    }
    static thread_local LaunchBufs bufs;
    std::vector<ChainJob> jobs(1);
    ChainJob &j = jobs[0];
    memset(&j, 0, sizeof(j));
    j.ctx = ctx;
    j.seed = seed;
    j.first = first;
    j.n_moves = n_moves;
    j.mix = *mix;
    j.trace = trace;
    j.result = GCMC_OK;
    j.agg.energy = ctx->energy;
    for (int q = 0; q < kMaxSpecies; ++q) j.agg.n[q] = ctx->n_host[q];
    j.agg.virial = j.agg.sum_virial = NAN;
    ctx->last_refetch = 0;
    ctx->last_refines = 0;
    std::string err;
    st = run_jobs(jobs, ctx->stream, ctx->precision == GCMC_FP32, 0, bufs, &ctx->launches, &err, false, nullptr, true);
    if (st != GCMC_OK) return fail(ctx, st, err);
    if (j.result == GCMC_ERR_NONFINITE) fail(ctx, j.result, "gcmc_run_moves_micro: the running energy is not finite");
    j.agg.chain_ms = 0.0;
    for (double &v : ctx->last_prof) v = 0.0;
    if (stats) *stats = j.agg;
    return j.result;
}

gcmc_status run_batch(gcmc_ctx *const *ctxs, int K, const uint64_t *seeds, uint64_t first, int64_t n_moves,
                      const gcmc_move_mix *mixes, gcmc_move_stats *stats, int &config, int64_t *launches,
                      std::string *err, cudaStream_t stream, bool use_graph, double *probe_ms, double *dev_ms,
                      gcmc_trace *const *traces)
{
    if (dev_ms) *dev_ms = 0.0;
    if (K <= 0) return GCMC_OK;
    const bool f32 = ctxs[0]->precision == GCMC_FP32;
    for (int k = 0; k < K; ++k) {
        if (!ctxs[k] || !ctxs[k]->built) {
            if (err) *err = "gcmc_batch_run_moves: a context has no cells";
            return GCMC_ERR_STATE;
        }
        if ((ctxs[k]->precision == GCMC_FP32) != f32) {
            if (err) *err = "gcmc_batch_run_moves: contexts of different precision";
            return GCMC_ERR_INVALID_ARG;
        }
        gcmc_status st = check_chain_fits(ctxs[k]);
        if (st != GCMC_OK) {
            if (err) *err = ctxs[k]->err;
            return st;
        }
        if (!ctxs[k]->energy_valid) {
            st = total_energy(ctxs[k], nullptr);
            if (st != GCMC_OK) {
                if (err) *err = ctxs[k]->err;
                return st;
            }
        }
        if ((mixes[k].flags & GCMC_MIX_VIRIAL) && !ctxs[k]->virial_valid) {
            st = total_energy(ctxs[k], nullptr, true);
            if (st != GCMC_OK) {
                if (err) *err = ctxs[k]->err;
                return st;
            }
        }
    }
    static thread_local LaunchBufs bufs;
    std::vector<ChainJob> jobs(K);
    // the chains' own streams first: their earlier work must be complete
    for (int k = 0; k < K; ++k) {
        cudaError_t e = cudaStreamSynchronize(ctxs[k]->stream);
        if (e != cudaSuccess) {
            if (err) *err = cudaGetErrorString(e);
            return GCMC_ERR_CUDA;
        }
    }
    for (int k = 0; k < K; ++k) {
        ChainJob &j = jobs[k];
        memset(&j, 0, sizeof(j));
        j.ctx = ctxs[k];
        j.seed = seeds[k];
        j.chain = (uint32_t)k;
        j.first = first;
        j.n_moves = n_moves;
        j.mix = mixes[k];
        j.trace = traces ? traces[k] : nullptr;
        j.result = GCMC_OK;
        const bool vir = (mixes[k].flags & GCMC_MIX_VIRIAL) != 0;
        j.agg.virial = vir ? ctxs[k]->virial : NAN;
        j.agg.sum_virial = vir ? 0.0 : NAN;
        ctxs[k]->last_refetch = 0;
        ctxs[k]->last_refines = 0;
        for (double &v : ctxs[k]->last_prof) v = 0.0;
    }
    gcmc_status st = run_jobs_tuned(jobs, stream, f32, config, bufs, launches, err, use_graph && stream != nullptr,
                                    probe_ms, dev_ms);
    if (st != GCMC_OK) return st;
    gcmc_status worst = GCMC_OK;
    for (int k = 0; k < K; ++k) {
        if (stats) stats[k] = jobs[k].agg;
        if (jobs[k].result != GCMC_OK && worst == GCMC_OK) worst = jobs[k].result;
    }
    return worst;
}

}  // namespace gcmc
