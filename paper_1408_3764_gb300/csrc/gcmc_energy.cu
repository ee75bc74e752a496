// gcmc_energy.cu -- cell-list energies on the compact cell-major layout:
//   k_trial_energy   energy of many trial points against their 27 cells
//                    (Algorithms 6 and 7); the points are binned by cell and
//                    one CTA evaluates all points of a cell against its
//                    neighbourhood, staged once into shared memory;
//   k_cell_energy    full-system energy and virial, one CTA per home cell
//                    over its half shell (the cell-list CalculateTotalEnergy
//                    of Sec. 3.1.1);
//   k_cell_grad      its hand-written gradient (positions, eps, sigma, virial).
// FP32 mode: an FP32 screen of every candidate, compensated FP32 pair terms
// and sums for the energies (float-float, lj_ff), FP32 pair terms for the
// gradient with compensated scalar sums; sums across cells in FP64.
// FP64 mode: everything in FP64.  k_cell_energy_padded (allocation-free
// energy) keeps plain FP32 pair terms and per-lane sums in FP32 mode.
#include <cmath>
#include <cstring>
#include <mutex>
#include <string>
#include <type_traits>

#include "gcmc_ctx.h"
#include "gcmc_stage.cuh"

namespace gcmc {

// Per-lane accumulators.  FP32 mode: plain FP32 sums (a lane adds a few
// dozen terms, so their rounding stays near 1e-6 of the terms' magnitudes);
// FP64 mode: FP64.
template <bool F32>
struct Acc;
template <>
struct Acc<true> {
    float e = 0.f, a = 0.f, w = 0.f;  // energy, |terms|, virial r U'(r) = -(3 m + 9 u)
    __device__ __forceinline__ void add(float u, float m)
    {
        e += u;
        a += m;
        w -= fmaf(3.f, m, 9.f * u);
    }
    __device__ __forceinline__ double ev() const { return (double)e; }
    __device__ __forceinline__ double av() const { return (double)a; }
};
template <>
struct Acc<false> {
    double e = 0.0, a = 0.0, w = 0.0;
    __device__ __forceinline__ void add(double u, double m)
    {
        e += u;
        a += m;
        w -= 3.0 * m + 9.0 * u;
    }
    __device__ __forceinline__ double ev() const { return e; }
    __device__ __forceinline__ double av() const { return a; }
};

template <bool F32>
__device__ __forceinline__ void pair_acc(const uint4 &p, const uint4 &q, uint32_t excl, uint64_t R2,
                                         int t, const FieldF &ff, const FieldD &fd, Acc<F32> &acc)
{
    if (q.w == excl) return;
    const GridSep s = grid_sep(p, q);
    if (s.g >= R2) return;
    const int k = t * kMaxSpecies + (int)tag_species(q.w);
    if constexpr (F32) {
        float u, m;
        lj_f32(s, ff.c4e[k], ff.sig2[k], u, m);
        acc.add(u, m);
    } else {
        double u, m;
        lj_f64(s, fd.rep[k], fd.att[k], u, m);
        acc.add(u, m);
    }
}


// ---------------------------------------------------------------------------
// Neighbourhood kernels.  One CTA per cell: the cell's neighbourhood (the 27
// cells, or the home cell and its half shell) is staged into shared memory
// by bulk copies (gcmc_stage.cuh), at most kBuf records per pass, and each
// staged record is converted once to float coordinates relative to the home
// cell's centre.  Warps take the cell's points (trial points or home
// particles) a few at a time, lanes the staged records, 32 a row: the FP32
// squared distance minus a bound just above rc^2 is accumulated from the
// bound, and its sign bit is shifted into the point's mask, so that a row
// costs seven instructions per point and one shared load for all of them.
// The set bits -- the ~15 % of the candidates inside the cutoff -- are then
// written to the warp's list and evaluated 32 at a time, where the exact
// integer squared distance decides: in compensated FP32 (lj_ff) in FP32 mode,
// in FP64 in FP64 mode, with every lane busy.
// What bounds them: instruction issue (FP32 mode), the FP64 pipe (FP64 mode).
// Screening with a vote and two population counts per row and a band test took
// 55 instructions per 32 candidates and 1,350 per trial point, now 760: 10^6
// points in the 2^20-particle mixture 1.49 -> 0.91 ms a call, its total energy
// with the cell build 1.22 -> 0.83 ms, a gradient step of 262,144 particles
// 1.88 -> 1.45 ms.
// Minimum image relative to the cell centre c: a partner within rc of a
// point p of the cell lies, along each axis, within rc + S/2 of c.  When
// S >= rc (T = floor(L / rc) >= 3) that is at most 1.5 S <= L / 2, so the
// wrapped difference q - c already gives the image nearest to p.  A box
// with 2 rc <= L < 3 rc has T = 3 and S < rc: there the FP32 separation is
// wrapped once more into [-L/2, L/2] (wrap = 1).  The queued pairs use the
// exact wrapped integer difference p - q.
// ---------------------------------------------------------------------------
// staged records per pass, in rows of 32 (a mask word holds at most 32): a
// little more than a neighbourhood of 27 cells (14 for the half shell) holds
// at liquid densities, so that most cells take one pass and shared memory
// holds many CTAs (nine of four warps).  With 768 for both (six CTAs) the
// trial energies took 1.09 ms and the total energy 0.95 ms.
constexpr int kBufFull = 544, kBufHalf = 384;
// ... and where plain FP32 sums of a point's terms are results (forces, table
// gradients, magnitudes): their order, the pairs of a pass by staged index, is
// part of the result to its last digits
constexpr int kBufOrdered = 896;
constexpr int kPChunk = 64;   // points per chunk (per-point sums in shared memory)
constexpr int kNbWarps = 4;   // warps of a neighbourhood CTA (two: trial energies 14 % slower; eight: total energy 18 %)
constexpr int kNbQ = 128;     // queue entries per warp of the other trial kernels (a ring: up to 31 + 2 x 32 pending)
static_assert(kBufFull % 32 == 0 && kBufHalf % 32 == 0 && kBufOrdered % 32 == 0 && kBufFull <= 1024 &&
                  kBufHalf <= 1024 && kBufOrdered <= 1024 && kPChunk <= 64,
              "list entries and masks");

// Grid coordinate of the centre of cell k along an axis of T cells.
__device__ __forceinline__ uint32_t cell_centre(int k, int T)
{
    return (uint32_t)((((unsigned long long)(2 * k + 1)) << 32) / (unsigned long long)(2 * T));
}

__device__ __forceinline__ float rel_f(uint32_t a, uint32_t c) { return (float)(int)(a - c); }

// Shared state of a neighbourhood CTA.
template <int KB>
struct __align__(16) NbShared {
    static constexpr int kBuf = KB;
    uint4 raw[KB];       // staged records (X, Y, Z, tag)
    float4 fl[KB];       // the same relative to the home cell centre, tag bits in .w
    // pairs inside the cutoff: staged index | point << 10; up to 31 left over
    // and a point's pairs
    unsigned short list[kNbWarps][KB + 32];
    RunList runs;
    uint64_t bar;
    // the species pairs' constants: FP32 mode float4 (c4e, c4e_lo, sig2,
    // sig2_lo), FP64 mode (rep, att), for the gradient (c4e, sig2) -- lanes of
    // one warp read several
    union {
        float4 f[kMaxSpecies * kMaxSpecies];
        double2 d[kMaxSpecies * kMaxSpecies];
    } field;
};

template <bool F32, bool GRAD, class SH>
__device__ __forceinline__ void nb_field(SH &sh, const FieldF &ff, const FieldD &fd)
{
    for (int k = threadIdx.x; k < kMaxSpecies * kMaxSpecies; k += blockDim.x) {
        if constexpr (F32) sh.field.f[k] = make_float4(ff.c4e[k], ff.c4e_lo[k], ff.sig2[k], ff.sig2_lo[k]);
        else sh.field.d[k] = GRAD ? make_double2(fd.c4e[k], fd.sig2[k]) : make_double2(fd.rep[k], fd.att[k]);
    }
}

__device__ __forceinline__ float wrap_grid(float d)
{
    return fmaf(-4294967296.0f, rintf(d * 2.3283064365386963e-10f), d);  // d - 2^32 rint(d / 2^32)
}

// Screens the staged records of `rows` rows against NP points (coordinates
// relative to the centre): bit rows - 1 - r of mask[p] in lane l stands for
// record 32 r + l.  BAND: inner[p] holds those inside by more than `band` too.
template <bool WRAP, int NP, bool BAND>
__device__ __forceinline__ void nb_rows(const float4 *fl, int rows, const float3 *pf, float r2hi, float band,
                                        uint32_t *mask, uint32_t *inner)
{
    fl += threadIdx.x & 31;
#pragma unroll
    for (int p = 0; p < NP; ++p) {
        mask[p] = 0u;
        if (BAND) inner[p] = 0u;
    }
#pragma unroll 2
    for (int r = 0; r < rows; ++r) {
        const float4 q = fl[32 * r];
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            float dx = pf[p].x - q.x, dy = pf[p].y - q.y, dz = pf[p].z - q.z;
            if (WRAP) {
                dx = wrap_grid(dx);
                dy = wrap_grid(dy);
                dz = wrap_grid(dz);
            }
            const float d = fmaf(dx, dx, fmaf(dy, dy, fmaf(dz, dz, -r2hi)));
            mask[p] = __funnelshift_l(__float_as_uint(d), mask[p], 1);
            if (BAND) inner[p] = __funnelshift_l(__float_as_uint(d + band), inner[p], 1);
        }
    }
}

// The same for the nst staged records (what lies behind them is left out):
// those below the bound r2hi, a little above the cutoff.
template <int NP>
__device__ __forceinline__ void nb_screen(const float4 *fl, int nst, const float3 *pf, float r2hi, bool wrap,
                                          uint32_t *mask)
{
    const int rows = (nst + 31) >> 5;
    if (wrap) nb_rows<true, NP, false>(fl, rows, pf, r2hi, 0.f, mask, nullptr);
    else nb_rows<false, NP, false>(fl, rows, pf, r2hi, 0.f, mask, nullptr);
    const uint32_t keep = 32 * (rows - 1) + (int)(threadIdx.x & 31) < nst ? ~0u : ~1u;
#pragma unroll
    for (int p = 0; p < NP; ++p) mask[p] &= keep;
}

// Exactly those inside the cutoff: the exact integer test decides in the thin
// band around it.
template <int NP>
__device__ __forceinline__ void nb_screen_exact(const float4 *fl, const uint4 *raw, int nst, const uint4 *P,
                                                const float3 *pf, uint64_t R2, float r2hi, bool wrap, uint32_t *mask)
{
    const int rows = (nst + 31) >> 5, lane = threadIdx.x & 31;
    const float band = 2e-5f * r2hi;
    uint32_t inner[NP];
    if (wrap) nb_rows<true, NP, true>(fl, rows, pf, r2hi, band, mask, inner);
    else nb_rows<false, NP, true>(fl, rows, pf, r2hi, band, mask, inner);
    const uint32_t keep = 32 * (rows - 1) + lane < nst ? ~0u : ~1u;
#pragma unroll
    for (int p = 0; p < NP; ++p) {
        mask[p] &= keep;
        uint32_t x = mask[p] & ~inner[p];
        while (x) {
            const int b = 31 - __clz((int)x);
            if (grid_sep(P[p], raw[32 * (rows - 1 - b) + lane]).g >= R2) mask[p] ^= 1u << b;
            x ^= 1u << b;
        }
    }
}

// Writes the records of a mask to the list by ascending index; returns their
// number.
__device__ __forceinline__ int nb_list_ordered(unsigned short *list, uint32_t mask, int rows)
{
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    int n = 0;
#pragma unroll 2
    for (int r = 0; r < rows; ++r) {
        const bool in = (mask >> (rows - 1 - r)) & 1u;
        const unsigned b = __ballot_sync(0xffffffffu, in);
        if (in) list[n + __popc(b & lt)] = (unsigned short)(32 * r + lane);
        n += __popc(b);
    }
    return n;
}

// Appends the records of a mask to the warp's list of n entries (tag in the
// bits above the staged index); returns the new length.
__device__ __forceinline__ int nb_append(unsigned short *list, int n, uint32_t mask, int rows, int tag)
{
    const int c = __popc(mask), inc = warp_inclusive_scan(c);
    unsigned short *q = list + n + inc - c;
    const int f0 = (rows - 1) * 32 + (int)(threadIdx.x & 31) + tag;
    while (mask) {
        const int b = 31 - __clz((int)mask);
        *q++ = (unsigned short)(f0 - 32 * b);
        mask ^= 1u << b;
    }
    return n + __shfl_sync(0xffffffffu, inc, 31);
}

// Evaluates the whole list, 32 entries at a time.
template <typename Drain>
__device__ __forceinline__ void nb_flush(const unsigned short *list, int n, Drain &D)
{
    __syncwarp();
    for (int h = (int)(threadIdx.x & 31); h < n; h += 32) D(list[h]);
    __syncwarp();
}

// Evaluates whole groups of 32 and moves the rest to the front; returns its
// length.
template <typename Drain>
__device__ __forceinline__ int nb_drain(unsigned short *list, int n, Drain &D)
{
    const int lane = threadIdx.x & 31, full = n & ~31;
    __syncwarp();
    for (int h = lane; h < full; h += 32) D(list[h]);
    unsigned short v = 0;
    if (full + lane < n) v = list[full + lane];
    __syncwarp();
    if (full && full + lane < n) list[lane] = v;
    return n - full;
}

// Sums of several values across the warp at once: each step adds half of the
// lanes' values to the other half's and halves their number, so V values take
// about V + 5 - log2 V additions instead of 5 V.  V a power of two up to 16;
// the sum of value k ends in every lane l with (l >> (5 - log2 V)) == k.
__device__ __forceinline__ double shfl_xor(double v, int o) { return __shfl_xor_sync(0xffffffffu, v, o); }
__device__ __forceinline__ FF shfl_xor(FF v, int o)
{
    return FF{__shfl_xor_sync(0xffffffffu, v.hi, o), __shfl_xor_sync(0xffffffffu, v.lo, o)};
}
__device__ __forceinline__ double sum_of(double a, double b) { return a + b; }
__device__ __forceinline__ FF sum_of(FF a, FF b) { return ff_add(a, b); }

template <int V, typename T>
__device__ __forceinline__ T warp_sum_many(T *v)
{
    const int lane = threadIdx.x & 31;
    int o = 16;
#pragma unroll
    for (int half = V / 2; half > 0; half >>= 1) {
        const bool up = lane & o;
#pragma unroll
        for (int k = 0; k < half; ++k) {
            const T keep = up ? v[k + half] : v[k], send = up ? v[k] : v[k + half];
            v[k] = sum_of(keep, shfl_xor(send, o));
        }
        o >>= 1;
    }
    T x = v[0];
#pragma unroll
    for (int k = V; k < 32; k <<= 1) {
        x = sum_of(x, shfl_xor(x, o));
        o >>= 1;
    }
    return x;
}
// Stages the items [w0, w1) of the neighbourhood into the shared buffers
// (bulk copies, then the float conversion).  Returns false -- in every
// thread -- when the copy did not land within the wait limit; the timeout
// bit is then set and the block must return.
template <class SH>
__device__ __forceinline__ bool nb_stage(SH &sh, const uint4 *__restrict__ cpos, int w0, int w1,
                                         uint32_t cx0, uint32_t cy0, uint32_t cz0, unsigned &parity,
                                         int *__restrict__ status)
{
    __syncthreads();  // the previous pass's readers are done with the buffers
    if (w1 <= w0) return true;
    if (threadIdx.x == 0) stage_issue(cpos, sh.runs, w0, w1, sh.raw, &sh.bar);
    const bool ok = stage_wait(&sh.bar, parity, 1000000000ull);
    if (__syncthreads_or(!ok)) {
        if (threadIdx.x == 0) {
            atomicOr(status, kStatusTimeout);
            stage_wait(&sh.bar, parity, 1000000000ull);  // the copies in flight land before the block ends
        }
        __syncthreads();
        return false;
    }
    parity ^= 1u;
    for (int f = threadIdx.x; f < w1 - w0; f += blockDim.x) {
        const uint4 r = sh.raw[f];
        sh.fl[f] = make_float4(rel_f(r.x, cx0), rel_f(r.y, cy0), rel_f(r.z, cz0), __uint_as_float(r.w));
    }
    __syncthreads();
    return true;
}

// ---- trial energies ---------------------------------------------------
// Per trial point: species, the excluded particle's tag, the grid position.
struct TrialPt {
    uint4 P;       // grid X, Y, Z; .w = species
    uint32_t excl; // tag of the excluded particle, or ~0
    int idx;       // the point's input index
};

template <bool F32, class SH>
struct TrialDrain {
    const SH &sh;
    uint4 P;
    uint32_t excl;
    unsigned long long R2;
    float eh = 0.f, el = 0.f, mag = 0.f;
    double rep = 0.0, att = 0.0;
    __device__ TrialDrain(const SH &s, const TrialPt &p, unsigned long long r) : sh(s), P(p.P), excl(p.excl), R2(r)
    {
    }
    __device__ __forceinline__ void operator()(int f)
    {
        const uint4 r = sh.raw[f];
        const int ex = (int)(P.x - r.x), ey = (int)(P.y - r.y), ez = (int)(P.z - r.z);
        const unsigned long long g = (unsigned long long)((long long)ex * ex) +
                                     (unsigned long long)((long long)ey * ey) +
                                     (unsigned long long)((long long)ez * ez);
        if (g >= R2 || r.w == excl) return;
        const int k = (int)P.w * kMaxSpecies + (int)tag_species(r.w);
        if constexpr (F32) {
            const float4 c = sh.field.f[k];
            float uh, ul, m;
            lj_ff(ex, ey, ez, c.x, c.y, c.z, c.w, uh, ul, m);
            ff_acc(eh, el, uh, ul);
            mag += m;
        } else {
            const double2 c = sh.field.d[k];
            lj_f64_add(g, c.x, c.y, rep, att);
        }
    }
};

// Trial points binned by cell: cell c holds the points pts[ps[c] .. ps[c+1]).
// Each warp screens two points together (they share the loads of the staged
// records), evaluates the pairs of each and sums both across its lanes at once.
// ABS (FP64 mode): with the sums of |rep| + |att|.
template <bool F32, bool ABS>
__global__ void __launch_bounds__(kNbWarps * 32) k_trial_energy(
    const TrialPt *__restrict__ pts, const int32_t *__restrict__ ps, const uint4 *__restrict__ cpos,
    const int32_t *__restrict__ cs, int T, int64_t ncell, uint64_t R2, float r2hi, bool wrap,
    const __grid_constant__ FieldF ff, const __grid_constant__ FieldD fd, double *__restrict__ out,
    double *__restrict__ out_abs, int *__restrict__ status)
{
    extern __shared__ __align__(128) unsigned char dyn[];
    static_assert(!(F32 && ABS), "k_trial_scaled");
    using SH = NbShared<kBufFull>;
    constexpr int kBuf = SH::kBuf;
    SH &sh = *reinterpret_cast<SH *>(dyn);
    // per-point sums over the passes: FP32 mode float-float; FP64 mode energy
    // and uabs
    __shared__ typename std::conditional<F32, float2, double2>::type part[kPChunk];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (threadIdx.x == 0) mbar_init(&sh.bar, 1);
    nb_field<F32, false>(sh, ff, fd);
    __syncthreads();
    unsigned parity = 0;
    for (int64_t c = blockIdx.x; c < ncell; c += gridDim.x) {
        const int p0 = ps[c], p1 = ps[c + 1];
        if (p1 == p0) continue;  // uniform across the block
        const int cx = (int)(c % T), cy = (int)((c / T) % T), cz = (int)(c / ((int64_t)T * T));
        __syncthreads();
        if (w == 0) runs27(cs, T, cx, cy, cz, sh.runs);
        __syncthreads();
        const int total = sh.runs.end[17];
        const uint32_t cx0 = cell_centre(cx, T), cy0 = cell_centre(cy, T), cz0 = cell_centre(cz, T);
        for (int pb = p0; pb < p1; pb += kPChunk) {
            const int pn = min(kPChunk, p1 - pb);
            for (int base = 0; base < max(total, 1); base += kBuf) {
                const int nst = max(min(kBuf, total - base), 0);
                if ((base > 0 || pb == p0 || total > kBuf) &&
                    !nb_stage(sh, cpos, base, base + nst, cx0, cy0, cz0, parity, status))
                    return;
                const int rows = (nst + 31) >> 5;
                for (int i = 2 * w; i < pn; i += 2 * kNbWarps) {
                    const TrialPt t0 = pts[pb + i], t1 = pts[pb + min(i + 1, pn - 1)];
                    const float3 pf[2] = {make_float3(rel_f(t0.P.x, cx0), rel_f(t0.P.y, cy0), rel_f(t0.P.z, cz0)),
                                          make_float3(rel_f(t1.P.x, cx0), rel_f(t1.P.y, cy0), rel_f(t1.P.z, cz0))};
                    uint32_t mask[2];
                    TrialDrain<F32, SH> D0(sh, t0, R2), D1(sh, t1, R2);
                    unsigned short *list = sh.list[w];
                    nb_screen<2>(sh.fl, nst, pf, r2hi, wrap, mask);
                    nb_flush(list, nb_append(list, 0, mask[0], rows, 0), D0);
                    if (i + 1 < pn) nb_flush(list, nb_append(list, 0, mask[1], rows, 0), D1);
                    // lane 0 gets point i, lane 16 point i + 1
                    const int k = i + (lane >> 4);
                    const bool mine = (lane & 15) == 0 && k < pn;
                    if constexpr (F32) {
                        FF e[2] = {FF{D0.eh, D0.el}, FF{D1.eh, D1.el}};
                        FF s = warp_sum_many<2>(e);
                        if (mine) {
                            if (base > 0) s = ff_add(FF{part[k].x, part[k].y}, s);
                            part[k] = make_float2(s.hi, s.lo);
                        }
                    } else {
                        double e[2] = {D0.rep - D0.att, D1.rep - D1.att}, m[2] = {D0.rep + D0.att, D1.rep + D1.att};
                        double s = warp_sum_many<2>(e), a = 0.0;
                        if constexpr (ABS) a = warp_sum_many<2>(m);
                        if (mine) {
                            if (base > 0) {
                                s += part[k].x;
                                a += part[k].y;
                            }
                            part[k] = make_double2(s, a);
                        }
                    }
                }
            }
            __syncthreads();
            for (int i = threadIdx.x; i < pn; i += blockDim.x) {
                const int k = pts[pb + i].idx;
                out[k] = F32 ? ff_value((float)part[i].x, (float)part[i].y) : (double)part[i].x;
                if constexpr (ABS) out_abs[k] = part[i].y;
            }
            __syncthreads();  // the sums are read before the next chunk's
        }
    }
}

// FP32 mode with the sums of |rep| + |att|, which are plain FP32: their order --
// the pairs of a pass of kBufOrdered records by ascending index, 32 at a time --
// is part of the result to its last digits.  One point per warp, two rows a
// step, a vote and a population count each, which lists the pairs in that order
// as it screens them.  Masks and lists as above, put in order afterwards, took
// 1.40 instead of 1.25 ms for 800,000 points against 2^20 particles.
constexpr int kScaledWarps = 8;
struct __align__(16) ScaledShared {
    uint4 raw[kBufOrdered];
    float4 fl[kBufOrdered];
    int q[kScaledWarps][kNbQ];
    RunList runs;
    uint64_t bar;
    union {
        float4 f[kMaxSpecies * kMaxSpecies];
        double2 d[kMaxSpecies * kMaxSpecies];
    } field;
};

__global__ void __launch_bounds__(kScaledWarps * 32) k_trial_scaled(
    const TrialPt *__restrict__ pts, const int32_t *__restrict__ ps, const uint4 *__restrict__ cpos,
    const int32_t *__restrict__ cs, int T, int64_t ncell, uint64_t R2, float r2hi, bool wrap,
    const __grid_constant__ FieldF ff, const __grid_constant__ FieldD fd, double *__restrict__ out,
    double *__restrict__ out_abs, int *__restrict__ status)
{
    extern __shared__ __align__(128) unsigned char dyn[];
    using SH = ScaledShared;
    SH &sh = *reinterpret_cast<SH *>(dyn);
    __shared__ float4 part[kPChunk];  // per-point sums over the passes: hi, lo, uabs
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const unsigned lt = (1u << lane) - 1u;
    const float r2lo = r2hi - 2e-5f * r2hi;
    if (threadIdx.x == 0) mbar_init(&sh.bar, 1);
    nb_field<true, false>(sh, ff, fd);
    __syncthreads();
    unsigned parity = 0;
    int *Q = sh.q[w];
    for (int64_t c = blockIdx.x; c < ncell; c += gridDim.x) {
        const int p0 = ps[c], p1 = ps[c + 1];
        if (p1 == p0) continue;  // uniform across the block
        const int cx = (int)(c % T), cy = (int)((c / T) % T), cz = (int)(c / ((int64_t)T * T));
        __syncthreads();
        if (w == 0) runs27(cs, T, cx, cy, cz, sh.runs);
        __syncthreads();
        const int total = sh.runs.end[17];
        const uint32_t cx0 = cell_centre(cx, T), cy0 = cell_centre(cy, T), cz0 = cell_centre(cz, T);
        for (int pb = p0; pb < p1; pb += kPChunk) {
            const int pn = min(kPChunk, p1 - pb);
            for (int base = 0; base < max(total, 1); base += kBufOrdered) {
                const int nst = max(min(kBufOrdered, total - base), 0);
                if ((base > 0 || pb == p0 || total > kBufOrdered) &&
                    !nb_stage(sh, cpos, base, base + nst, cx0, cy0, cz0, parity, status))
                    return;
                for (int i = w; i < pn; i += kScaledWarps) {
                    const TrialPt tp = pts[pb + i];
                    const float3 pf = make_float3(rel_f(tp.P.x, cx0), rel_f(tp.P.y, cy0), rel_f(tp.P.z, cz0));
                    TrialDrain<true, SH> D(sh, tp, R2);
                    int head = 0, n = 0;
                    for (int b = 0; b < nst; b += 64) {
                        bool in[2], band[2];
#pragma unroll
                        for (int u = 0; u < 2; ++u) {
                            const int f = b + 32 * u + lane;
                            in[u] = band[u] = false;
                            if (f < nst) {
                                const float4 q = sh.fl[f];
                                float dx = pf.x - q.x, dy = pf.y - q.y, dz = pf.z - q.z;
                                if (wrap) {
                                    dx = wrap_grid(dx);
                                    dy = wrap_grid(dy);
                                    dz = wrap_grid(dz);
                                }
                                const float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
                                const bool other = __float_as_uint(q.w) != tp.excl;
                                in[u] = other && r2 < r2lo;
                                band[u] = other && r2 >= r2lo && r2 <= r2hi;
                            }
                        }
                        // inside the thin band around rc^2 the exact integer test decides
                        if (__any_sync(0xffffffffu, band[0] || band[1])) {
#pragma unroll
                            for (int u = 0; u < 2; ++u)
                                if (band[u]) in[u] = grid_sep(tp.P, sh.raw[b + 32 * u + lane]).g < R2;
                        }
                        const unsigned b0 = __ballot_sync(0xffffffffu, in[0]), b1 = __ballot_sync(0xffffffffu, in[1]);
                        if ((b0 | b1) == 0u) continue;
                        const int end = head + n, n0 = __popc(b0);
                        if (in[0]) Q[(end + __popc(b0 & lt)) & (kNbQ - 1)] = b + lane;
                        if (in[1]) Q[(end + n0 + __popc(b1 & lt)) & (kNbQ - 1)] = b + 32 + lane;
                        n += n0 + __popc(b1);
                        if (n >= 32) {
                            __syncwarp();
                            do {
                                D(Q[(head + lane) & (kNbQ - 1)]);
                                head = (head + 32) & (kNbQ - 1);
                                n -= 32;
                            } while (n >= 32);
                            __syncwarp();
                        }
                    }
                    __syncwarp();
                    if (lane < n) D(Q[(head + lane) & (kNbQ - 1)]);
                    __syncwarp();
                    FF s = ff_warp_sum(FF{D.eh, D.el});
                    float a = warp_sum(D.mag);
                    if (lane == 0) {
                        if (base > 0) {
                            s = ff_add(FF{part[i].x, part[i].y}, s);
                            a += part[i].z;
                        }
                        part[i] = make_float4(s.hi, s.lo, a, 0.f);
                    }
                }
            }
            __syncthreads();
            for (int i = threadIdx.x; i < pn; i += blockDim.x) {
                const int k = pts[pb + i].idx;
                out[k] = ff_value(part[i].x, part[i].y);
                out_abs[k] = (double)part[i].z;
            }
            __syncthreads();  // the sums are read before the next chunk's
        }
    }
}

// ---- a few trial points ---------------------------------------------------
// One CTA per point, straight from the caller's arrays: four warps take the
// records of the 27 cells (18 runs of the compact layout) two per lane and
// pass, the FP32 squared distance screens them, and the pairs that pass are
// queued and evaluated 32 at a time, the exact integer test deciding.  A call
// is one launch and one wait: binning the points takes two fills, five
// launches and a copy before and after the energies, and a pass over every
// cell, which is what bounds small calls: 64 points against 2,048 particles
// take 16 us instead of 52 (FP64), against 2^20 particles 16 instead of 78.
// Many points share their cell's staged records, so the binned path wins where
// the points are many, the later the more cells they are spread over (about
// 12 ns a cell that holds some).  Direct and binned, against 2,048 / 20,000 /
// 2^20 particles: FP64 at 4,096 points 44 / 44 / 45 us and (8,192 points) 61 /
// 62 / 126, where direct takes twice the 44; FP32 at 16,384 points 53 / 54 / 62
// and 71 / 61 / 153; with |rep| + |att| 41 / 35 / 60 and 85 / 74 / 224.  The
// lines below follow these, with a share of the cells for large boxes.
constexpr int kDirectWarps = 4;
static int64_t direct_points(const gcmc_ctx *ctx, bool abs)
{
    if (ctx->precision == GCMC_FP64) return std::max<int64_t>(4096, ctx->ncell / 6);
    return abs ? std::max<int64_t>(32768, 2 * ctx->ncell) : std::max<int64_t>(16384, ctx->ncell);
}

// ORDERED (FP32 mode with |rep| + |att|): one warp per point, the pairs listed
// by ascending index in passes of kBufOrdered records as the binned path lists
// them, so that the plain FP32 sums are the same bits.
template <bool F32, bool ORDERED>
__global__ void __launch_bounds__((ORDERED ? 1 : kDirectWarps) * 32) k_trial_direct(
    const double *__restrict__ pos, const int32_t *__restrict__ species, const int64_t *__restrict__ exclude, double q,
    int T, int S, const uint4 *__restrict__ cpos, const int32_t *__restrict__ cs, uint64_t R2, float r2hi,
    const __grid_constant__ FieldF ff, const __grid_constant__ FieldD fd, double *__restrict__ out,
    double *__restrict__ out_abs, volatile int *__restrict__ host_status)
{
    constexpr int NW = ORDERED ? 1 : kDirectWarps, NT = NW * 32;
    constexpr int kPass = ORDERED ? kBufOrdered : 1 << 30;
    static_assert(kBufOrdered % (2 * 32) == 0, "a pass is whole steps");
    __shared__ RunList runs;
    __shared__ int4 queue[NW][kNbQ];
    __shared__ double2 red[NW];
    __shared__ float4 redf[NW];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t k = blockIdx.x;
    const int t = species[k];
    bool ok = t >= 0 && t < S;
    uint32_t X[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) X[a] = quantize_axis(pos[3 * k + a], q, ok);
    if (!ok) {  // uniform across the block
        if (threadIdx.x == 0) {
            *host_status = kStatusBadInput;
            out[k] = __longlong_as_double(0x7ff8000000000000ll);
            if (out_abs) out_abs[k] = out[k];
        }
        return;
    }
    uint32_t excl = 0xFFFFFFFFu;
    if (exclude) {
        const int64_t x = exclude[k];
        if (x >= 0) excl = make_tag((uint32_t)(x & 0xFFFFFFFFll), (uint32_t)(x >> 32));
    }
    if (w == 0)
        runs27(cs, T, cell_coord(X[0], (uint32_t)T), cell_coord(X[1], (uint32_t)T), cell_coord(X[2], (uint32_t)T), runs);
    __syncthreads();
    const int total = runs.end[17];
    int4 *Q = queue[w];
    const unsigned lt = (1u << lane) - 1u;
    int head = 0, nq = 0;
    float eh = 0.f, el = 0.f, mag = 0.f;
    double rep = 0.0, att = 0.0;
    FF sum = {0.f, 0.f};  // ORDERED: of the passes
    float sum_mag = 0.f;
    auto drain = [&](int n) {
        __syncwarp();
        if (lane < n) {
            const int4 p = Q[(head + lane) & (kNbQ - 1)];
            const unsigned long long g = (unsigned long long)((long long)p.x * p.x) +
                                         (unsigned long long)((long long)p.y * p.y) +
                                         (unsigned long long)((long long)p.z * p.z);
            if (g < R2) {
                const int c = t * kMaxSpecies + p.w;
                if constexpr (F32) {
                    float uh, ul, m;
                    lj_ff(p.x, p.y, p.z, ff.c4e[c], ff.c4e_lo[c], ff.sig2[c], ff.sig2_lo[c], uh, ul, m);
                    ff_acc(eh, el, uh, ul);
                    mag += m;
                } else {
                    lj_f64_add(g, fd.rep[c], fd.att[c], rep, att);
                }
            }
        }
        head = (head + n) & (kNbQ - 1);
        nq -= n;
        __syncwarp();
    };
    for (int base = 0; base < total; base += 2 * NT) {
        uint4 r[2];
        bool have[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int f = base + u * NT + (int)threadIdx.x;
            have[u] = f < total;
            r[u] = make_uint4(0, 0, 0, 0);
            if (have[u]) {
                // the first run that ends after f
                int lo = 0, hi = kMaxRuns - 1;
                while (lo < hi) {
                    const int mid = (lo + hi) >> 1;
                    if (runs.end[mid] > f) hi = mid;
                    else lo = mid + 1;
                }
                r[u] = cpos[runs.start[lo] + f - (lo ? runs.end[lo - 1] : 0)];
            }
        }
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int ex = (int)(X[0] - r[u].x), ey = (int)(X[1] - r[u].y), ez = (int)(X[2] - r[u].z);
            const float gx = (float)ex, gy = (float)ey, gz = (float)ez;
            bool in = have[u] && r[u].w != excl && fmaf(gx, gx, fmaf(gy, gy, gz * gz)) <= r2hi;
            if (ORDERED && in) in = grid_sep(make_uint4(X[0], X[1], X[2], 0u), r[u]).g < R2;
            const unsigned b = __ballot_sync(0xffffffffu, in);
            if (in) Q[(head + nq + __popc(b & lt)) & (kNbQ - 1)] = make_int4(ex, ey, ez, (int)tag_species(r[u].w));
            nq += __popc(b);
        }
        while (nq >= 32) drain(32);
        if (ORDERED && ((base + 2 * NT) % kPass == 0 || base + 2 * NT >= total)) {
            if (nq > 0) drain(nq);
            sum = ff_add(sum, ff_warp_sum(FF{eh, el}));
            sum_mag += warp_sum(mag);
            eh = el = mag = 0.f;
        }
    }
    if (nq > 0) drain(nq);
    if constexpr (F32) {
        const FF s = ORDERED ? sum : ff_warp_sum(FF{eh, el});
        const float a = ORDERED ? sum_mag : warp_sum(mag);
        if (lane == 0) redf[w] = make_float4(s.hi, s.lo, a, 0.f);
    } else {
        const double e = warp_sum(rep - att), a = warp_sum(rep + att);
        if (lane == 0) red[w] = make_double2(e, a);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double e, a;
        if constexpr (F32) {
            FF s = {redf[0].x, redf[0].y};
            float ua = redf[0].z;
            for (int i = 1; i < NW; ++i) {
                s = ff_add(s, FF{redf[i].x, redf[i].y});
                ua += redf[i].z;
            }
            e = ff_value(s.hi, s.lo);
            a = (double)ua;
        } else {
            e = red[0].x;
            a = red[0].y;
            for (int i = 1; i < NW; ++i) {
                e += red[i].x;
                a += red[i].y;
            }
        }
        out[k] = e;
        if (out_abs) out_abs[k] = a;
    }
}

// Quantises the trial points, bins them by cell (count per cell) and keeps
// their exclusion tags; bad input gets NaN at once and no cell.
__global__ void k_trial_bin(const double *__restrict__ pos, const int32_t *__restrict__ species,
                            const int64_t *__restrict__ exclude, int64_t m, double q, int T, int S,
                            TrialPt *__restrict__ tmp, int32_t *__restrict__ cellid, int32_t *__restrict__ count,
                            double *__restrict__ out, double *__restrict__ out_abs, int *__restrict__ status)
{
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < m; k += (int64_t)gridDim.x * blockDim.x) {
        const int s = species[k];
        bool ok = s >= 0 && s < S;
        uint32_t X[3] = {0u, 0u, 0u};
#pragma unroll
        for (int a = 0; a < 3; ++a) X[a] = quantize_axis(pos[3 * k + a], q, ok);
        if (!ok) {
            atomicOr(status, kStatusBadInput);
            out[k] = __longlong_as_double(0x7ff8000000000000ll);
            if (out_abs) out_abs[k] = out[k];
            cellid[k] = -1;
            continue;
        }
        uint32_t excl = 0xFFFFFFFFu;
        if (exclude) {
            const int64_t x = exclude[k];
            if (x >= 0) excl = make_tag((uint32_t)(x & 0xFFFFFFFFll), (uint32_t)(x >> 32));
        }
        const int c = cell_of(X[0], X[1], X[2], T);
        TrialPt tp;
        tp.P = make_uint4(X[0], X[1], X[2], (uint32_t)s);
        tp.excl = excl;
        tp.idx = (int)k;
        tmp[k] = tp;
        cellid[k] = c;
        atomicAdd(&count[c], 1);
    }
}

// Scatters the binned points into their cells' ranges (order within a cell
// does not matter: each point's sum is computed by one warp on its own).
__global__ void k_trial_place(const TrialPt *__restrict__ tmp, const int32_t *__restrict__ cellid, int64_t m,
                              const int32_t *__restrict__ ps, int32_t *__restrict__ fill, TrialPt *__restrict__ pts)
{
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < m; k += (int64_t)gridDim.x * blockDim.x) {
        const int c = cellid[k];
        if (c < 0) continue;
        pts[ps[c] + atomicAdd(&fill[c], 1)] = tmp[k];
    }
}

// ---- full-system energy ---------------------------------------------------
// List entries of the full-system energy: the staged partner's index, the
// home particle's index in the chunk above it, so that the pairs of several
// home particles share one evaluation pass.
template <bool F32, class SH>
struct PairDrain {
    const SH &sh;
    const uint4 *home;
    unsigned long long R2;
    float eh = 0.f, el = 0.f, wh = 0.f, wl = 0.f;
    double rep = 0.0, att = 0.0;
    __device__ PairDrain(const SH &s, const uint4 *h, unsigned long long r) : sh(s), home(h), R2(r) {}
    __device__ __forceinline__ void operator()(int e)
    {
        const uint4 P = home[e >> 10];
        const uint4 r = sh.raw[e & 1023];
        const int k = (int)tag_species(P.w) * kMaxSpecies + (int)tag_species(r.w);
        const int ex = (int)(P.x - r.x), ey = (int)(P.y - r.y), ez = (int)(P.z - r.z);
        const unsigned long long g = (unsigned long long)((long long)ex * ex) +
                                     (unsigned long long)((long long)ey * ey) +
                                     (unsigned long long)((long long)ez * ez);
        if (g >= R2) return;
        if constexpr (F32) {
            const float4 c = sh.field.f[k];
            float uh, ul, m;
            lj_ff(ex, ey, ez, c.x, c.y, c.z, c.w, uh, ul, m);
            ff_acc(eh, el, uh, ul);
            ff_acc(wh, wl, -fmaf(3.f, m, 9.f * uh), 0.f);  // r U'(r) = -12 rep + 6 att
        } else {
            const double2 c = sh.field.d[k];
            lj_f64_add(g, c.x, c.y, rep, att);
        }
    }
};

// One CTA per home cell; each unordered pair once: the home cell against
// itself (partners after the particle) and against the 13 cells of its half
// shell; the other 13 neighbours see the cell from their own half shells.
// partial[2c], partial[2c+1] = the cell's energy and virial sums.
template <bool F32>
__global__ void __launch_bounds__(kNbWarps * 32) k_cell_energy(const uint4 *__restrict__ cpos,
                                                               const int32_t *__restrict__ cs, int T, int64_t ncell,
                                                               uint64_t R2, float r2hi, bool wrap,
                                                               const __grid_constant__ FieldF ff,
                                                               const __grid_constant__ FieldD fd,
                                                               double *__restrict__ partial, int *__restrict__ status)
{
    constexpr int NP = 2;  // home particles a warp screens together
    extern __shared__ __align__(128) unsigned char dyn[];
    using SH = NbShared<kBufHalf>;
    constexpr int kBuf = SH::kBuf;
    SH &sh = *reinterpret_cast<SH *>(dyn);
    __shared__ double red[kNbWarps][2];
    __shared__ float2 redf[kNbWarps][2];
    __shared__ uint4 home[kPChunk];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (threadIdx.x == 0) mbar_init(&sh.bar, 1);
    nb_field<F32, false>(sh, ff, fd);
    __syncthreads();
    unsigned parity = 0;
    unsigned short *list = sh.list[w];
    for (int64_t c = blockIdx.x; c < ncell; c += gridDim.x) {
        const int h0 = cs[c], nh = cs[c + 1] - h0;
        PairDrain<F32, SH> D(sh, home, R2);
        if (nh > 0) {
            const int cx = (int)(c % T), cy = (int)((c / T) % T), cz = (int)(c / ((int64_t)T * T));
            __syncthreads();
            if (w == 0) runs_half(cs, T, cx, cy, cz, sh.runs);
            __syncthreads();
            const int total = sh.runs.end[9];
            const uint32_t cx0 = cell_centre(cx, T), cy0 = cell_centre(cy, T), cz0 = cell_centre(cz, T);
            for (int pb = 0; pb < nh; pb += kPChunk) {
                const int pn = min(kPChunk, nh - pb);
                __syncthreads();
                for (int i = threadIdx.x; i < pn; i += blockDim.x) home[i] = cpos[h0 + pb + i];
                for (int base = 0; base < total; base += kBuf) {
                    const int nst = min(kBuf, total - base);
                    if (!nb_stage(sh, cpos, base, base + nst, cx0, cy0, cz0, parity, status)) return;
                    const int rows = (nst + 31) >> 5;
                    int n = 0;
                    for (int i0 = NP * w; i0 < pn; i0 += NP * kNbWarps) {
                        float3 pf[NP];
                        uint32_t mask[NP];
#pragma unroll
                        for (int p = 0; p < NP; ++p) {
                            const uint4 P = home[min(i0 + p, pn - 1)];
                            pf[p] = make_float3(rel_f(P.x, cx0), rel_f(P.y, cy0), rel_f(P.z, cz0));
                        }
                        nb_screen<NP>(sh.fl, nst, pf, r2hi, wrap, mask);
#pragma unroll 1
                        for (int p = 0; p < NP && i0 + p < pn; ++p) {
                            uint32_t x = mask[0];
#pragma unroll
                            for (int u = 1; u < NP; ++u) x = p == u ? mask[u] : x;
                            // the home items come first: those up to the particle
                            // itself (the top bits of the lane's mask) are left out
                            const int last = pb + i0 + p - base - lane;
                            if (last >= 0) {
                                const int out = min(rows, (last >> 5) + 1);
                                x = out >= rows ? 0u : x & ((1u << (rows - out)) - 1u);
                            }
                            n = nb_drain(list, nb_append(list, n, x, rows, (i0 + p) << 10), D);
                        }
                    }
                    nb_flush(list, n, D);  // before the staged records are replaced
                }
            }
        }
        if constexpr (F32) {
            // float-float across the warp and the block, one FP64 value per sum
            const FF s = ff_warp_sum(FF{D.eh, D.el});
            const FF v = ff_warp_sum(FF{D.wh, D.wl});
            if (lane == 0) {
                redf[w][0] = make_float2(s.hi, s.lo);
                redf[w][1] = make_float2(v.hi, v.lo);
            }
            __syncthreads();
            if (threadIdx.x < 2) {
                FF sum = {0.f, 0.f};
                for (int k = 0; k < kNbWarps; ++k) sum = ff_add(sum, FF{redf[k][threadIdx.x].x, redf[k][threadIdx.x].y});
                partial[2 * c + threadIdx.x] = ff_value(sum.hi, sum.lo);
            }
        } else {
            const double e = warp_sum(D.rep - D.att), vw = warp_sum(6.0 * D.att - 12.0 * D.rep);  // r U'(r)
            if (lane == 0) {
                red[w][0] = e;
                red[w][1] = vw;
            }
            __syncthreads();
            if (threadIdx.x < 2) {
                double sum = 0.0;
                for (int k = 0; k < kNbWarps; ++k) sum += red[k][threadIdx.x];
                partial[2 * c + threadIdx.x] = sum;
            }
        }
        __syncthreads();
    }
}

// Column sums of partial[n][width] (per-cell partial sums) in a fixed order,
// in two launches: block b of k_sum_rows sums the rows [b n / B, (b + 1) n / B)
// of every column (each thread a strided share, the lanes of a warp by
// shuffles, the warps in order), and k_sum_blocks adds the B block sums of each
// column, a warp a column.  The result does not depend on timing.  Bound by
// latency: a shared-memory tree per column and one thread per column over the
// block sums took 16 + 10 us for the ten columns of a 262,144-particle
// gradient.  With the shuffles the total energy of 87,296 particles with its
// cell build takes 241 instead of 253 us, a gradient step of 6,001 particles of
// three species 708 instead of 732.
constexpr int kSumBlocks = 128;  // row blocks, at most
constexpr int kSumThreads = 256;
constexpr int kSumWidth = 2 + 2 * kMaxSpecies * kMaxSpecies;  // columns, at most
static_assert(kSumWidth <= kSumThreads, "a thread finishes a column");

__global__ void __launch_bounds__(kSumThreads) k_sum_rows(const double *__restrict__ partial, int64_t n, int width,
                                                          double *__restrict__ blk)
{
    __shared__ double sh[kSumThreads / 32][kSumWidth];
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    const int64_t r0 = n * blockIdx.x / gridDim.x, r1 = n * (blockIdx.x + 1) / gridDim.x;
#pragma unroll 2
    for (int j = 0; j < width; ++j) {
        double s = 0.0;
        for (int64_t i = r0 + t; i < r1; i += kSumThreads) s += partial[i * width + j];
        s = warp_sum(s);
        if (lane == 0) sh[w][j] = s;
    }
    __syncthreads();
    if (t < width) {
        double s = 0.0;
#pragma unroll
        for (int k = 0; k < kSumThreads / 32; ++k) s += sh[k][t];
        blk[(int64_t)blockIdx.x * width + t] = s;
    }
}

__global__ void __launch_bounds__(1024) k_sum_blocks(const double *__restrict__ blk, int nb, int width,
                                                     double *__restrict__ out)
{
    const int lane = threadIdx.x & 31;
    for (int j = threadIdx.x >> 5; j < width; j += blockDim.x >> 5) {
        double s = 0.0;
        for (int b = lane; b < nb; b += 32) s += blk[(int64_t)b * width + j];
        s = warp_sum(s);
        if (lane == 0) out[j] = s;
    }
}

// Launches the two column-sum kernels; blk holds kSumBlocks x width doubles.
static void sum_partials(gcmc_ctx *ctx, const double *partial, int64_t n, int width, double *blk, double *out)
{
    const int nb = (int)std::max<int64_t>(1, std::min<int64_t>(kSumBlocks, (n + kSumThreads - 1) / kSumThreads));
    k_sum_rows<<<nb, kSumThreads, 0, ctx->stream>>>(partial, n, width, blk);
    k_sum_blocks<<<1, std::min(32 * width, 1024), 0, ctx->stream>>>(blk, nb, width, out);
    ctx->launches += 2;
}

// ---------------------------------------------------------------------------
// Gradient.  In grid units (s^2 = sig2 / r_g^2, rep = 4 eps s^12, att = 4 eps s^6):
//   dE/dx_i = sum_j (-12 rep + 6 att) / r_g^2 * dx_g / h,
//   r U'(r) = -12 rep + 6 att,
//   dE/deps_ab (half of each ordered pair) += 2 (s^12 - s^6),
//   dE/dsigma_ab (same) += (12 rep - 6 att) / (2 sigma_ab).
// One CTA per home cell with its 27 cells staged; a warp screens two home
// particles together and sums the forces of each alone; every pair is met from
// both of its particles, so nothing is scattered.  The per-cell
// scalars go to `partial` rows of width 2 + 2 S^2: [E, virial, deps...,
// dsigma...].  order: the forces are stored at the particles' input rows (the
// last build's order), otherwise species-major.  NS: partner species in
// registers (1, 2, 4 or kMaxSpecies).
// FP32 mode: FP32 pair terms from the exact integer r^2, forces and tables
// summed in FP32 per lane and particle, everything beyond that (lanes,
// particles, energy, virial) in float-float; FP64 mode: FP64 throughout.
// ---------------------------------------------------------------------------
template <bool F32, int NS, class SH>
struct GradDrain {
    using R = typename std::conditional<F32, float, double>::type;
    const SH &sh;
    uint4 P;
    int t;
    R fx, fy, fz, aEps[NS], aSig[NS];              // of one home particle
    float eh = 0.f, el = 0.f, wh = 0.f, wl = 0.f;  // FP32 mode: of all
    double de = 0.0, dw = 0.0;                    // FP64 mode: of all
    __device__ GradDrain(const SH &s) : sh(s) {}
    __device__ __forceinline__ void start(const uint4 &p)
    {
        P = p;
        t = (int)tag_species(p.w);
        fx = fy = fz = 0;
#pragma unroll
        for (int q = 0; q < NS; ++q) aEps[q] = aSig[q] = 0;
    }
    __device__ __forceinline__ void operator()(int f)
    {
        const uint4 r = sh.raw[f];
        const int ts = (int)tag_species(r.w);
        const int k = t * kMaxSpecies + ts;
        const int ex = (int)(P.x - r.x), ey = (int)(P.y - r.y), ez = (int)(P.z - r.z);
        const unsigned long long g = (unsigned long long)((long long)ex * ex) +
                                     (unsigned long long)((long long)ey * ey) +
                                     (unsigned long long)((long long)ez * ez);
        // s^2 is bounded where s^12 is far beyond the floats (coincident pairs:
        // beyond the doubles, whatever their eps), so that s^6 is finite and
        // rep - att is +inf, not a difference of infinities.  y: about 1 / r^2.
        R c4e, s2, r2, y;
        if constexpr (F32) {
            const float4 c = sh.field.f[k];
            r2 = fmaf(__uint2float_rn((uint32_t)(g >> 32)), 4294967296.0f, __uint2float_rn((uint32_t)g));
            y = rcp_approx(r2);
            c4e = r2 == 0.f ? 1.f : c.x;
            s2 = fminf(c.z / r2, 1e11f);
        } else {
            const double2 c = sh.field.d[k];
            r2 = u64_to_f64(g);
            c4e = g == 0ull ? 1.0 : c.x;
            s2 = div_by_g(c.y, r2, g, y);
            if (g == 0ull) s2 = 1e80;
        }
        const R s6 = s2 * s2 * s2;
        const R rep = c4e * s6 * s6, att = c4e * s6;
        const R rdu = (R)(-12) * rep + (R)6 * att;  // r U'(r)
        // rdu / r^2 with one rounding: the quotient corrected by its residual, in as
        // many instructions as a reciprocal and a product take
        R coef = rdu * y;
        coef = fma(fma(-coef, r2, rdu), y, coef);
        if constexpr (F32) coef = fmaxf(coef, -3.402823466e38f);  // no force along an axis without distance
        fx += coef * (R)ex;
        fy += coef * (R)ey;
        fz += coef * (R)ez;
        if constexpr (F32) {
            ff_acc(eh, el, 0.5f * (rep - att), 0.f);
            ff_acc(wh, wl, 0.5f * rdu, 0.f);
        } else {
            de += 0.5 * (rep - att);
            dw += 0.5 * rdu;
        }
        const R ge = (R)2 * (s6 * s6 - s6);
        const R gs = (R)0.5 * ((R)12 * rep - (R)6 * att);
#pragma unroll
        for (int q = 0; q < NS; ++q) {
            if (NS == 1 || q == ts) {
                aEps[q] += ge;
                aSig[q] += gs;
            }
        }
    }
};

// A running sum over the pairs of many particles: float-float in FP32 mode,
// FP64 in FP64 mode.
__device__ __forceinline__ void sum_add(FF &a, float x) { a = ff_add_f(a, x); }
__device__ __forceinline__ void sum_add(double &a, double x) { a += x; }
__device__ __forceinline__ FF to_sum(float x) { return FF{x, 0.f}; }
__device__ __forceinline__ double to_sum(double x) { return x; }
__device__ __forceinline__ double sum_value(FF a) { return ff_value(a.hi, a.lo); }
__device__ __forceinline__ double sum_value(double a) { return a; }

template <bool F32, int NS>
__global__ void __launch_bounds__(kNbWarps * 32, 5) k_cell_grad(const uint4 *__restrict__ cpos,
                                                             const int32_t *__restrict__ cs, int T, int64_t ncell,
                                                             uint64_t R2, float r2hi, bool wrap, int S,
                                                             const __grid_constant__ FieldF ff,
                                                             const __grid_constant__ FieldD fd, double inv_h,
                                                             const int64_t *__restrict__ d_n,
                                                             const int32_t *__restrict__ order, float *__restrict__ dpos,
                                                             double *__restrict__ partial, int *__restrict__ status)
{
    constexpr int kW = 2 + 2 * NS * NS;
    using Sum = typename std::conditional<F32, FF, double>::type;
    extern __shared__ __align__(128) unsigned char dyn[];
    using SH = NbShared<kBufOrdered>;
    constexpr int kBuf = SH::kBuf;
    SH &sh = *reinterpret_cast<SH *>(dyn);
    __shared__ double red[kNbWarps][kW];
    __shared__ Sum fpart[kPChunk][3];  // per-point forces over the passes
    __shared__ uint4 home[kPChunk];
    // with up to two species the table sums of a cell stay in registers, per
    // lane, and cross the warp once per cell; with more, once per particle
    constexpr bool kRegSums = NS <= 2;
    constexpr int NR = kRegSums ? NS : 1;
    Sum sEp[NR][NR], sSg[NR][NR];
    __shared__ long long base_s[kMaxSpecies];  // first species-major row of each species
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int width = 2 + 2 * S * S;
    if (threadIdx.x == 0) {
        long long b = 0;
        for (int s = 0; s < kMaxSpecies; ++s) {
            base_s[s] = b;
            b += (s < S) ? d_n[s] : 0;
        }
        mbar_init(&sh.bar, 1);
    }
    nb_field<F32, true>(sh, ff, fd);
    __syncthreads();
    unsigned parity = 0;
    unsigned short *list = sh.list[w];
    for (int64_t c = blockIdx.x; c < ncell; c += gridDim.x) {
        const int h0 = cs[c], nh = cs[c + 1] - h0;
        for (int k = lane; k < width; k += 32) red[w][k] = 0.0;
        __syncwarp();
        GradDrain<F32, NS, SH> D(sh);
#pragma unroll
        for (int a = 0; a < NR; ++a)
#pragma unroll
            for (int q = 0; q < NR; ++q) sEp[a][q] = sSg[a][q] = Sum{};
        if (nh > 0) {
            const int cx = (int)(c % T), cy = (int)((c / T) % T), cz = (int)(c / ((int64_t)T * T));
            if (w == 0) runs27(cs, T, cx, cy, cz, sh.runs);
            __syncthreads();
            const int total = sh.runs.end[17];
            // the home cell lies in the middle row's first run
            const int own = sh.runs.end[3] + h0 - sh.runs.start[4];
            const uint32_t cx0 = cell_centre(cx, T), cy0 = cell_centre(cy, T), cz0 = cell_centre(cz, T);
            for (int pb = 0; pb < nh; pb += kPChunk) {
                const int pn = min(kPChunk, nh - pb);
                __syncthreads();
                for (int i = threadIdx.x; i < pn; i += blockDim.x) home[i] = cpos[h0 + pb + i];
                for (int base = 0; base < total; base += kBuf) {
                    const int nst = min(kBuf, total - base);
                    if (!nb_stage(sh, cpos, base, base + nst, cx0, cy0, cz0, parity, status)) return;
                    const int rows = (nst + 31) >> 5;
                    for (int i0 = 2 * w; i0 < pn; i0 += 2 * kNbWarps) {
                        uint4 P[2];
                        float3 pf[2];
                        uint32_t mask[2];
#pragma unroll
                        for (int p = 0; p < 2; ++p) {
                            P[p] = home[min(i0 + p, pn - 1)];
                            pf[p] = make_float3(rel_f(P[p].x, cx0), rel_f(P[p].y, cy0), rel_f(P[p].z, cz0));
                        }
                        nb_screen_exact<2>(sh.fl, sh.raw, nst, P, pf, R2, r2hi, wrap, mask);
#pragma unroll 1
                        for (int i = i0; i < min(i0 + 2, pn); ++i) {
                            D.start(home[i]);
                            uint32_t x = i == i0 ? mask[0] : mask[1];
                            const int self = own + pb + i - base;  // the particle's own record
                            if (self >= 0 && self < nst && (self & 31) == lane) x &= ~(1u << (rows - 1 - (self >> 5)));
                            nb_flush(list, nb_list_ordered(list, x, rows), D);
                            // lanes 0, 8, 16 get the force's x, y, z
                            Sum f[4] = {to_sum(D.fx), to_sum(D.fy), to_sum(D.fz), Sum{}};
                            const Sum force = warp_sum_many<4>(f);
                            if ((lane & 7) == 0 && lane < 24)
                                fpart[i][lane >> 3] = base > 0 ? sum_of(fpart[i][lane >> 3], force) : force;
                            if constexpr (kRegSums) {
#pragma unroll
                                for (int t = 0; t < NR; ++t) {
                                    if (NR == 1 || t == D.t) {  // the same in every lane
#pragma unroll
                                        for (int q = 0; q < NR; ++q) {
                                            sum_add(sEp[t][q], D.aEps[q]);
                                            sum_add(sSg[t][q], D.aSig[q]);
                                        }
                                    }
                                }
                            } else {
                                Sum v[2 * NS];
#pragma unroll
                                for (int q = 0; q < NS; ++q) {
                                    v[q] = to_sum(D.aEps[q]);
                                    v[NS + q] = to_sum(D.aSig[q]);
                                }
                                const Sum x = warp_sum_many<2 * NS>(v);
                                const int k = lane / (16 / NS), q = k % NS;
                                if (lane % (16 / NS) == 0 && q < S)
                                    red[w][2 + (k >= NS ? S * S : 0) + D.t * S + q] += sum_value(x);
                            }
                        }
                    }
                }
                __syncthreads();
                if (dpos) {
                    for (int i = threadIdx.x; i < pn; i += blockDim.x) {
                        const uint32_t tg = home[i].w;
                        const int64_t row = order ? order[h0 + pb + i] : base_s[tag_species(tg)] + tag_index(tg);
#pragma unroll
                        for (int a = 0; a < 3; ++a) {
                            if constexpr (F32) {
                                const FF f = fpart[i][a];
                                dpos[3 * row + a] = (isinf(f.hi) ? f.hi : f.hi + f.lo) * (float)inv_h;
                            }
                            else dpos[3 * row + a] = (float)(fpart[i][a] * inv_h);
                        }
                    }
                }
            }
        }
        {
            Sum v[2];
            if constexpr (F32) {
                v[0] = FF{D.eh, D.el};
                v[1] = FF{D.wh, D.wl};
            } else {
                v[0] = D.de;
                v[1] = D.dw;
            }
            const Sum x = warp_sum_many<2>(v);
            if ((lane & 15) == 0) red[w][lane >> 4] = sum_value(x);
        }
        if constexpr (kRegSums) {
            Sum v[2 * NR * NR];
#pragma unroll
            for (int a = 0; a < NR; ++a)
#pragma unroll
                for (int q = 0; q < NR; ++q) {
                    v[a * NR + q] = sEp[a][q];
                    v[NR * NR + a * NR + q] = sSg[a][q];
                }
            const Sum x = warp_sum_many<2 * NR * NR>(v);  // NR == S
            constexpr int kLanes = 16 / (NR * NR);
            if (lane % kLanes == 0) red[w][2 + lane / kLanes] = sum_value(x);
        }
        __syncthreads();
        for (int j = threadIdx.x; j < width; j += blockDim.x) {
            double s = 0.0;
            for (int k = 0; k < kNbWarps; ++k) s += red[k][j];
            partial[c * width + j] = s;
        }
        __syncthreads();
    }
}

static unsigned blocks_for(gcmc_ctx *ctx, int64_t work, int per_block)
{
    int64_t b = (work + per_block - 1) / per_block;
    const int64_t cap = (int64_t)ctx->num_sms * 16;
    if (b > cap) b = cap;
    return (unsigned)(b < 1 ? 1 : b);
}

// The screen's bound above the grid cutoff R2: FP32 squared distances above
// r2hi are outside; below it the exact integer test decides.  The FP32
// separations carry a relative error below 1e-6 of the cell edge (coordinates
// relative to the cell centre), far inside the margin.
// wrap: the cells are narrower than rc (2 rc <= L < 3 rc), so the FP32
// separations need their own periodic wrap.
static void screen_bound(const gcmc_ctx *ctx, float &r2hi, bool &wrap)
{
    r2hi = (float)((double)ctx->R2 * (1.0 + 1e-5));
    wrap = (double)ctx->T * ctx->rc > ctx->L;
}

// Grid size of a neighbourhood kernel: one CTA per cell, at most 48 per SM, five
// to ten times what is resident (nine CTAs of k_trial_energy and k_cell_energy,
// five of k_cell_grad).
static unsigned nb_blocks(const gcmc_ctx *ctx, int64_t cells)
{
    const int64_t cap = (int64_t)ctx->num_sms * 6 * 8;
    return (unsigned)std::max<int64_t>(1, std::min<int64_t>(cells, cap));
}

// The neighbourhood kernels take more than 48 KB of shared memory.
template <typename K>
static gcmc_status nb_smem(gcmc_ctx *ctx, K kern, size_t bytes)
{
    const cudaError_t e =
        cudaFuncSetAttribute((const void *)kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e != cudaSuccess) return cuda_fail(ctx, e, "cudaFuncSetAttribute (neighbourhood kernel)");
    return GCMC_OK;
}

gcmc_status trial_energy(gcmc_ctx *ctx, const double *pos, const int32_t *species, const int64_t *exclude,
                         int64_t m, double *out, double *out_abs)
{
    gcmc_status st = make_compact(ctx);
    if (st != GCMC_OK) return st;
    if (m <= 0) return GCMC_OK;
    if (m > (int64_t)INT32_MAX) return fail(ctx, GCMC_ERR_INVALID_ARG, "gcmc_trial_energy: too many points");
    cudaStream_t s = ctx->stream;
    float r2hi;
    bool wrap;
    screen_bound(ctx, r2hi, wrap);
    if (m <= direct_points(ctx, out_abs != nullptr)) {
        st = ensure_pinned(ctx, kPinnedBytes);
        if (st != GCMC_OK) return st;
        // the status word lies in pinned host memory, written by the kernel
        volatile int *status = (volatile int *)((double *)ctx->h_pinned + 13);
        *status = 0;
        auto launch = [&](auto kern, int warps) {
            kern<<<(unsigned)m, warps * 32, 0, s>>>(pos, species, exclude, ctx->q, ctx->T, ctx->S, ctx->cpos,
                                                    ctx->cell_start, ctx->R2, r2hi, ctx->ff, ctx->fd, out, out_abs,
                                                    status);
        };
        if (ctx->precision == GCMC_FP64) launch(k_trial_direct<false, false>, kDirectWarps);
        else if (out_abs) launch(k_trial_direct<true, true>, 1);
        else launch(k_trial_direct<true, false>, kDirectWarps);
        ctx->launches += 1;
        GCMC_CUDA(ctx, cudaGetLastError());
        GCMC_CUDA(ctx, cudaStreamSynchronize(s));
        if (*status & kStatusBadInput)
            return fail(ctx, GCMC_ERR_INVALID_ARG, "gcmc_trial_energy: species out of range or coordinate not finite");
        return GCMC_OK;
    }
    // scratch: binned points, unbinned points, cell ids, per-cell counts and
    // starts, fill counters, scan partials
    const int64_t ncell = ctx->ncell;
    const int64_t nbs = (ncell + 1023) / 1024 + 1;
    auto al = [](size_t b) { return (b + 255) / 256 * 256; };
    const size_t b_pts = al(m * sizeof(TrialPt)), b_tmp = b_pts, b_cid = al(m * sizeof(int32_t)),
                 b_cnt = al(ncell * sizeof(int32_t)), b_ps = al((ncell + 1) * sizeof(int32_t)),
                 b_part = al(nbs * sizeof(int32_t) + 64);
    st = ensure_scratch(ctx, b_pts + b_tmp + b_cid + 2 * b_cnt + b_ps + b_part);
    if (st != GCMC_OK) return st;
    char *p = (char *)ctx->scratch;
    TrialPt *pts = (TrialPt *)p;
    TrialPt *tmp = (TrialPt *)(p += b_pts);
    int32_t *cid = (int32_t *)(p += b_tmp);
    int32_t *cnt = (int32_t *)(p += b_cid);
    int32_t *fill = (int32_t *)(p += b_cnt);
    int32_t *ps = (int32_t *)(p += b_cnt);
    int32_t *part = (int32_t *)(p += b_ps);
    int *vmax = part + nbs;
    GCMC_CUDA(ctx, cudaMemsetAsync(ctx->d_status, 0, sizeof(int), s));
    GCMC_CUDA(ctx, cudaMemsetAsync(cnt, 0, 2 * b_cnt, s));  // counts and fill counters
    const unsigned gb = blocks_for(ctx, m, 256);
    k_trial_bin<<<gb, 256, 0, s>>>(pos, species, exclude, m, ctx->q, ctx->T, ctx->S, tmp, cid, cnt, out, out_abs,
                                   ctx->d_status);
    st = exclusive_scan(ctx, cnt, ncell, ps, part, vmax);
    if (st != GCMC_OK) return st;
    k_trial_place<<<gb, 256, 0, s>>>(tmp, cid, m, ps, fill, pts);
    const unsigned nb = nb_blocks(ctx, ncell);
    auto launch = [&](auto kern, int warps, size_t smem) {
        gcmc_status r = nb_smem(ctx, kern, smem);
        if (r == GCMC_OK)
            kern<<<nb, warps * 32, smem, s>>>(pts, ps, ctx->cpos, ctx->cell_start, ctx->T, ncell, ctx->R2, r2hi, wrap,
                                              ctx->ff, ctx->fd, out, out_abs, ctx->d_status);
        return r;
    };
    if (ctx->precision == GCMC_FP32)
        st = out_abs ? launch(k_trial_scaled, kScaledWarps, sizeof(ScaledShared))
                     : launch(k_trial_energy<true, false>, kNbWarps, sizeof(NbShared<kBufFull>));
    else
        st = out_abs ? launch(k_trial_energy<false, true>, kNbWarps, sizeof(NbShared<kBufFull>))
                     : launch(k_trial_energy<false, false>, kNbWarps, sizeof(NbShared<kBufFull>));
    if (st != GCMC_OK) return st;
    ctx->launches += 3;
    GCMC_CUDA(ctx, cudaGetLastError());
    int bits = 0;
    st = read_status(ctx, &bits);
    if (st != GCMC_OK) return st;
    if (bits & kStatusTimeout)
        return fail(ctx, GCMC_ERR_TIMEOUT, "gcmc_trial_energy: a bulk copy did not complete within the wait limit");
    if (bits & kStatusBadInput)
        return fail(ctx, GCMC_ERR_INVALID_ARG, "gcmc_trial_energy: species out of range or coordinate not finite");
    return GCMC_OK;
}

gcmc_status total_energy_begin(gcmc_ctx *ctx, bool virial_only)
{
    gcmc_status st = make_compact(ctx);
    if (st != GCMC_OK) return st;
    st = ensure_red(ctx, 2 * (size_t)ctx->ncell + 8 + 2 * kSumBlocks);
    if (st != GCMC_OK) return st;
    st = ensure_pinned(ctx, kPinnedBytes);
    if (st != GCMC_OK) return st;
    float r2hi;
    bool wrap;
    screen_bound(ctx, r2hi, wrap);
    const unsigned nb = nb_blocks(ctx, ctx->ncell);
    GCMC_CUDA(ctx, cudaMemsetAsync(ctx->d_status, 0, sizeof(int), ctx->stream));
    if (ctx->precision == GCMC_FP32) {
        st = nb_smem(ctx, k_cell_energy<true>, sizeof(NbShared<kBufHalf>));
        if (st != GCMC_OK) return st;
        k_cell_energy<true><<<nb, kNbWarps * 32, sizeof(NbShared<kBufHalf>), ctx->stream>>>(
            ctx->cpos, ctx->cell_start, ctx->T, ctx->ncell, ctx->R2, r2hi, wrap, ctx->ff, ctx->fd, ctx->d_red,
            ctx->d_status);
    } else {
        st = nb_smem(ctx, k_cell_energy<false>, sizeof(NbShared<kBufHalf>));
        if (st != GCMC_OK) return st;
        k_cell_energy<false><<<nb, kNbWarps * 32, sizeof(NbShared<kBufHalf>), ctx->stream>>>(
            ctx->cpos, ctx->cell_start, ctx->T, ctx->ncell, ctx->R2, r2hi, wrap, ctx->ff, ctx->fd, ctx->d_red,
            ctx->d_status);
    }
    sum_partials(ctx, ctx->d_red, ctx->ncell, 2, ctx->d_red + 2 * ctx->ncell + 8, ctx->d_red + 2 * ctx->ncell);
    ctx->launches += 1;
    GCMC_CUDA(ctx, cudaGetLastError());
    double *hp = (double *)ctx->h_pinned;
    const double *dsum = ctx->d_red + 2 * ctx->ncell;
    GCMC_CUDA(ctx, cudaMemcpyAsync(hp + 10, dsum, 2 * sizeof(double), cudaMemcpyDeviceToHost, ctx->stream));
    GCMC_CUDA(ctx, cudaMemcpyAsync(hp + 12, ctx->d_status, sizeof(int), cudaMemcpyDeviceToHost, ctx->stream));
    // the running values on the device come from the device (no second host round trip)
    if (virial_only)
        GCMC_CUDA(ctx, cudaMemcpyAsync(ctx->d_energy + 1, dsum + 1, sizeof(double), cudaMemcpyDeviceToDevice,
                                       ctx->stream));
    else
        GCMC_CUDA(ctx, cudaMemcpyAsync(ctx->d_energy, dsum, 2 * sizeof(double), cudaMemcpyDeviceToDevice,
                                       ctx->stream));
    return GCMC_OK;
}

gcmc_status total_energy_finish(gcmc_ctx *ctx, double *energy, bool virial_only)
{
    const double *hp = (const double *)ctx->h_pinned;
    int bits = 0;
    memcpy(&bits, hp + 12, sizeof(int));
    if (bits & kStatusTimeout)
        return fail(ctx, GCMC_ERR_TIMEOUT, "gcmc_total_energy: a bulk copy did not complete within the wait limit");
    const double e = hp[10];
    ctx->virial = hp[11];
    ctx->virial_valid = true;
    if (!virial_only) {
        ctx->energy = e;
        ctx->energy_valid = true;
    }
    if (energy) *energy = e;
    return GCMC_OK;
}

gcmc_status total_energy(gcmc_ctx *ctx, double *energy, bool virial_only)
{
    gcmc_status st = total_energy_begin(ctx, virial_only);
    if (st != GCMC_OK) return st;
    GCMC_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
    return total_energy_finish(ctx, energy, virial_only);
}

gcmc_status energy_grad_begin(gcmc_ctx *ctx, float *dpos, bool input_order)
{
    gcmc_status st = make_compact(ctx);
    if (st != GCMC_OK) return st;
    const int S = ctx->S;
    const int width = 2 + 2 * S * S;
    st = ensure_red(ctx, (size_t)ctx->ncell * width + width + (size_t)kSumBlocks * width);
    if (st != GCMC_OK) return st;
    st = ensure_pinned(ctx, kPinnedBytes);
    if (st != GCMC_OK) return st;
    float r2hi;
    bool wrap;
    screen_bound(ctx, r2hi, wrap);
    const unsigned nb = nb_blocks(ctx, ctx->ncell);
    double *part = ctx->d_red;
    double *res = ctx->d_red + (size_t)ctx->ncell * width;
    FieldF ff = ctx->ff;  // dE/deps of a pair with eps = 0 needs its sigma
    for (int k = 0; k < kMaxSpecies * kMaxSpecies; ++k) set_sig2(ff, k, ctx->fd.sig2[k]);
    GCMC_CUDA(ctx, cudaMemsetAsync(ctx->d_status, 0, sizeof(int), ctx->stream));
#define GCMC_GRAD(F, NSP)                                                                                     \
    do {                                                                                                      \
        st = nb_smem(ctx, k_cell_grad<F, NSP>, sizeof(NbShared<kBufOrdered>));                                \
        if (st != GCMC_OK) return st;                                                                         \
        k_cell_grad<F, NSP><<<nb, kNbWarps * 32, sizeof(NbShared<kBufOrdered>), ctx->stream>>>(               \
            ctx->cpos, ctx->cell_start, ctx->T, ctx->ncell, ctx->R2, r2hi, wrap, S, ff, ctx->fd,               \
            1.0 / ctx->h, ctx->d_n, input_order ? ctx->order : nullptr, dpos, part, ctx->d_status);           \
    } while (0)
    if (ctx->precision == GCMC_FP32) {
        if (S == 1) GCMC_GRAD(true, 1);
        else if (S == 2) GCMC_GRAD(true, 2);
        else if (S <= 4) GCMC_GRAD(true, 4);
        else GCMC_GRAD(true, kMaxSpecies);
    } else {
        if (S == 1) GCMC_GRAD(false, 1);
        else if (S == 2) GCMC_GRAD(false, 2);
        else if (S <= 4) GCMC_GRAD(false, 4);
        else GCMC_GRAD(false, kMaxSpecies);
    }
#undef GCMC_GRAD
    sum_partials(ctx, part, ctx->ncell, width, res + width, res);
    ctx->launches += 1;
    GCMC_CUDA(ctx, cudaGetLastError());
    double *hp = (double *)ctx->h_pinned + 16;
    GCMC_CUDA(ctx, cudaMemcpyAsync(hp, res, width * sizeof(double), cudaMemcpyDeviceToHost, ctx->stream));
    GCMC_CUDA(ctx, cudaMemcpyAsync(hp + width, ctx->d_status, sizeof(int), cudaMemcpyDeviceToHost, ctx->stream));
    return GCMC_OK;
}

gcmc_status energy_grad_finish(gcmc_ctx *ctx, double *deps, double *dsigma, double *energy, double *virial)
{
    const int S = ctx->S;
    const int width = 2 + 2 * S * S;
    const double *h = (const double *)ctx->h_pinned + 16;
    int bits = 0;
    memcpy(&bits, h + width, sizeof(int));
    if (bits & kStatusTimeout)
        return fail(ctx, GCMC_ERR_TIMEOUT, "gcmc_energy_grad: a bulk copy did not complete within the wait limit");
    if (energy) *energy = h[0];
    if (virial) *virial = h[1];
    for (int a = 0; a < S; ++a)
        for (int b = 0; b < S; ++b) {
            if (deps) deps[a * S + b] = h[2 + a * S + b];
            if (dsigma) dsigma[a * S + b] = h[2 + S * S + a * S + b] / ctx->sigma[a * kMaxSpecies + b];
        }
    return GCMC_OK;
}

gcmc_status energy_grad(gcmc_ctx *ctx, float *dpos, double *deps, double *dsigma, double *energy,
                        double *virial, bool input_order)
{
    gcmc_status st = energy_grad_begin(ctx, dpos, input_order);
    if (st != GCMC_OK) return st;
    GCMC_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
    return energy_grad_finish(ctx, deps, dsigma, energy, virial);
}

// ---- the configuration as real coordinates -----------------------------
__global__ void k_export(const uint4 *__restrict__ pos_by_id, const int64_t *__restrict__ d_n, int S, int64_t maxN,
                         double h, double *__restrict__ pos, int32_t *__restrict__ species)
{
    __shared__ long long base[kMaxSpecies + 1];
    if (threadIdx.x == 0) {
        long long b = 0;
        for (int s = 0; s < S; ++s) {
            base[s] = b;
            b += d_n[s];
        }
        base[S] = b;
    }
    __syncthreads();
    const long long N = base[S];
    for (long long r = (long long)blockIdx.x * blockDim.x + threadIdx.x; r < N;
         r += (long long)gridDim.x * blockDim.x) {
        int s = 0;
        while (r >= base[s + 1]) ++s;
        const uint4 v = pos_by_id[(long long)s * maxN + (r - base[s])];
        // the centre of the grid cell quantises back to the same grid point
        pos[3 * r + 0] = ((double)v.x + 0.5) * h;
        pos[3 * r + 1] = ((double)v.y + 0.5) * h;
        pos[3 * r + 2] = ((double)v.z + 0.5) * h;
        species[r] = s;
    }
}

gcmc_status export_positions(gcmc_ctx *ctx, double *pos, int32_t *species)
{
    int64_t N = 0;
    for (int s = 0; s < ctx->S; ++s) N += ctx->n_host[s];
    if (N == 0) return GCMC_OK;
    k_export<<<blocks_for(ctx, N, 256), 256, 0, ctx->stream>>>(ctx->pos_by_id, ctx->d_n, ctx->S, ctx->maxN, ctx->h,
                                                              pos, species);
    ctx->launches += 1;
    GCMC_CUDA(ctx, cudaGetLastError());
    return GCMC_OK;
}


// ---------------------------------------------------------------------------
// Allocation-free full-system energy.  Some callers may not allocate device
// memory at the point where they need the energy: code under a fixed
// device-memory budget owned by another allocator, or a real-time loop that
// must not enter the driver's allocator (which can block or fail when memory
// runs short).  This variant reads the padded cell layout that the chain keeps
// current (so no compact copy has to be built or grown) and keeps its
// per-cell partial sums in one file-scope device array instead of the
// context's scratch.  The array is shared by every call on a device: two
// calls whose kernels overlap on the GPU race on it.
// ---------------------------------------------------------------------------
constexpr int kStage = 2048;  // staged partners per pass (32 KB)
constexpr int64_t kStaticMaxCells = GCMC_NOALLOC_MAX_CELLS;  // T <= 50; 1 MiB of partials
static __device__ __align__(256) double g_static_partials[kStaticMaxCells];

constexpr int kMaxDevicesStatic = 64;
static std::mutex g_static_mu;
static double *g_static_ptr[kMaxDevicesStatic] = {};

// Full-system energy on the padded cell-major layout: one CTA per home cell
// (grid-stride), the 27 neighbour cells staged in shared memory, partial[c]
// written for every cell (nothing has to start at zero).
template <bool F32>
__global__ void __launch_bounds__(256) k_cell_energy_padded(const uint4 *__restrict__ cell_pos,
                                                            const int32_t *__restrict__ cell_count, int cap, int T,
                                                            int64_t ncell, uint64_t R2, const FieldF ff,
                                                            const FieldD fd, double *__restrict__ partial)
{
    __shared__ uint4 stage[kStage];
    __shared__ int nb_cell[27], nb_end[27];
    __shared__ double red[8];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (int64_t c = blockIdx.x; c < ncell; c += gridDim.x) {
        const int cx = (int)(c % T), cy = (int)((c / T) % T), cz = (int)(c / ((int64_t)T * T));
        if (w == 0) {
            int cell = 0, n = 0;
            if (lane < 27) {
                const int dx = lane % 3 - 1, dy = (lane / 3) % 3 - 1, dz = lane / 9 - 1;
                const int x = (cx + dx + T) % T, y = (cy + dy + T) % T, z = (cz + dz + T) % T;
                cell = (z * T + y) * T + x;
                n = cell_count[cell];
            }
            const int inc = warp_inclusive_scan(n);
            if (lane < 27) {
                nb_cell[lane] = cell;
                nb_end[lane] = inc;
            }
        }
        __syncthreads();
        const int total = nb_end[26];
        const int nh = cell_count[c];
        const uint4 *home = cell_pos + c * (int64_t)cap;
        Acc<F32> acc;
        for (int base = 0; base < total; base += kStage) {
            const int nst = min(kStage, total - base);
            for (int f = threadIdx.x; f < nst; f += blockDim.x) {
                const int g = base + f;
                int r = 0;
                while (g >= nb_end[r]) ++r;
                stage[f] = cell_pos[(int64_t)nb_cell[r] * cap + (g - (r ? nb_end[r - 1] : 0))];
            }
            __syncthreads();
            for (int i = w; i < nh; i += 8) {
                const uint4 p = home[i];
                const int t = (int)tag_species(p.w);
                for (int f = lane; f < nst; f += 32) pair_acc<F32>(p, stage[f], p.w, R2, t, ff, fd, acc);
            }
            __syncthreads();
        }
        const double e = warp_sum(acc.ev());
        if (lane == 0) red[w] = e;
        __syncthreads();
        if (threadIdx.x == 0) {
            double sum = 0.0;
            for (int k = 0; k < 8; ++k) sum += red[k];
            partial[c] = sum;
        }
        __syncthreads();
    }
}

// out[0] = 1/2 * sum of partial[0 .. n) (one block, fixed order): every pair
// was visited from both of its particles.
__global__ void __launch_bounds__(1024) k_half_sum(const double *__restrict__ partial, int64_t n,
                                                   double *__restrict__ out)
{
    __shared__ double sh[1024];
    double sum = 0.0;
    for (int64_t i = threadIdx.x; i < n; i += blockDim.x) sum += partial[i];
    sh[threadIdx.x] = sum;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) out[0] = 0.5 * sh[0];
}

// Device address of the static partials on the current device, looked up
// once per device (cudaGetSymbolAddress allocates nothing).
static gcmc_status static_partials(gcmc_ctx *ctx, int device, double **out)
{
    if (device < 0 || device >= kMaxDevicesStatic)
        return fail(ctx, GCMC_ERR_INVALID_ARG, "gcmc_total_energy_noalloc: device ordinal out of range");
    std::lock_guard<std::mutex> lock(g_static_mu);
    if (!g_static_ptr[device]) {
        void *p = nullptr;
        const cudaError_t e = cudaGetSymbolAddress(&p, g_static_partials);
        if (e != cudaSuccess) return cuda_fail(ctx, e, "cudaGetSymbolAddress(g_static_partials)");
        g_static_ptr[device] = (double *)p;
    }
    *out = g_static_ptr[device];
    return GCMC_OK;
}

static gcmc_status total_energy_noalloc_on_device(gcmc_ctx *ctx, double *energy_dev)
{
    if (ctx->ncell > kStaticMaxCells)
        return fail(ctx, GCMC_ERR_INVALID_ARG,
                    "gcmc_total_energy_noalloc: " + std::to_string(ctx->ncell) +
                        " cells exceed the static scratch of " + std::to_string(kStaticMaxCells) + " cells");
    cudaPointerAttributes attr{};
    GCMC_CUDA(ctx, cudaPointerGetAttributes(&attr, energy_dev));
    if (attr.type != cudaMemoryTypeDevice && attr.type != cudaMemoryTypeManaged)
        return fail(ctx, GCMC_ERR_INVALID_ARG, "gcmc_total_energy_noalloc: energy must be device memory");
    if (attr.type == cudaMemoryTypeDevice && attr.device != ctx->device)
        return fail(ctx, GCMC_ERR_INVALID_ARG,
                    "gcmc_total_energy_noalloc: energy is memory of device " + std::to_string(attr.device) +
                        ", the context's device is " + std::to_string(ctx->device));
    double *partial = nullptr;
    gcmc_status st = static_partials(ctx, ctx->device, &partial);
    if (st != GCMC_OK) return st;
    const unsigned nb = (unsigned)std::min<int64_t>(ctx->ncell, (int64_t)ctx->num_sms * 8);
    if (ctx->precision == GCMC_FP32)
        k_cell_energy_padded<true><<<nb, 256, 0, ctx->stream>>>(ctx->cell_pos, ctx->cell_count, ctx->cap, ctx->T,
                                                               ctx->ncell, ctx->R2, ctx->ff, ctx->fd, partial);
    else
        k_cell_energy_padded<false><<<nb, 256, 0, ctx->stream>>>(ctx->cell_pos, ctx->cell_count, ctx->cap, ctx->T,
                                                                ctx->ncell, ctx->R2, ctx->ff, ctx->fd, partial);
    k_half_sum<<<1, 1024, 0, ctx->stream>>>(partial, ctx->ncell, energy_dev);
    ctx->launches += 2;
    GCMC_CUDA(ctx, cudaGetLastError());
    return GCMC_OK;
}

gcmc_status total_energy_noalloc(gcmc_ctx *ctx, double *energy_dev)
{
    int prev = 0;
    GCMC_CUDA(ctx, cudaGetDevice(&prev));
    if (prev != ctx->device) GCMC_CUDA(ctx, cudaSetDevice(ctx->device));
    const gcmc_status st = total_energy_noalloc_on_device(ctx, energy_dev);
    if (prev != ctx->device) {
        const cudaError_t e = cudaSetDevice(prev);
        if (st == GCMC_OK && e != cudaSuccess) return cuda_fail(ctx, e, "cudaSetDevice (restore)");
    }
    return st;
}

}  // namespace gcmc
