// mover.cuh -- the fused per-particle time step ("particle mover" of the paper,
// Section 2 and Listing 7) for one precision T:
//
//   gather   a = A[j] + f (A[j+1] - A[j]), one fused multiply-add on the node pair
//            (A_j, A_{j+1} - A_j)                   (Listing 7, moveb())
//   push     u += a, or the Boris rotation when B != 0 (Boris 1970)
//   move     f += u_x; the integer part moves the particle across cells
//   wall     periodic wrap inline; a particle that leaves through an absorbing or
//            source wall is queued for the event kernel and leaves the store
//   MCC      null collision: the collision clock in the cell word says when the
//            particle's next candidate step is; at a test step Philox(id, step,
//            COLLIDE) word 0 sets the clock; a candidate is queued for the event
//            kernel, which selects the process and does the kinematics
//   deposit  cloud-in-cell in fixed point: node j gets S - Q, node j+1 gets
//            Q = rint(f S), so every particle adds exactly S (S = 2^24 FP32,
//            2^48 FP64); reduced per node across the warp in registers, then one
//            64-bit reduction per node and warp into HBM.
//
// Work decomposition: a tile is 32 quads of four consecutive particles of one
// segment (instance, species), owned by one warp; each lane loads its quad with
// 128-bit accesses.  The particle id is not streamed: it is read only at clock test
// steps (once per 127 steps per particle) and by the event kernel.  Warps walk the
// tiles of all segments independently, with no block-level barrier, so an SM keeps
// the loads of many tiles in flight.  The common path has no calls: the rare events
// (collision candidates, wall hits) go to a queue that the event kernel
// (events.cuh) works through after the mover, so the common path keeps its whole
// state in registers.  Velocity changes do not move a particle, so a candidate is
// deposited here; a wall particle is deposited by the event kernel if it is
// re-injected.
#pragma once
#include <algorithm>
#include <climits>

#include "common.cuh"

namespace bitpic {

// Resident warps per SM the FP32 mover is built for.  With every warp's next tile on its
// way through shared memory, 32 warps keep HBM busy, and more of them only spread the
// accesses over more DRAM pages at a time (196.6 M particles: 0.646 ms at 32, 0.651 at 48
// in 256-thread blocks; 0.69 against 0.76 on a persistent grid).
#ifndef BITPIC_MOVE_MIN_WARPS
#define BITPIC_MOVE_MIN_WARPS 32
#endif
constexpr int kMoveMinWarps = BITPIC_MOVE_MIN_WARPS;
#ifndef BITPIC_MOVE_MIN_WARPS_FULL
#define BITPIC_MOVE_MIN_WARPS_FULL 32
#endif
// the FP32 variant for the steps on which every clock without a candidate tests (FULL):
// four draws in flight per lane want registers more than warps
constexpr int kMoveMinWarpsFull = BITPIC_MOVE_MIN_WARPS_FULL;
#ifndef BITPIC_MOVE_MIN_WARPS64
#define BITPIC_MOVE_MIN_WARPS64 24
#endif
// The same for the FP64 form: registers before warps (80 instead of 64 end its spills; the
// paper's case 246 -> 236 us a step), but two blocks of 512 threads (24 warps would be
// one: 196.6 M particles 1.61 against 1.81 ms a step).
constexpr int kMoveMinWarps64 = BITPIC_MOVE_MIN_WARPS64;
#ifndef BITPIC_MOVE_MIN_WARPS_MAG
#define BITPIC_MOVE_MIN_WARPS_MAG 32
#endif
constexpr int kMoveMinWarpsMag = BITPIC_MOVE_MIN_WARPS_MAG;  // the Boris (3V) variant, FP32
#ifndef BITPIC_MOVE_MIN_WARPS64_MAG
#define BITPIC_MOVE_MIN_WARPS64_MAG 24
#endif
constexpr int kMoveMinWarps64Mag = BITPIC_MOVE_MIN_WARPS64_MAG;  // the Boris variant, FP64

struct MoveArgs {
    int32_t* cell;
    void* off;
    void* ux;
    void* uy;
    void* uz;
    uint32_t* id;
    const SegParams* seg;
    const InstParams* inst;
    int nseg;
    const int64_t* tile_start;          // nseg+1 prefix of tiles
    const int64_t* seg_nmove;           // slots of each segment moved this step
    int chunk;                          // consecutive tiles a warp of k_move takes at a time, or
                                        // kSpread: spread_chunk's
                                        // (k_move_sort: rounds of a block's tiles)
    unsigned long long* seg_n;          // slots in use (appends for created particles)
    unsigned long long* seg_live;       // live particles
    const void* accel;                  // T pairs (A_j, A_{j+1} - A_j), segment node arrays
    unsigned long long* dep;            // fixed-point deposit, segment node arrays
    unsigned long long* wall_count;     // [nseg][2]
    double* wall_energy;                // [nseg][2]
    unsigned long long* collisions;     // [ninst][kMaxProc]
    Event* events;
    unsigned long long* ev_count;       // [ninst]
    unsigned* err;
    int64_t* step;                      // [1] steps completed, [0] the step under way
    uint64_t* rare;                     // queue of rare events of this step (rare_pack)
    // [0]: entries queued this step, [1]: entries of vlist, each emptied by the kernel that
    // works through it, whose finished blocks [2] and [3] count
    unsigned long long* rare_count;
    int64_t rare_cap;                   // queue entries
    // neutral particle targets (segment node arrays of the target segments): live
    // targets per cell as of the start of the step, ionization requests of the step,
    // and the sort histogram, which holds each cell's end position after a sort
    unsigned* tcount;
    unsigned* treq;
    // the target nodes with ionization requests this step (each once), for k_victims
    int64_t* vlist;
    int64_t vcap;
    const unsigned* hist;
    // the sort folded into the time step: the step before a sort counts each cell's
    // particles at the end of the step into `hist_out` (null: no counting); the sort
    // step reserves each particle's slot in the other store copy from `cursor` (the
    // scanned counts, by the cell at the start of the step) and writes it there
    unsigned* hist_out;
    unsigned* cursor;
    int32_t* dcell;
    void* doff;
    void* dux;
    void* duy;
    void* duz;
    uint32_t* did;
    // y coordinates of 2-D species (null when no species has one): this store copy's,
    // and the sort destination's
    void* yp;
    void* dyp;
};

// Variants of the mover for a time step, see k_move.
enum class MoveMode { kDirect, kAhead, kFull };

template <typename T> struct Prec;
template <> struct Prec<float> {
    using Q = uint32_t;  // fixed-point charge of one particle (< 2^25)
    using T2 = float2;
    static __device__ __forceinline__ float fma_(float a, float b, float c) { return __fmaf_rn(a, b, c); }
    // Boris vectors t, s of the segment in this precision
    static __device__ __forceinline__ float bt(const SegParams& P, int k) { return P.tf[k]; }
    static __device__ __forceinline__ float bs(const SegParams& P, int k) { return P.sf[k]; }
    static constexpr int min_warps = kMoveMinWarps;
    static constexpr int min_warps_512 = kMoveMinWarps;
    static constexpr int min_warps_mag = kMoveMinWarpsMag;
    static constexpr int min_warps_full = kMoveMinWarpsFull;
    static __device__ __forceinline__ uint64_t qright(float f)
    {
        return (uint64_t)__float2uint_rn(f * 16777216.0f);
    }
    static constexpr uint64_t S = 1ull << 24;
    // (w + 1/2) 2^-32 rounded to float, kept below 1
    static __device__ __forceinline__ float uni(uint32_t w)
    {
        return fminf(__fmaf_rn(__uint2float_rn(w), 0x1p-32f, 0x1p-33f), 0x1.fffffep-1f);
    }
    static __device__ __forceinline__ void sincos2pi(float u, float* s, float* c)
    {
        sincospif(2.0f * u, s, c);
    }
    static __device__ __forceinline__ float sqrt_(float x) { return sqrtf(x); }
    static __device__ __forceinline__ float log_(float x) { return logf(x); }
    static __device__ __forceinline__ float floor_(float x) { return floorf(x); }
    static __device__ __forceinline__ bool finite(float x) { return isfinite(x); }
    // move (Listing 7: x += nstep*vx with x the in-cell offset): f' = f + u, the integer
    // part of f' moves the particle across cells; an f' - floor(f') that rounds up to 1
    // (f' a tiny negative number) is renormalised to the next cell
    static __device__ __forceinline__ void move(float& f, float u, int& j)
    {
        const float xn = f + u;
        const float fl = floorf(xn);
        f = xn - fl;
        j += (int)fl;
        if (f >= 1.0f) {
            f = 0.0f;
            j += 1;
        }
    }
    // The same without the renormalisation: dj cells crossed; true when f' rounded up to
    // 1 or the velocity is not finite (f' is then a NaN), which move() handles.
    static __device__ __forceinline__ bool move_fast(float& f, float u, int& dj)
    {
        const float xn = f + u;
        const float fl = floorf(xn);
        f = xn - fl;
        dj = (int)fl;
        return !(f < 1.0f);
    }
};
template <> struct Prec<double> {
    using Q = uint64_t;  // fixed-point charge of one particle (< 2^49)
    using T2 = double2;
    static __device__ __forceinline__ double fma_(double a, double b, double c) { return __fma_rn(a, b, c); }
    static __device__ __forceinline__ double bt(const SegParams& P, int k) { return P.t[k]; }
    static __device__ __forceinline__ double bs(const SegParams& P, int k) { return P.s[k]; }
    static constexpr int min_warps = kMoveMinWarps64;
    static constexpr int min_warps_512 = 32;
    static constexpr int min_warps_mag = kMoveMinWarps64Mag;
    static constexpr int min_warps_full = kMoveMinWarps64Mag;
    // rint(f 2^48) for f in [0, 1), ties to even, from the bits: f = m 2^(e-1075), so
    // f 2^48 = m / 2^(1027-e) rounded to nearest even (integer ALU only).
    static __device__ __forceinline__ uint64_t qright(double f)
    {
        const unsigned long long b = (unsigned long long)__double_as_longlong(f);
        const int e = (int)(b >> 52);
        const int sh = 1027 - e;
        if (b == 0ull || sh >= 64) return 0ull;
        const unsigned long long m = (b & 0xFFFFFFFFFFFFFull) | 0x10000000000000ull;
        unsigned long long q = m >> sh;
        const unsigned long long rem = m & ((1ull << sh) - 1ull), half = 1ull << (sh - 1);
        if (rem > half || (rem == half && (q & 1ull))) q += 1ull;
        return q;
    }
    static constexpr uint64_t S = 1ull << 48;
    static __device__ __forceinline__ double uni(uint32_t w) { return ((double)w + 0.5) * 0x1p-32; }
    static __device__ __forceinline__ void sincos2pi(double u, double* s, double* c)
    {
        sincos(6.283185307179586476925286766559 * u, s, c);
    }
    static __device__ __forceinline__ double sqrt_(double x) { return sqrt(x); }
    static __device__ __forceinline__ double log_(double x) { return log(x); }
    static __device__ __forceinline__ double floor_(double x) { return floor(x); }
    // Finiteness from the exponent bits of the high word (integer ALU; the FP64 pipe
    // is this form's limit, and a test on the whole 64-bit pattern may be turned back
    // into a floating-point comparison by the compiler).
    static __device__ __forceinline__ bool finite(double x)
    {
        return (__double2hiint(x) & 0x7FF00000) != 0x7FF00000;
    }
    // The same move as the float form with the same rounding: f' - floor(f') and the
    // truncation.  For the common -1 < f' < 2 the floor is read from the bits, and only
    // a particle that crossed a cell edge needs f' - floor(f'): the one IEEE addition
    // f' + c, c = +1 or -1 (identical to the subtraction of -1 or 1).  The FP64 pipe is
    // this form's limit, so the addition sits in a branch that a warp takes only when
    // one of its particles crossed (most ion warps do not).  A result that rounds up to
    // 1 (f' a tiny negative number) is renormalised to the next cell from its bits.
    static __device__ __forceinline__ void move(double& f, double u, int& j)
    {
        const double xn = f + u;
        const int hi = __double2hiint(xn);
        const int e = (hi >> 20) & 0x7FF;
        if (__builtin_expect(e < 1023 || (e == 1023 && hi >= 0), 1)) {
            const bool neg = hi < 0;   // -1 < f' < 0, or f' = -0
            const bool up = e == 1023; // 1 <= f' < 2
            double fk = xn;            // 0 <= f' < 1: f' itself
            if (__builtin_expect(neg || up, 0)) {
                fk = xn + __hiloint2double(neg ? 0x3FF00000 : (int)0xBFF00000u, 0);
                j += neg ? -1 : 1;
                if (__double2hiint(fk) == 0x3FF00000) {  // fk in [0, 1]: this is fk == 1
                    fk = 0.0;
                    j += 1;
                }
            }
            f = fk;
            return;
        }
        const double fl = floor(xn);
        double fk = xn - fl;
        j += (int)fl;
        if (fk >= 1.0) {
            fk = 0.0;
            j += 1;
        }
        f = fk;
    }
    // The same in two halves.  First f' alone and the cells crossed, -1, 0 or 1, as if
    // -1 < f' < 2; then, for the quad's crossed particles, add_crossed: the one addition
    // f' - dj, and what is_far() finds outside.
    static __device__ __forceinline__ bool move_fast(double& f, double u, int& dj)
    {
        f = f + u;
        dj = near_cells(f);
        return false;
    }
    static __device__ __forceinline__ int near_cells(double x)
    {
        const int hi = __double2hiint(x);
        return hi < 0 ? -1 : (hi >= 0x3FF00000 ? 1 : 0);
    }
    // not -1 < x < 2 (or not a number)
    static __device__ __forceinline__ bool is_far(double x)
    {
        const int hi = __double2hiint(x);
        return (hi & 0x7FFFFFFF) >= (hi < 0 ? 0x3FF00000 : 0x40000000);
    }
    // floor(x) of |x| >= 1 from the bits (integer ALU); INT_MIN, where no cell lies, from 2^21
    // cells on and for an x that is not finite.
    static __device__ __forceinline__ int far_cells(double x)
    {
        const int hi = __double2hiint(x), e = ((hi >> 20) & 0x7FF) - 1023;
        if (e > 20) return INT_MIN;
        const int m = (hi & 0xFFFFF) | 0x100000, whole = m >> (20 - e);
        const bool part = (m & ((1 << (20 - e)) - 1)) != 0 || __double2loint(x) != 0;
        return hi < 0 ? -whole - (part ? 1 : 0) : whole;
    }
};

// Resident blocks per SM each mover variant is compiled for (its register budget).
// FULL: the variant for the steps on which every clock tests.
template <typename T, bool MAG, int NT, bool FULL = false>
struct MoveOccupancy {
    static constexpr int warps = MAG ? Prec<T>::min_warps_mag
                                 : FULL ? Prec<T>::min_warps_full
                                 : NT == 512 ? Prec<T>::min_warps_512 : Prec<T>::min_warps;
    static constexpr int blocks = warps / (NT / 32) > 0 ? warps / (NT / 32) : 1;
};

// The quad's four values of one array with one 128-bit access (two for double).  The
// particle arrays are streamed (each byte is read and written once per step, and the
// store is far larger than L2), so the accesses carry the evict-first hint and leave L2
// to the node arrays, the deposit and the rare-event queue.
__device__ __forceinline__ void ld4(const float* p, float v[4])
{
    const float4 t = __ldcs(reinterpret_cast<const float4*>(p));
    v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
}
__device__ __forceinline__ void ld4(const double* p, double v[4])
{
    const double2 a = __ldcs(reinterpret_cast<const double2*>(p));
    const double2 b = __ldcs(reinterpret_cast<const double2*>(p) + 1);
    v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
}
__device__ __forceinline__ void st4(float* p, const float v[4])
{
    __stcs(reinterpret_cast<float4*>(p), make_float4(v[0], v[1], v[2], v[3]));
}
__device__ __forceinline__ void st4(double* p, const double v[4])
{
    __stcs(reinterpret_cast<double2*>(p), make_double2(v[0], v[1]));
    __stcs(reinterpret_cast<double2*>(p) + 1, make_double2(v[2], v[3]));
}

// Warp-level deposit of four particles per lane.  With Q = rint(f S) the charge of one
// particle is S - Q on node j and Q on node j+1; a tile of 128 particles puts at most
// 128 S on a node, so a node's sum fits 32 bits (FP64: two words).  The
// warp forms the sums of the nodes of its range [wmin, wmax + 1]; lane l then owns node
// wmin + l and adds its sum to HBM with one 64-bit reduction (no return value, so nothing
// waits on it).  A warp whose particles sit in a few cells (the store was sorted
// recently) forms them by register reductions, one per node: a lane's shares of node i
// are S - Q of its particles in cell i and Q of those in cell i-1, which the round before
// has added up.  One whose particles have spread over more cells (late in a sort cycle)
// adds each particle's two shares into a window of 32 nodes in shared memory (`win`, the
// warp's own, zero outside this call; kDepReps copies side by side, a lane's by its
// number, so that lanes in one cell seldom meet), which costs the same few instructions
// whatever the spread; FP64 adds its count and its Q to its cell instead, two words where two
// shares are four, and node i gets n_i S - R_i + R_{i-1} (n particles in the cell, R the sum
// of their Q).  Beyond 32 nodes every particle goes to HBM on its own.
// A negative jd marks an empty slot: as unsigned it is never the minimum of a live cell,
// as signed never the maximum, and it matches no cell.
// gdep null (OPT variants): only the counts, for a species whose deposit stands.
// Register reductions up to kDepLoop cells: 196.6 M particles, FP32, 256-thread blocks: 0.644
// ms at 2, 0.655 at 3, 0.662 at 5; FP64 1.384 at 2, 1.402 at 3, 1.409 at 4 (with a window of
// four atomics a particle, two halves of two shares, 1.402 at its best, 3).
constexpr int kDepLoop = 2;
constexpr int kDepReps = 4;

// Words of a warp's deposit window: 32 nodes of kDepReps copies.  FP64: 32 cells, first the
// low 21 bits of Q above a count, then its high 27 bits; a copy sees at most 32 particles of
// a tile, so the counts fit six bits, and either word's sum 32.
template <typename Q>
struct DepWin {
    static constexpr int words = 32 * kDepReps * (sizeof(Q) / 4);
};

// Clear the warp's window (once, before its first deposit).
template <typename Q>
__device__ __forceinline__ void dep_win_clear(uint32_t* win)
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int i = 0; i < DepWin<Q>::words / 32; ++i) win[32 * i + lane] = 0u;
    __syncwarp();
}

// A lane's copies in the window, which are cleared.
__device__ __forceinline__ uint4 dep_win_take(uint32_t* win)
{
    uint4* const p = reinterpret_cast<uint4*>(win) + (threadIdx.x & 31);
    const uint4 v = *p;
    *p = make_uint4(0u, 0u, 0u, 0u);
    return v;
}

template <typename Q, bool OPT = false>
__device__ __forceinline__ void warp_deposit(const int jd[4], const Q qr[4],
                                             unsigned long long S,
                                             unsigned long long* __restrict__ gdep,
                                             unsigned* __restrict__ ghist,
                                             uint32_t* __restrict__ win)
{
    static_assert(kDepReps == 4, "dep_win_take reads the copies as one uint4");
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const unsigned lmin = min(min((unsigned)jd[0], (unsigned)jd[1]), min((unsigned)jd[2], (unsigned)jd[3]));
    const int lmax = max(max(jd[0], jd[1]), max(jd[2], jd[3]));
    const int wmin = (int)__reduce_min_sync(FULL, lmin);
    if (wmin < 0) return;  // no live particle in the tile
    const int wmax = __reduce_max_sync(FULL, lmax);
    const int ncell = wmax - wmin + 1;
    if (ncell < 32) {
        if (!OPT || gdep) {
            unsigned long long tot = 0;  // the sum of node wmin + lane
            if (ncell <= kDepLoop) {
                Q left[4], carry = 0;
#pragma unroll
                for (int k = 0; k < 4; ++k) left[k] = (Q)S - qr[k];
#pragma unroll 1
                for (int i = 0; i <= ncell; ++i) {
                    Q l = carry, rr = 0;
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        if (jd[k] == wmin + i) {
                            l += left[k];
                            rr += qr[k];
                        }
                    carry = rr;
                    if (sizeof(Q) == 4) {
                        const uint32_t t = __reduce_add_sync(FULL, (uint32_t)l);
                        if (lane == i) tot = t;
                    } else {
                        const uint32_t lo = __reduce_add_sync(FULL, (uint32_t)((uint64_t)l & 0xFFFFFFu));
                        const uint32_t hi = __reduce_add_sync(FULL, (uint32_t)((uint64_t)l >> 24));
                        if (lane == i) tot = ((unsigned long long)hi << 24) + lo;
                    }
                }
            } else {
                uint32_t* const w = win + (lane & (kDepReps - 1));
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    if (jd[k] < 0) continue;
                    if (sizeof(Q) == 4) {
                        uint32_t* const p = w + kDepReps * (jd[k] - wmin);
                        atomicAdd(p, (uint32_t)S - (uint32_t)qr[k]);
                        atomicAdd(p + kDepReps, (uint32_t)qr[k]);
                    } else {
                        // (Q = S, an offset that rounds up to 1: the next cell's, with Q = 0)
                        const uint64_t q = (uint64_t)qr[k];
                        uint32_t* const p = w + kDepReps * (jd[k] - wmin + (int)(q >> 48));
                        atomicAdd(p, ((uint32_t)q & 0x1FFFFFu) << 6 | 1u);
                        atomicAdd(p + 32 * kDepReps, (uint32_t)(q >> 21) & 0x7FFFFFFu);
                    }
                }
                __syncwarp();
                if (sizeof(Q) == 4) {
                    const uint4 v = dep_win_take(win);
                    tot = (v.x + v.y) + (v.z + v.w);
                } else {
                    const uint4 a = dep_win_take(win), b = dep_win_take(win + 32 * kDepReps);
                    const uint32_t n = (a.x & 63u) + (a.y & 63u) + (a.z & 63u) + (a.w & 63u);
                    const uint32_t lo = (a.x >> 6) + (a.y >> 6) + (a.z >> 6) + (a.w >> 6);
                    const uint64_t hi = ((uint64_t)b.x + b.y) + ((uint64_t)b.z + b.w);
                    const unsigned long long R = (hi << 21) + lo;
                    const unsigned long long prev = __shfl_up_sync(FULL, R, 1);
                    tot = S * n - R + (lane > 0 ? prev : 0ull);
                }
                __syncwarp();
            }
            // (lanes past the range hold zeros)
            if (tot != 0) atomicAdd(gdep + wmin + lane, tot);
        }
        if (ghist) {  // the particles per cell, for a sort in the next step
            uint32_t n = 0;
#pragma unroll 1
            for (int i = 0; i < ncell; ++i) {
                uint32_t t = 0;
#pragma unroll
                for (int k = 0; k < 4; ++k) t += __popc(__ballot_sync(FULL, jd[k] == wmin + i));
                if (lane == i) n = t;
            }
            if (n != 0u) atomicAdd(ghist + wmin + lane, n);
        }
    } else {
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (jd[k] >= 0) {
                const unsigned long long l = S - (unsigned long long)qr[k], rr = qr[k];
                if (!OPT || gdep) {
                    atomicAdd(gdep + jd[k], l);
                    atomicAdd(gdep + jd[k] + 1, rr);
                }
                if (ghist) atomicAdd(ghist + jd[k], 1u);
            }
    }
}

// Sort step: the slot of each particle that was in the quad at the start of the step
// (-1: none) from its group's reservation and its rank in the group; a reservation past
// the segment (a histogram that does not match the store, which no path produces) is
// refused and latched rather than written.
__device__ __forceinline__ void sort_destinations(const MoveArgs& a, const SegParams& P,
                                                  const unsigned grp[4], const unsigned rbase[4],
                                                  unsigned had, int64_t to[4])
{
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const unsigned b = __shfl_sync(0xffffffffu, rbase[k], __ffs(grp[k]) - 1);
        to[k] = -1;
        if (had & (1u << k)) {
            const int64_t r = (int64_t)b + __popc(grp[k] & lt);
            if (r < P.cap) to[k] = P.base + r;
            else set_error(a.err, kErrCapacity);
        }
    }
}

// Sort step: the quad's particles into their slots of the other store copy (a particle
// that left through a wall goes there as an empty slot with its velocity, for the event
// kernel).  Streaming stores: the next step reads the copy back from HBM anyway, and
// evict-first lines leave L2 to the partly written lines of other warps' runs.
template <typename T>
__device__ __forceinline__ void sort_write(const MoveArgs& a, const int64_t to[4], const int c[4],
                                           const T f[4], const T ux[4], const T uy[4],
                                           const T uz[4], const uint32_t id[4])
{
    T* const doff = static_cast<T*>(a.doff);
    T* const dux = static_cast<T*>(a.dux);
    T* const duy = static_cast<T*>(a.duy);
    T* const duz = static_cast<T*>(a.duz);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        if (to[k] < 0) continue;
        const int64_t g = to[k];
        __stcs(a.dcell + g, c[k]);
        __stcs(doff + g, f[k]);
        __stcs(dux + g, ux[k]);
        __stcs(duy + g, uy[k]);
        __stcs(duz + g, uz[k]);
        __stcs(a.did + g, id[k]);
    }
}

// The push of one particle (step 2) in cells per own step: u += acc with acc the
// acceleration at its position, or (smag) the Boris rotation with acc half of it
// (SegParams.accel carries the half of a magnetized instance).  PLANAR: B lies in the x-y
// plane (t_z = s_z = 0), where the four multiply-adds with t_z and s_z would only add a
// zero, which leaves every value but the sign of a zero; without them and the halving the
// FP64 form, bound by the FP64 pipe, does 12 operations instead of 17 a particle (40
// magnetized instances, 39 M particles: mover 1.45 -> 1.08 ms; 4,096 cells x 200 x 2: 110 ->
// 95 us a step).  An infinite u_y then no longer meets a product
// with 0, so the caller tests all three components for finiteness.
template <typename T, bool MAG, bool PLANAR>
__device__ __forceinline__ void push(const SegParams& P, bool smag, T acc, T& ux, T& uy, T& uz)
{
    if (!MAG || !smag) {
        ux = ux + acc;
        return;
    }
    const T t0 = Prec<T>::bt(P, 0), t1 = Prec<T>::bt(P, 1), t2 = Prec<T>::bt(P, 2);
    const T s0 = Prec<T>::bs(P, 0), s1 = Prec<T>::bs(P, 1), s2 = Prec<T>::bs(P, 2);
    const T mx = ux + acc, my = uy, mz = uz;
    // v' = v + v x t, v+ = v + v' x s, each component as two fused
    // multiply-adds (m_x + m_y t_z - m_z t_y = fma(m_y, t_z, fma(-m_z, t_y, m_x)))
    const T px0 = Prec<T>::fma_(-mz, t1, mx), py0 = PLANAR ? my : Prec<T>::fma_(-mx, t2, my);
    const T px = PLANAR ? px0 : Prec<T>::fma_(my, t2, px0);
    const T py = Prec<T>::fma_(mz, t0, py0);
    const T pz = Prec<T>::fma_(mx, t1, Prec<T>::fma_(-my, t0, mz));
    const T qx0 = Prec<T>::fma_(-pz, s1, mx), qy0 = PLANAR ? my : Prec<T>::fma_(-px, s2, my);
    const T qx = PLANAR ? qx0 : Prec<T>::fma_(py, s2, qx0);
    ux = qx + acc;
    uy = Prec<T>::fma_(pz, s0, qy0);
    uz = Prec<T>::fma_(px, s1, Prec<T>::fma_(-py, s0, mz));
}

// A tile's state on its way through shared memory: each lane copies its own quad (16
// bytes an access) with cp.async one tile ahead and reads it back itself, so a warp keeps
// a whole tile's loads in flight while it works on the tile before, without registers
// for them.  Once its instructions had gone from 448 to 289 a tile the FP32 mover waited
// for HBM with 46 warps' loads in flight (0.730 ms for 196.6 M particles); with the ring
// and kMoveChunk (engine.cu) it takes 0.64-0.65 ms, 6.1 TB/s of the 20 B a particle it
// moves in fact.  One stage: the cell words, off and ux of a warp's tile.
template <typename T>
struct TileRing {
    static constexpr int words = 128 + 2 * 128 * (int)(sizeof(T) / 4);  // one stage
    static constexpr size_t bytes(int nt) { return (size_t)(nt / 32) * 2 * words * 4; }
};
// Dynamic shared memory of a block of the mover: the rings of the variants that fetch ahead.
template <typename T, MoveMode MODE>
constexpr size_t ring_bytes(int nt)
{
    return MODE == MoveMode::kAhead ? TileRing<T>::bytes(nt) : 0;
}
// L2 policy of streamed reads: evict first (as the 128-bit loads' hint).
__device__ __forceinline__ uint64_t stream_policy()
{
    uint64_t p;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
    return p;
}
__device__ __forceinline__ void copy16(uint32_t dst, const void* src, uint64_t policy)
{
    asm volatile("cp.async.cg.shared.global.L2::cache_hint [%0], [%1], 16, %2;" ::"r"(dst), "l"(src),
                 "l"(policy)
                 : "memory");
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void copy_wait_1() { asm volatile("cp.async.wait_group 1;" ::: "memory"); }
// The lane's share of one array of a tile: four values of type V.
template <typename V>
__device__ __forceinline__ void copy_quad(uint32_t dst, const V* src, uint64_t policy)
{
    const uint32_t d = dst + (threadIdx.x & 31) * 4 * sizeof(V);
    copy16(d, src, policy);
    if (sizeof(V) == 8) copy16(d + 16, src + 2, policy);
}
__device__ __forceinline__ void take_quad(const uint32_t* p, float v[4])
{
    const float4 t = reinterpret_cast<const float4*>(p)[threadIdx.x & 31];
    v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
}
__device__ __forceinline__ void take_quad(const uint32_t* p, double v[4])
{
    const double2* q = reinterpret_cast<const double2*>(p) + 2 * (threadIdx.x & 31);
    const double2 a = q[0], b = q[1];
    v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
}

// Put a particle on the step's list for the event kernel.
__device__ __forceinline__ void queue_rare(const MoveArgs& a, int s, int64_t slot, uint32_t kind)
{
    const unsigned long long e = atomicAdd(a.rare_count, 1ull);
    if (e < (unsigned long long)a.rare_cap) a.rare[e] = rare_pack(slot, s, kind);
    else set_error(a.err, kErrEvents);
}

// The clock bits that follow a test at own step mown whose draw gives `run` candidate-free
// own steps; dgrid: the own steps to the species' next multiple of kGapMax.  now: a
// candidate on this very step.
__device__ __forceinline__ uint32_t clock_after_test(int run, int64_t mown, int dgrid, bool& now)
{
    const int g = min(run, dgrid);
    now = g == 0;
    return clock_bits(now ? mown + 1 : mown + g, g > 0 && g < dgrid);
}

// Steps 1-5 of the time step for one live particle: gather, push, move, walls,
// collision clock.  c, f, u* hold its state on entry and its new state on exit (cell
// word -1: left through a wall).  mown is the species' own index of this step (its
// clock's time), dgrid the own steps to its next multiple of kGapMax; run() gives the
// candidate-free run of this step's test draw.  Returns what the event kernel has to do
// with the particle (kRareCandidate, kRareWallLow, kRareWallHigh) or -1.
template <typename T, bool MAG, typename Run>
__device__ __forceinline__ int particle_step(const MoveArgs& a, const SegParams& P, bool smag,
                                             int64_t mown, int dgrid, Run run, int& c, T& f, T& ux,
                                             T& uy, T& uz)
{
    using T2 = typename Prec<T>::T2;
    const int N = P.ncells;
    int j = (int)((uint32_t)c & kCellMask);
    uint32_t clk = (uint32_t)c >> kClockShift;
    if (!in_range(a.err, j, 0, N)) {  // (bounds-checked build only)
        c = -1;
        return -1;
    }
    // 1. gather (Listing 7) from the node pair (A_j, A_{j+1} - A_j)
    const T2 pr = __ldg(static_cast<const T2*>(a.accel) + P.node + j);
    T fk = f;
    // 2. push
    if (MAG && P.planar) push<T, MAG, true>(P, smag, Prec<T>::fma_(fk, pr.y, pr.x), ux, uy, uz);
    else push<T, MAG, false>(P, smag, Prec<T>::fma_(fk, pr.y, pr.x), ux, uy, uz);
    if (!Prec<T>::finite(ux) || (MAG && smag && !(Prec<T>::finite(uy) && Prec<T>::finite(uz))))
        set_error(a.err, kErrNonFinite);
    // 3. move (Listing 7: x += nstep*vx, x the in-cell offset)
    Prec<T>::move(fk, ux, j);
    f = fk;
    // 4. walls: periodic wrap here; an absorbed or re-injected particle
    // leaves the store and the event kernel takes over
    if (j < 0 || j >= N) {
        if (P.bc != PIC_BC_PERIODIC) {
            c = -1;
            return j < 0 ? (int)kRareWallLow : (int)kRareWallHigh;
        }
        j %= N;
        if (j < 0) j += N;
    }
    // 5. null collision.  The candidate steps of a particle form a
    // Bernoulli(P) sequence; its clock names the own step of its next event
    // step.  At an event step without a pending candidate (a test), Philox word
    // 0 gives the candidate-free run g from this step, cut at the next multiple
    // of 127 (D steps away): g = 0 candidate now, g < D a candidate g steps
    // later, g = D none before then.  The cut puts the tests of all particles on
    // the same steps.  Candidates go to the event kernel.  Between events the
    // clock, and so the word, does not change.
    int ev = -1;
    if (P.collide && (clk & kClockDue) == (uint32_t)(mown & (int64_t)kClockDue)) {
        if (clk & kClockPending) {
            ev = (int)kRareCandidate;
            // a test next step (the event kernel draws it when it takes the
            // candidate and puts its outcome in the clock)
            clk = (uint32_t)((mown + 1) & (int64_t)kClockDue);
        } else {
            bool now;
            clk = clock_after_test(run(), mown, dgrid, now) >> kClockShift;
            if (now) ev = (int)kRareCandidate;
        }
    }
    c = (int)((uint32_t)j | (clk << kClockShift));
    return ev;
}

// The FP64 additions of a tile's crossed particles (move_fast), `cross` a bit per quad
// position.  A tenth of the electrons cross a cell edge in a step, so with an addition
// per quad position nearly every warp would issue all four for a few lanes each; the FP64
// pipe, which takes a warp's addition at the same price however few its lanes, is this
// form's limit.  The crossed values are brought together in `scr` (32 doubles of the
// warp) and added 32 at a time: one addition a tile.  Particles that crossed more than one
// edge, or are not finite, are looked for here, among the crossed ones: their cell words take
// the edges that near_cells did not count, and their addition is f' - floor(f').  (Left to
// rare_quad, one quad at a time: at a thermal speed of 0.8 cells a step the mover of 9.8 M
// particles took 203 us, 176 now; of 3.3 M magnetized ones 179, 124.)  True when a sum
// rounded up to 1 or a far particle left [0, N) (one that near_cells' step takes past a wall
// has left it: the steps have one sign).
__device__ __forceinline__ bool add_crossed(int c[4], int N, double f[4], unsigned cross, double* scr)
{
    using D = Prec<double>;
    const unsigned FULL = 0xffffffffu;
    if (!__any_sync(FULL, cross != 0u)) return false;
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    int at[4], n = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const unsigned b = __ballot_sync(FULL, cross >> k & 1u);
        at[k] = (cross >> k & 1u) ? n + __popc(b & lt) : -1;
        n += __popc(b);
    }
    bool odd = false;
#pragma unroll 1
    for (int r0 = 0; r0 < n; r0 += 32) {
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if ((unsigned)(at[k] - r0) < 32u && at[k] >= 0) scr[at[k] - r0] = f[k];
        __syncwarp();
        bool far = false;
        if (r0 + lane < n) {
            const double x = scr[lane];
            far = D::is_far(x);
            scr[lane] = x + __hiloint2double(__double2hiint(x) < 0 ? 0x3FF00000 : (int)0xBFF00000u, 0);
        }
        if (__any_sync(FULL, far)) {
            __syncwarp();  // (the owners write over the lanes' sums)
#pragma unroll 1
            for (int k = 0; k < 4; ++k) {
                const double x = k == 0 ? f[0] : k == 1 ? f[1] : k == 2 ? f[2] : f[3];
                const int p = k == 0 ? at[0] : k == 1 ? at[1] : k == 2 ? at[2] : at[3];
                if (p < r0 || p >= r0 + 32 || !D::is_far(x)) continue;
                const int dj = D::far_cells(x), more = (int)((uint32_t)dj - (uint32_t)D::near_cells(x));
                const int ck = k == 0 ? c[0] : k == 1 ? c[1] : k == 2 ? c[2] : c[3];
                const uint32_t w = (uint32_t)ck + (uint32_t)more;
                odd |= ((w - (uint32_t)dj) & kCellMask) + (uint32_t)dj >= (uint32_t)N;
                c[0] = k == 0 ? (int)w : c[0];
                c[1] = k == 1 ? (int)w : c[1];
                c[2] = k == 2 ? (int)w : c[2];
                c[3] = k == 3 ? (int)w : c[3];
                scr[p - r0] = x - floor(x);
            }
        }
        __syncwarp();
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if ((unsigned)(at[k] - r0) < 32u && at[k] >= 0) {
                f[k] = scr[at[k] - r0];
                odd |= __double2hiint(f[k]) == 0x3FF00000;
            }
        __syncwarp();
    }
    return odd;
}
__device__ __forceinline__ bool add_crossed(int*, int, float*, unsigned, double*) { return false; }
// Words of that scratch.
template <typename T>
struct CrossScratch {
    static constexpr int words = sizeof(T) == 8 ? 64 : 0;
};

// The segment constants of the common path, held in registers across the tiles of a
// segment.  A particle's clock is due when (c ^ due) & clkmask == 0; a species without
// collisions gets a pattern that only an empty slot (bit 31) matches.
struct SegFast {
    int N;
    uint32_t clkmask, due;
    bool planar;
    __device__ __forceinline__ void set(const SegParams& P, int64_t mown)
    {
        N = P.ncells;
        planar = P.planar != 0;
        clkmask = P.collide ? kClockDue << kClockShift : 0x80000000u;
        due = P.collide ? ((uint32_t)mown & kClockDue) << kClockShift : 0x80000000u;
    }
};

// The particles of a quad that the common path moved through an absorbing or source wall:
// their slots emptied and `walls` set, bit k at the low wall and bit 4+k at the high one.
// Cell words as quad_fast leaves them (the cells crossed added, so that the low bits are the
// cell's, of either sign).  False, with nothing changed, when the quad needs more than that:
// an offset that rounded up to 1, a velocity that is not finite or takes a particle further
// than the bits show.
template <typename T>
__device__ __forceinline__ bool quad_walls(int N, int c[4], const T f[4], const T ux[4], int& walls)
{
    constexpr int far = 1 << 20;  // (far_cells counts to twice that)
    bool ok = N <= 2 * far;
#pragma unroll
    for (int k = 0; k < 4; ++k) ok = ok && f[k] < T(1) && ux[k] < T(far) && ux[k] > T(-far);
    if (!ok) return false;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int j = (int)((uint32_t)c[k] << (32 - kClockShift)) >> (32 - kClockShift);
        if ((uint32_t)j < (uint32_t)N) continue;
        c[k] = -1;
        walls |= (j < 0 ? 1 : 16) << k;
    }
    return true;
}

// Steps 1-5 for the four particles of one quad (a lane's share of a tile), the common
// case: live particles that stay inside the walls.  The mover is bound by its
// instructions as much as by HBM, so this runs without branches: the cell is the word's
// low bits, so the new word is the old one plus the cells crossed.  due: a clock of the
// quad is due (quad_due), or a particle left through a wall (WALLS, quad_walls).  Returns true
// when some particle needs more than that: the whole quad is then done over by rare_quad from
// the state in memory, which must not have been written before.  (A wrapped particle is left
// to it as well: with the others of its tile it would spread the warp's deposit from the
// first cell to the last.)  WALLS: the plain push alone; in the Boris form and the sort step
// the code costs the common path more registers than the rare quads cost.
template <typename T, bool MAG, bool WALLS = false>
__device__ __forceinline__ bool quad_fast(const SegParams& P, const SegFast& F, bool smag,
                                          const typename Prec<T>::T2* __restrict__ accn, int c[4],
                                          T f[4], T ux[4], T uy[4], T uz[4], bool& moved, bool& due,
                                          int& walls, double* scr)
{
    using T2 = typename Prec<T>::T2;
    // an empty slot is given a particle at rest in the first cell, its clock not due, and
    // emptied again below
    unsigned empty = 0;
    if ((c[0] | c[1] | c[2] | c[3]) < 0) {
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (c[k] < 0) {
                empty |= 1u << k;
                c[k] = (int)((F.due ^ (1u << kClockShift)) & (kClockDue << kClockShift));
                f[k] = T(0.5);
                ux[k] = T(0);
                if (MAG) uy[k] = uz[k] = T(0);
            }
    }
    T2 pr[4];
#pragma unroll
    for (int k = 0; k < 4; ++k)  // (the clamp only bounds a corrupted word)
        pr[k] = __ldg(accn + min((uint32_t)c[k] & kCellMask, (uint32_t)F.N));
    bool rare = false;
    int crossed = 0;
    unsigned cross = 0;
    due = false;
    if (MAG && F.planar) {
#pragma unroll
        for (int k = 0; k < 4; ++k)
            push<T, MAG, true>(P, smag, Prec<T>::fma_(f[k], pr[k].y, pr[k].x), ux[k], uy[k], uz[k]);
    } else {
#pragma unroll
        for (int k = 0; k < 4; ++k)
            push<T, MAG, false>(P, smag, Prec<T>::fma_(f[k], pr[k].y, pr[k].x), ux[k], uy[k], uz[k]);
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        int dj;
        rare |= Prec<T>::move_fast(f[k], ux[k], dj);
        if (MAG) rare |= !Prec<T>::finite(uy[k]) || !Prec<T>::finite(uz[k]);
        rare |= (uint32_t)((int)((uint32_t)c[k] & kCellMask) + dj) >= (uint32_t)F.N;
        due |= (((uint32_t)c[k] ^ F.due) & F.clkmask) == 0u;
        c[k] += dj;
        crossed |= dj;
        if (sizeof(T) == 8 && dj != 0) cross |= 1u << k;
    }
    rare |= add_crossed(c, F.N, f, cross, scr);
    if (WALLS && rare && P.bc != PIC_BC_PERIODIC) {
        rare = !quad_walls<T>(F.N, c, f, ux, walls);
        due |= walls != 0;
    }
    if (empty) {
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (empty >> k & 1) c[k] = -1;
    }
    moved = crossed != 0;
    return rare;
}

// A quad of the common path with a due clock: in bits 0-3 its pending collision candidates,
// whose clocks are set to the test that follows (the event kernel draws it when it takes
// the candidate), in bits 4-7 the clocks that test on this step, left to test_clock.
__device__ __forceinline__ int quad_due(const SegFast& F, int c[4])
{
    constexpr uint32_t pend = kClockPending << kClockShift;
    const uint32_t mask = F.clkmask | pend, next = (F.due + (1u << kClockShift)) & F.clkmask;
    int ev = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        if (c[k] < 0) continue;
        const uint32_t d = ((uint32_t)c[k] ^ F.due) & mask;
        if (d == 0u) ev |= 16 << k;
        if (d == pend) {
            ev |= 1 << k;
            c[k] = (int)(((uint32_t)c[k] & kCellMask) | next);
        }
    }
    return ev;
}

// The species' own index of step `step` (its clock's time) and the own steps to its next
// multiple of kGapMax.
__device__ __forceinline__ void own_time(const SegParams& P, int64_t step, int64_t& mown, int& dgrid)
{
    mown = P.nstep == 1 ? step : (step + 1) / P.nstep - 1;
    dgrid = kGapMax - (int)(mown % kGapMax);
}

// The clock test of one particle of the common path, whose word after the move is c: the
// word with the clock that follows, its candidate of this step queued at slot `to` (-1:
// none, nothing is queued).
__device__ __forceinline__ int test_clock(const MoveArgs& a, const SegParams& P, int s, int64_t step,
                                          int64_t mown, int dgrid, uint32_t id, int c, int64_t to)
{
    bool now;
    const uint32_t clk = clock_after_test(
        gap_steps(P.gap, P.glog, draw(id, step, kRngCollide, P.key0, P.key1).x), mown, dgrid, now);
    if (now && to >= 0) queue_rare(a, s, to, kRareCandidate);
    return (int)(((uint32_t)c & kCellMask) | clk);
}

// The clock tests of a quad that is in memory again after its step (plain step), `test` a bit
// per quad position.  Only the clocks are left to do: the quad's move and its share of the
// warp's deposit are the common path's.  (Doing such quads over one particle at a time, with
// two 64-bit atomics each, took 5.5 ms for the 14.3 M particles of a 256-cell plasma on the
// steps on which every clock tests, and 72 us on the others.)
__device__ __forceinline__ void test_quad(const MoveArgs& a, int s, int64_t step, int64_t slot, int test)
{
    const SegParams& P = a.seg[s];
    int64_t mown;
    int dgrid;
    own_time(P, step, mown, dgrid);
    const uint4 id = __ldcs(reinterpret_cast<const uint4*>(a.id + slot));
    const int4 c = *reinterpret_cast<const int4*>(a.cell + slot);
#pragma unroll 1
    for (int k = 0; k < 4; ++k)
        if (test >> k & 1)
            a.cell[slot + k] = test_clock(a, P, s, step, mown, dgrid,
                                          k == 0 ? id.x : k == 1 ? id.y : k == 2 ? id.z : id.w,
                                          k == 0 ? c.x : k == 1 ? c.y : k == 2 ? c.z : c.w, slot + k);
}

// test_quad called: inlined, its registers moved the schedule of the plain push's loop (196.6 M
// particles, FP32: 650 against 646 us; the sort step, below, 2.28 against 2.22 ms).  The
// Boris form takes it inlined, with rare_quad: a call reads the kernel's arguments through
// memory, which every step with an ionization product waits for (256 cells x 100 x 2: FP32
// 22.7 against 20.8 us a step, FP64 36.7 against 34.6).
static __device__ __noinline__ void test_quad_called(const MoveArgs& a, int s, int64_t step,
                                                     int64_t slot, int test)
{
    test_quad(a, s, step, slot, test);
}

// The same of a quad staged for the sort at the places pk of the chunk's arrays (-1: none);
// `ev` as quad_due gives it.
static __device__ __noinline__ void test_staged(const MoveArgs& a, int s, int64_t step, int ev, short4 pk,
                                                int* s_cell, const uint32_t* s_id,
                                                const uint32_t* s_dst)
{
    const SegParams& P = a.seg[s];
    int64_t mown;
    int dgrid;
    own_time(P, step, mown, dgrid);
#pragma unroll 1
    for (int k = 0; k < 4; ++k) {
        const int p = k == 0 ? pk.x : k == 1 ? pk.y : k == 2 ? pk.z : pk.w;
        if (!(ev >> k & 16) || p < 0) continue;
        const uint32_t d = s_dst[p];
        s_cell[p] = test_clock(a, P, s, step, mown, dgrid, s_id[p], s_cell[p],
                               d == 0xFFFFFFFFu ? (int64_t)-1 : P.base + (int64_t)d);
    }
}

// One particle of a quad the common path left, from the state in memory at slot g:
// steps 1-5, its deposit (and count) straight to HBM, its event queued at slot `to` (where
// it lies after the step; -1: none, nothing is queued).  The caller writes the state.
template <typename T, bool MAG>
__device__ __forceinline__ void rare_particle(const MoveArgs& a, const SegParams& P, int s,
                                              bool smag, int64_t step, int64_t mown, int dgrid,
                                              int64_t g, int64_t to, int& c, T& f, T& ux, T& uy,
                                              T& uz)
{
    f = static_cast<const T*>(a.off)[g];
    ux = static_cast<const T*>(a.ux)[g];
    if (MAG && smag) {
        uy = static_cast<const T*>(a.uy)[g];
        uz = static_cast<const T*>(a.uz)[g];
    }
    const int ev = particle_step<T, MAG>(
        a, P, smag, mown, dgrid,
        [&] { return gap_steps(P.gap, P.glog, draw(__ldg(a.id + g), step, kRngCollide, P.key0, P.key1).x); },
        c, f, ux, uy, uz);
    if (ev >= 0 && to >= 0) queue_rare(a, s, to, (uint32_t)ev);
    const int j = (int)((uint32_t)c & kCellMask);
    if (c >= 0 && in_range(a.err, j, 0, P.ncells)) {
        const unsigned long long qr = Prec<T>::qright(f);
        atomicAdd(a.dep + P.node + j, Prec<T>::S - qr);
        atomicAdd(a.dep + P.node + j + 1, qr);
        if (a.hist_out) atomicAdd(a.hist_out + P.node + j, 1u);
    }
}

// A quad the common path left (plain step): its particles one by one, in place.
template <typename T, bool MAG>
__device__ __forceinline__ void rare_quad(const MoveArgs& a, int s, bool smag, int64_t step,
                                          int64_t slot)
{
    const SegParams& P = a.seg[s];
    int64_t mown;
    int dgrid;
    own_time(P, step, mown, dgrid);
#pragma unroll 1
    for (int64_t g = slot; g < slot + 4; ++g) {
        int c = a.cell[g];
        if (c < 0) continue;
        T f, ux, uy = T(0), uz = T(0);
        rare_particle<T, MAG>(a, P, s, smag, step, mown, dgrid, g, g, c, f, ux, uy, uz);
        a.cell[g] = c;
        static_cast<T*>(a.off)[g] = f;
        static_cast<T*>(a.ux)[g] = ux;
        if (MAG && smag) {
            static_cast<T*>(a.uy)[g] = uy;
            static_cast<T*>(a.uz)[g] = uz;
        }
    }
}

// The consecutive tiles a warp takes in a batch whose segments are short (MoveArgs.chunk =
// kSpread): up to some 32 (8: 209 against 203 us for 500 instances of 100 cells, FP64), so
// many that all warps get the same number of chunks, from the tiles that are alive.
constexpr int kSpread = 0;
// Not the FP64 Boris form, which is launched a block for every NT/32 or twice as many tiles, nor
// FP64 in blocks of 512 threads, whose 64 registers have none to spare for it (196.6 M
// particles: 1.460 against 1.466 ms; as little for quad_walls).
__host__ __device__ constexpr bool can_spread(bool f64, bool mag, int nt)
{
    return !(f64 && (mag || nt == 512));
}
__device__ __forceinline__ int spread_chunk(int total, int warps)
{
    const int tiles = max((total + warps - 1) / warps, 1), times = max((tiles + 16) / 32, 1);
    return (tiles + times - 1) / times;
}

// The fused time step.  Work unit: a warp tile of 32 quads (128 consecutive particles
// of one segment); each lane owns one quad and moves it with 128-bit accesses.  Warps
// walk the tiles of all segments independently (no block-level barrier), so every SM
// keeps many tiles' loads in flight.  The gather reads each particle's node pair with
// one vector load (the node arrays are small and stay in L1/L2).  The common
// path is free of calls; walls and collision candidates are queued for the event kernel.
// SUB: some species of the batch is subcycled (else every segment moves every step).
// MIXED (with MAG): the batch mixes magnetized and unmagnetized instances, so the push is
// chosen per segment.  MODE: kDirect loads a tile when its turn comes, for batches whose
// warps have a tile or two (a ring of two 16 KB stages a block buys nothing there and its
// set-up costs 1.5 us a step) and for the Boris form (5 to 9 KB of ring a warp; 31 M
// particles in 26 magnetized instances, FP32: 284 us a step direct, 310 fetched ahead, 125 M
// the same either way; the FP64 one is bound by the FP64 pipe);
// kAhead fetches one tile ahead (TileRing); kFull is the variant of large batches
// for the steps on which the clocks of a whole species test (the multiples of kGapMax, the
// first step after a load):
// the quad's ids are read with its state and its four draws and table lookups go side by
// side before the physics; the other steps' variant draws them one after another once the
// tile is done (test_quad), with the same results.  A segment that rests on this step
// (subcycling, a neutral particle target) keeps its deposit, so its tiles are skipped, or
// only counted per cell on the step before a sort: the 30,011-cell plasma with ions moved
// every fourth step (42 M particles, FP32) went from 212 to 183 us a step.  (The step
// that ends a sort cycle runs k_move_sort below instead.)
template <typename T, int NT, bool MAG, bool MOVE, bool SUB, bool MIXED, MoveMode MODE>
__global__ void __launch_bounds__(NT, MoveOccupancy<T, MAG, NT, MODE == MoveMode::kFull>::blocks)
k_move(const __grid_constant__ MoveArgs a)
{
    using Q = typename Prec<T>::Q;
    using T2 = typename Prec<T>::T2;
    constexpr bool PF = MODE == MoveMode::kAhead, FULL = MODE == MoveMode::kFull;
    constexpr bool WALLS = !MAG && !(sizeof(T) == 8 && NT == 512);
    static_assert(!(PF && MAG), "the Boris form loads directly");
    const int lane = threadIdx.x & 31;
    T* const offp = static_cast<T*>(a.off);
    T* const uxp = static_cast<T*>(a.ux);
    T* const uyp = static_cast<T*>(a.uy);
    T* const uzp = static_cast<T*>(a.uz);
    const int64_t step = MOVE ? a.step[1] : 0;
    // the step under way, for the kernels after the mover
    if (MOVE && blockIdx.x == 0 && threadIdx.x == 0) a.step[0] = step;
    // the warps' deposit windows and (FP64) scratch of add_crossed
    __shared__ __align__(16) uint32_t s_dwin[NT / 32][DepWin<Q>::words + CrossScratch<T>::words];
    uint32_t* const dwin = s_dwin[threadIdx.x >> 5];
    double* const scr = reinterpret_cast<double*>(dwin + DepWin<Q>::words);
    // (fewer than 2^31 tiles: 2^38 particles would not fit)
    const int total = (int)a.tile_start[a.nseg];
    // the tile ahead: its segment (tiles only increase) with that segment's last tile + 1 and
    // slots (ahead0: as if tile 0 were its), and the slot of the lane's quad
    const int chunk = !can_spread(sizeof(T) == 8, MAG, NT) || a.chunk != kSpread
                          ? a.chunk : spread_chunk(total, gridDim.x * (NT / 32));
    int tile = (blockIdx.x * (NT / 32) + (threadIdx.x >> 5)) * chunk, left = chunk - 1;
    if (tile >= total) return;  // (blocks for a reserve that is not alive)
    dep_win_clear<Q>(dwin);
    int sa = 0, sa_end = -1;
    int64_t ahead0 = 0, ahead_end = 0, ahead = 0;
    const auto next = [&]() {
        ++tile;
        if (--left < 0) {  // on to the warp's next chunk
            left = chunk - 1;
            tile += (int)(gridDim.x * (NT / 32) - 1) * chunk;
        }
    };
    const auto look = [&]() {
        while (tile < total && tile >= sa_end) {
            sa = advance_segment(a.tile_start, a.nseg, sa, tile);
            sa_end = (int)__ldg(a.tile_start + sa + 1);
            const SegParams& P = a.seg[sa];
            ahead0 = P.base - 128 * __ldg(a.tile_start + sa) + 4 * lane;
            ahead_end = P.base + a.seg_nmove[sa];
            // a species that rests keeps its deposit: the warp goes on with its first tile
            // past the segment
            if (MOVE && SUB && !a.hist_out && !moves_on(P, step))
                while (tile < sa_end) next();
        }
        ahead = ahead0 + (int64_t)tile * 128;
    };
    extern __shared__ __align__(16) uint32_t s_ring[];
    constexpr int SW = TileRing<T>::words;
    uint32_t* const ring = s_ring + (threadIdx.x >> 5) * 2 * SW;
    const uint32_t ring_at = PF ? (uint32_t)__cvta_generic_to_shared(ring) : 0u;
    const uint64_t policy = PF ? stream_policy() : 0ull;
    const auto fetch = [&](int stage) {
        if (tile < total && ahead < ahead_end) {
            const uint32_t d = ring_at + stage * SW * 4;
            copy_quad(d, a.cell + ahead, policy);
            copy_quad(d + 512, offp + ahead, policy);
            copy_quad(d + 512 + 128 * sizeof(T), uxp + ahead, policy);
        }
        copy_commit();
    };
    int s = -1;             // segment of the current tile
    int64_t node0 = 0;      // its nodes
    bool moves = MOVE;      // it moves this step (subcycling)
    bool smag = MAG;        // its instance is magnetized
    SegFast F = {0, 0u, 0u, false};
    look();
    if (PF) fetch(0);
    for (int stage = 0; tile < total; stage ^= 1) {
        const int64_t slot = ahead;
        const bool act = slot < ahead_end && in_range(a.err, slot + 3, a.seg[sa].base, a.seg[sa].base + a.seg[sa].cap);
        const bool fresh = s != sa;  // the segment's first tile here
        s = sa;
        if (fresh && MAG && MIXED) {
            // in a batch that mixes magnetized and unmagnetized instances, the latter
            // keep the plain push (and never touch uy, uz), as they would alone
            smag = a.seg[s].mag != 0;
        }
        if (fresh && MOVE && SUB) moves = moves_on(a.seg[s], step);
        int c[4] = {-1, -1, -1, -1};
        T f[4] = {T(0), T(0), T(0), T(0)}, ux[4] = {T(0), T(0), T(0), T(0)};
        T uy[4] = {T(0), T(0), T(0), T(0)}, uz[4] = {T(0), T(0), T(0), T(0)};
        uint32_t idq[4] = {0u, 0u, 0u, 0u};
        if (PF) {
            next();
            look();
            fetch(stage ^ 1);
            copy_wait_1();
            if (act) {
                const uint32_t* const w = ring + stage * SW;
                const int4 cc = reinterpret_cast<const int4*>(w)[lane];
                c[0] = cc.x; c[1] = cc.y; c[2] = cc.z; c[3] = cc.w;
                take_quad(w + 128, f);
                take_quad(w + 128 + 32 * sizeof(T), ux);
            }
        } else if (act) {
            const int4 cc = __ldcs(reinterpret_cast<const int4*>(a.cell + slot));
            c[0] = cc.x; c[1] = cc.y; c[2] = cc.z; c[3] = cc.w;
            ld4(offp + slot, f);
            if (MOVE && (!SUB || moves)) ld4(uxp + slot, ux);
            if (MOVE && MAG && smag && (!SUB || moves)) {
                ld4(uyp + slot, uy);
                ld4(uzp + slot, uz);
            }
            if (FULL) {
                const uint4 ii = __ldcs(reinterpret_cast<const uint4*>(a.id + slot));
                idq[0] = ii.x; idq[1] = ii.y; idq[2] = ii.z; idq[3] = ii.w;
            }
        }
        if (!PF) {
            next();
            look();
        }
        if (fresh) {
            const SegParams& P = a.seg[s];
            node0 = P.node;
            int64_t mown;
            int dgrid;
            own_time(P, step, mown, dgrid);
            F.set(P, mown);
        }
        // what the quad leaves until the tile is done: -1 all of it (rare_quad), else a bit per
        // clock that tests (test_quad)
        int todo = 0;
        if (MOVE && (!SUB || moves)) {
            const SegParams& P = a.seg[s];
            bool moved = false;
            if (FULL) {
                // a clock that does not test ignores its draw
                int gq[4] = {0, 0, 0, 0};
                if (P.collide) {
                    uint32_t w[4];
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        w[k] = draw(idq[k], step, kRngCollide, P.key0, P.key1).x;
#pragma unroll
                    for (int k = 0; k < 4; ++k) gq[k] = gap_steps(P.gap, P.glog, w[k]);
                }
                int64_t mown;
                int dgrid;
                own_time(P, step, mown, dgrid);
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    if (c[k] < 0) continue;
                    const int cw = c[k];
                    const int ev = particle_step<T, MAG>(a, P, smag, mown, dgrid,
                                                         [&] { return gq[k]; }, c[k], f[k], ux[k],
                                                         uy[k], uz[k]);
                    if (ev >= 0) queue_rare(a, s, slot + k, (uint32_t)ev);
                    moved |= c[k] != cw;
                }
            } else {
                bool due;
                int walls = 0;
                const bool rare = quad_fast<T, MAG, WALLS>(P, F, smag, static_cast<const T2*>(a.accel) + node0,
                                                           c, f, ux, uy, uz, moved, due, walls, scr);
                if (rare && act) todo = -1;
                if (due && act && !rare) {
                    const int ev = quad_due(F, c);
                    todo = ev >> 4;
                    moved = true;
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        if (ev >> k & 1) queue_rare(a, s, slot + k, kRareCandidate);
                        if (WALLS && (walls >> k & 17))
                            queue_rare(a, s, slot + k, walls >> k & 1 ? kRareWallLow : kRareWallHigh);
                    }
                }
            }
            // the cell words go back only where one of them changed (a cell crossing, a
            // wall, a collision event: a few per cent of the particles a step), decided
            // per 32-byte sector (two lanes) so that memory sees whole sectors
            const int chg = moved ? 1 : 0;
            const bool wcell = (chg | __shfl_xor_sync(0xffffffffu, chg, 1)) != 0;
            if (act && todo >= 0) {
                if (wcell)
                    __stcs(reinterpret_cast<int4*>(a.cell + slot), make_int4(c[0], c[1], c[2], c[3]));
                st4(offp + slot, f);
                st4(uxp + slot, ux);
                if (MAG && smag) {
                    st4(uyp + slot, uy);
                    st4(uzp + slot, uz);
                }
            }
        }
        // 6. deposit of the (new) positions; an empty slot has jd < 0 (bit 31 of its word), and
        // so have the quads left to rare_quad
        int jd[4];
        Q qr[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            jd[k] = todo < 0 ? -1 : (int)((uint32_t)c[k] & (kCellMask | 0x80000000u));
            if (kChecked && jd[k] >= 0 && !in_range(a.err, jd[k], 0, a.seg[s].ncells)) jd[k] = -1;
            qr[k] = (Q)Prec<T>::qright(f[k]);
        }
        warp_deposit<Q, MOVE && SUB>(jd, qr, Prec<T>::S,
                                     MOVE && SUB && !moves ? nullptr : a.dep + node0,
                                     a.hist_out ? a.hist_out + node0 : nullptr, dwin);
        if (!FULL && todo != 0) {
            if (todo < 0) rare_quad<T, MAG>(a, s, smag, step, slot);
            else if (MAG) test_quad(a, s, step, slot, todo);
            else test_quad_called(a, s, step, slot, todo);
        }
    }
}

// ---- the step that ends a sort cycle -------------------------------------------------
// Every particle present at the start of the step goes to its slot of the other store
// copy, in the order of a counting sort by its cell at the start of the step (`cursor`:
// each cell's next free slot, from the counts the step before made).  A block works on
// NT/32 consecutive tiles at a time (a chunk of up to 128 NT/32 particles).  When the
// chunk lies in one segment and its particles' start cells span fewer than kSortSpan
// cells (the common case: the store was sorted one cycle ago), the block counts them
// per cell in shared memory, reserves each cell's run with one global atomic per cell,
// stages the moved particles in shared memory in that order and writes every run with
// consecutive threads, so the scattered writes of a sort become coalesced runs of
// about a cell's share of the chunk.  Otherwise (a chunk across two segments, or
// particles spread widely) each warp reserves per cell and quad position and writes
// its particles directly.
constexpr int kSortSpan = 128;

template <typename T, int NT, bool YP>
struct SortSmem {
    static constexpr int NW = NT / 32;
    static constexpr int C = NW * 128;  // particles of a chunk
    // staged particles (off, ux, uy, uz and with YP yp in T; cell word, id; destination
    // in the segment), then the per-cell counts, run offsets in the chunk, global run starts, and
    // the per-warp summaries (segment, lowest and highest start cell) of two consecutive
    // chunks
    static constexpr size_t bytes = (size_t)C * ((YP ? 5 : 4) * sizeof(T) + 4 + 4 + 4) +
                                    (size_t)3 * kSortSpan * 4 + (size_t)2 * 3 * NW * 4;
};

// Resident blocks per SM the sort step is compiled for: registers before warps, since its
// particles keep their velocities, ids and ranks beside the move (FP64 spilled 156 bytes at
// 24 warps and 80 registers: 196.6 M particles 3.79 ms, 3.57 at 20 warps, 3.86 at 16; FP32 at
// 32 warps and 64 registers 2.22, 2.20 at 28, 2.17 at 24; 39 M magnetized 577, 565, 549 us).
// Larger blocks, which nothing but $BITPIC_SORT_BLOCK takes, keep the Boris form's warps.
template <typename T, int NT>
struct SortOccupancy {
    static constexpr int warps = NT != 128 ? MoveOccupancy<T, true, NT>::warps : sizeof(T) == 8 ? 20 : 24;
    static constexpr int blocks = warps / (NT / 32) > 0 ? warps / (NT / 32) : 1;
};

// YP: some species drifts in y (MoveArgs.yp): the y coordinates are sorted with the
// particles (a separate variant: carrying them costs the others registers).
template <typename T, int NT, bool MAG, bool SUB, bool MIXED, bool YP>
__global__ void __launch_bounds__(NT, SortOccupancy<T, NT>::blocks)
k_move_sort(const __grid_constant__ MoveArgs a)
{
    using Q = typename Prec<T>::Q;
    using T2 = typename Prec<T>::T2;
    constexpr int NW = NT / 32, C = NW * 128;
    const unsigned FULL = 0xffffffffu;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T* const s_off = reinterpret_cast<T*>(smem_raw);
    T* const s_ux = s_off + C;
    T* const s_uy = s_ux + C;
    T* const s_uz = s_uy + C;
    T* const s_yp = s_uz + C;  // (only with YP)
    int* const s_cell = reinterpret_cast<int*>(s_yp + (YP ? C : 0));
    uint32_t* const s_id = reinterpret_cast<uint32_t*>(s_cell + C);
    uint32_t* const s_dst = s_id + C;
    int* const cnt = reinterpret_cast<int*>(s_dst + C);
    int* const pre = cnt + kSortSpan;
    unsigned* const gb = reinterpret_cast<unsigned*>(pre + kSortSpan);
    // per-warp summaries, double-buffered by chunk parity: a warp may write the next
    // chunk's entry while another still reads this chunk's (the next chunk's first
    // barrier keeps it from getting further ahead)
    int* const wsum = reinterpret_cast<int*>(gb + kSortSpan);

    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned lt = (1u << lane) - 1u;
    // the warps' deposit windows and (FP64) scratch of add_crossed
    __shared__ __align__(16) uint32_t s_dwin[NW][DepWin<Q>::words + CrossScratch<T>::words];
    uint32_t* const dwin = s_dwin[warp];
    double* const scr = reinterpret_cast<double*>(dwin + DepWin<Q>::words);
    dep_win_clear<Q>(dwin);
    T* const offp = static_cast<T*>(a.off);
    T* const uxp = static_cast<T*>(a.ux);
    T* const uyp = static_cast<T*>(a.uy);
    T* const uzp = static_cast<T*>(a.uz);
    const int64_t step = a.step[1];
    if (blockIdx.x == 0 && threadIdx.x == 0) a.step[0] = step;
    const int64_t total = a.tile_start[a.nseg];
    int s = 0;
    int64_t s_begin = 0, s_end = -1;
    bool moves = true, smag = MAG;
    SegFast F = {0, 0u, 0u, false};
    // every warp of the block walks the same chunks, so the barriers below match
    int parity = 0;
    int64_t chunk = (int64_t)blockIdx.x * a.chunk;
    for (int left = a.chunk; chunk * NW < total; parity ^= 1) {
        int* const wseg = wsum + parity * 3 * NW;
        int* const wmin = wseg + NW;
        int* const wmax = wmin + NW;
        const int64_t tile = chunk * NW + warp;
        const bool have = tile < total;
        if (have && tile >= s_end) {
            s = advance_segment(a.tile_start, a.nseg, s, tile);
            s_begin = __ldg(a.tile_start + s);
            s_end = __ldg(a.tile_start + s + 1);
            if (MAG && MIXED) smag = a.seg[s].mag != 0;
            if (SUB) moves = moves_on(a.seg[s], step);
            int64_t mown;
            int dgrid;
            own_time(a.seg[s], step, mown, dgrid);
            F.set(a.seg[s], mown);
        }
        const SegParams& P = a.seg[s];
        const int64_t quad = (tile - s_begin) * 32 + lane;
        const int64_t slot = P.base + 4 * quad;
        const bool act = have && quad < (a.seg_nmove[s] >> 2) &&
                         in_range(a.err, slot + 3, P.base, P.base + P.cap);

        int c[4] = {-1, -1, -1, -1};
        T f[4] = {T(0), T(0), T(0), T(0)}, ux[4] = {T(0), T(0), T(0), T(0)};
        T uy[4] = {T(0), T(0), T(0), T(0)}, uz[4] = {T(0), T(0), T(0), T(0)};
        uint32_t idq[4] = {0u, 0u, 0u, 0u};
        if (act) {
            const int4 cc = __ldcs(reinterpret_cast<const int4*>(a.cell + slot));
            c[0] = cc.x; c[1] = cc.y; c[2] = cc.z; c[3] = cc.w;
            ld4(offp + slot, f);
            ld4(uxp + slot, ux);
            ld4(uyp + slot, uy);
            ld4(uzp + slot, uz);
            const uint4 ii = __ldcs(reinterpret_cast<const uint4*>(a.id + slot));
            idq[0] = ii.x; idq[1] = ii.y; idq[2] = ii.z; idq[3] = ii.w;
        }
        // start cells of the quad (-1: empty slot); the chunk's span and segments
        int j0[4];
        unsigned lmin = 0xFFFFFFFFu;
        int lmax = -1;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            j0[k] = c[k] >= 0 ? (int)((uint32_t)c[k] & kCellMask) : -1;
            if (j0[k] >= 0 && !in_range(a.err, j0[k], 0, P.ncells)) {  // (checked build)
                j0[k] = -1;
                c[k] = -1;
            }
            if (j0[k] >= 0) {
                lmin = min(lmin, (unsigned)j0[k]);
                lmax = max(lmax, j0[k]);
            }
        }
        const unsigned wmn = __reduce_min_sync(FULL, lmin);
        const int wmx = __reduce_max_sync(FULL, lmax);
        if (lane == 0) {
            wseg[warp] = wmx >= 0 ? s : -1;
            wmin[warp] = (int)wmn;
            wmax[warp] = wmx;
        }
        for (int i = threadIdx.x; i < kSortSpan; i += NT) cnt[i] = 0;
        __syncthreads();
        // the chunk's segment (one if every warp's live particles are in the same one)
        // and its span of start cells, from the per-warp summaries
        int bseg, bmin, bmax;
        bool one;
        {
            const int ws = lane < NW ? wseg[lane] : -1;
            const int mn = ws >= 0 ? wmin[lane] : INT_MAX;
            const int mx = ws >= 0 ? wmax[lane] : -1;
            const int smax = __reduce_max_sync(FULL, ws);
            const int smin = __reduce_min_sync(FULL, ws >= 0 ? ws : INT_MAX);
            bseg = smax;
            one = smax < 0 || smin == smax;
            bmin = __reduce_min_sync(FULL, mn);
            bmax = __reduce_max_sync(FULL, mx);
        }
        const bool staged = one && bseg >= 0 && bmax - bmin < kSortSpan;
        bool moved = false;
        int ev = 0;  // -1: a quad the common path left, else see quad_due
        const T2* const accn = static_cast<const T2*>(a.accel) + P.node;
        if (staged) {
            const SegParams& B = a.seg[bseg];
            // rank of each particle among the chunk's particles of its start cell: equal
            // cells of a quad position grouped across the warp, one shared atomic a group
            int key[4], rank[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                key[k] = j0[k] >= 0 ? j0[k] - bmin : -1;
                const unsigned grp = __match_any_sync(FULL, key[k] >= 0 ? key[k] : kSortSpan + lane);
                const int leader = __ffs(grp) - 1;
                int base = 0;
                if (key[k] >= 0 && lane == leader) base = atomicAdd(cnt + key[k], __popc(grp));
                base = __shfl_sync(FULL, base, leader);
                rank[k] = base + __popc(grp & lt);
            }
            __syncthreads();
            // each cell's run: its offset in the chunk (scan of the counts) and its global
            // start (one reservation per cell, waited for only after the move)
            unsigned gres = 0;
            if (threadIdx.x < kSortSpan) {
                const int n = cnt[threadIdx.x];
                if (n > 0) gres = atomicAdd(a.cursor + B.node + bmin + threadIdx.x, (unsigned)n);
            }
            if (warp == 0) {
                int v[kSortSpan / 32], sum = 0;
#pragma unroll
                for (int i = 0; i < kSortSpan / 32; ++i) {
                    v[i] = cnt[lane * (kSortSpan / 32) + i];
                    sum += v[i];
                }
                int inc = sum;
#pragma unroll
                for (int d = 1; d < 32; d <<= 1) {
                    const int t = __shfl_up_sync(FULL, inc, d);
                    if (lane >= d) inc += t;
                }
                int run = inc - sum;
#pragma unroll
                for (int i = 0; i < kSortSpan / 32; ++i) {
                    pre[lane * (kSortSpan / 32) + i] = run;
                    run += v[i];
                }
            }
            if (!SUB || moves) {
                bool due;
                int walls = 0;
                const bool rare = quad_fast<T, MAG>(P, F, smag, accn, c, f, ux, uy, uz, moved, due, walls, scr);
                if (rare && act) ev = -1;
                if (due && act && !rare) ev = quad_due(F, c);
            }
            if (threadIdx.x < kSortSpan) gb[threadIdx.x] = gres;
            __syncthreads();
            // stage every particle at its place in the chunk's cell order; a quad the
            // common path left is staged where it lay and put right below
            int pk[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                pk[k] = -1;
                if (key[k] < 0) continue;
                const int p = pre[key[k]] + rank[k];
                if (!in_range(a.err, p, 0, C)) continue;  // (bounds-checked build only)
                pk[k] = p;
                s_off[p] = f[k];
                s_ux[p] = ux[k];
                s_uy[p] = uy[k];
                s_uz[p] = uz[k];
                s_cell[p] = c[k];
                s_id[p] = idq[k];
                if (YP) s_yp[p] = static_cast<const T*>(a.yp)[slot + k];
                const int64_t r = (int64_t)gb[key[k]] + rank[k];
                s_dst[p] = r < B.cap ? (uint32_t)r : 0xFFFFFFFFu;
                if (ev > 0 && (ev >> k & 1) && r < B.cap) queue_rare(a, bseg, B.base + r, kRareCandidate);
            }
            if (ev > 15)
                test_staged(a, bseg, step, ev,
                            make_short4((short)pk[0], (short)pk[1], (short)pk[2], (short)pk[3]), s_cell,
                            s_id, s_dst);
            if (ev < 0) {
                int64_t mown;
                int dgrid;
                own_time(B, step, mown, dgrid);
#pragma unroll 1
                for (int k = 0; k < 4; ++k) {
                    const int p = k == 0 ? pk[0] : k == 1 ? pk[1] : k == 2 ? pk[2] : pk[3];
                    if (p < 0) continue;
                    int ck = a.cell[slot + k];
                    T fk, xk, yk = s_uy[p], zk = s_uz[p];
                    const uint32_t d = s_dst[p];
                    rare_particle<T, MAG>(a, B, bseg, smag, step, mown, dgrid, slot + k,
                                          d == 0xFFFFFFFFu ? (int64_t)-1 : B.base + (int64_t)d, ck,
                                          fk, xk, yk, zk);
                    s_cell[p] = ck;
                    s_off[p] = fk;
                    s_ux[p] = xk;
                    if (MAG && smag) {
                        s_uy[p] = yk;
                        s_uz[p] = zk;
                    }
                }
            }
            // (read before the barrier: the next chunk clears the counts after it)
            const int ntot = pre[kSortSpan - 1] + cnt[kSortSpan - 1];
            __syncthreads();
            // write the runs: consecutive threads, consecutive slots of a cell's run
            T* const doff = static_cast<T*>(a.doff);
            T* const dux = static_cast<T*>(a.dux);
            T* const duy = static_cast<T*>(a.duy);
            T* const duz = static_cast<T*>(a.duz);
#pragma unroll 4
            for (int p = threadIdx.x; p < ntot; p += NT) {
                const uint32_t r = s_dst[p];
                if (r == 0xFFFFFFFFu) {  // a histogram that does not match the store: refused
                    set_error(a.err, kErrCapacity);
                    continue;
                }
                const int64_t g = B.base + (int64_t)r;
                __stcs(a.dcell + g, s_cell[p]);
                __stcs(doff + g, s_off[p]);
                __stcs(dux + g, s_ux[p]);
                __stcs(duy + g, s_uy[p]);
                __stcs(duz + g, s_uz[p]);
                __stcs(a.did + g, s_id[p]);
                if (YP) static_cast<T*>(a.dyp)[g] = s_yp[p];
            }
        } else {
            // per warp: reserve each particle's slot by its start cell (equal cells of a
            // quad position grouped across the warp, one counter update per group)
            unsigned grp[4] = {0u, 0u, 0u, 0u}, rbase[4] = {0u, 0u, 0u, 0u}, had = 0u;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int kk = j0[k] >= 0 ? j0[k] : -1 - lane;
                grp[k] = __match_any_sync(FULL, kk);
                if (j0[k] >= 0) had |= 1u << k;
                if (j0[k] >= 0 && lane == __ffs(grp[k]) - 1)
                    rbase[k] = atomicAdd(a.cursor + P.node + kk, (unsigned)__popc(grp[k]));
            }
            if (!SUB || moves) {
                bool due;
                int walls = 0;
                const bool rare = quad_fast<T, MAG>(P, F, smag, accn, c, f, ux, uy, uz, moved, due, walls, scr);
                if (rare && act) ev = -1;
                if (due && act && !rare) ev = quad_due(F, c);
            }
            int64_t to[4];
            sort_destinations(a, P, grp, rbase, had, to);
            sort_write<T>(a, to, c, f, ux, uy, uz, idq);
            if (YP) {  // the y coordinates go along
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    if (to[k] >= 0)
                        static_cast<T*>(a.dyp)[to[k]] = static_cast<const T*>(a.yp)[slot + k];
            }
            if (ev > 0) {
                int64_t mown;
                int dgrid;
                own_time(P, step, mown, dgrid);
#pragma unroll 1
                for (int k = 0; k < 4; ++k) {
                    const int64_t g = k == 0 ? to[0] : k == 1 ? to[1] : k == 2 ? to[2] : to[3];
                    if (g < 0) continue;
                    if (ev >> k & 1) queue_rare(a, s, g, kRareCandidate);
                    if (ev >> k & 16)
                        a.dcell[g] = test_clock(a, P, s, step, mown, dgrid,
                                                k == 0 ? idq[0] : k == 1 ? idq[1] : k == 2 ? idq[2] : idq[3],
                                                k == 0 ? c[0] : k == 1 ? c[1] : k == 2 ? c[2] : c[3], g);
                }
            }
            if (ev < 0) {
                // put right what the common path left, in the slots just written
                int64_t mown;
                int dgrid;
                own_time(P, step, mown, dgrid);
#pragma unroll 1
                for (int k = 0; k < 4; ++k) {
                    const int64_t g = k == 0 ? to[0] : k == 1 ? to[1] : k == 2 ? to[2] : to[3];
                    int ck = a.cell[slot + k];
                    if (ck < 0) continue;
                    T fk, xk, yk = T(0), zk = T(0);
                    rare_particle<T, MAG>(a, P, s, smag, step, mown, dgrid, slot + k, g, ck, fk, xk,
                                          yk, zk);
                    if (g < 0) continue;
                    a.dcell[g] = ck;
                    static_cast<T*>(a.doff)[g] = fk;
                    static_cast<T*>(a.dux)[g] = xk;
                    if (MAG && smag) {
                        static_cast<T*>(a.duy)[g] = yk;
                        static_cast<T*>(a.duz)[g] = zk;
                    }
                }
            }
        }
        // 6. deposit of the new positions (that of a segment that rests stands)
        ++chunk;
        if (--left == 0) {  // on to the block's next rounds
            left = a.chunk;
            chunk += (int64_t)(gridDim.x - 1) * a.chunk;
        }
        if (SUB && !moves) continue;
        int jd[4];
        Q qr[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            jd[k] = ev < 0 ? -1 : (int)((uint32_t)c[k] & (kCellMask | 0x80000000u));
            if (kChecked && jd[k] >= 0 && !in_range(a.err, jd[k], 0, P.ncells)) jd[k] = -1;
            qr[k] = (Q)Prec<T>::qright(f[k]);
        }
        warp_deposit<Q>(jd, qr, Prec<T>::S, a.dep + P.node, nullptr, dwin);
    }
}

// Host side of k_move_sort: the launch with its shared memory, and the set-up of every
// variant (the dynamic shared-memory limit, needed above 48 KB) with the occupancy the
// grid is sized by.  The set-up runs when the handle sizes its grids, outside any
// stream capture.
template <typename T, int NT, bool MAG, bool SUB, bool MIXED, bool YP>
inline cudaError_t launch_sort_variant(const MoveArgs& a, int grid, cudaStream_t st)
{
    k_move_sort<T, NT, MAG, SUB, MIXED, YP><<<grid, NT, SortSmem<T, NT, YP>::bytes, st>>>(a);
    return cudaGetLastError();
}

template <typename T, int NT, bool YP>
inline cudaError_t launch_sort_step_yp(const MoveArgs& a, bool mag, bool sub, bool mixed,
                                       int grid, cudaStream_t st)
{
    if (!mag)
        return sub ? launch_sort_variant<T, NT, false, true, false, YP>(a, grid, st)
                   : launch_sort_variant<T, NT, false, false, false, YP>(a, grid, st);
    if (mixed)
        return sub ? launch_sort_variant<T, NT, true, true, true, YP>(a, grid, st)
                   : launch_sort_variant<T, NT, true, false, true, YP>(a, grid, st);
    return sub ? launch_sort_variant<T, NT, true, true, false, YP>(a, grid, st)
               : launch_sort_variant<T, NT, true, false, false, YP>(a, grid, st);
}

template <typename T, int NT>
inline cudaError_t launch_sort_step(const MoveArgs& a, bool mag, bool sub, bool mixed, int grid,
                                    cudaStream_t st)
{
    return a.yp ? launch_sort_step_yp<T, NT, true>(a, mag, sub, mixed, grid, st)
                : launch_sort_step_yp<T, NT, false>(a, mag, sub, mixed, grid, st);
}

template <typename T, int NT, bool YP>
inline cudaError_t sort_step_setup(int* blocks_mag, int* blocks_plain)
{
    const int sm = (int)SortSmem<T, NT, YP>::bytes;
    const cudaFuncAttribute A = cudaFuncAttributeMaxDynamicSharedMemorySize;
    cudaError_t e = cudaFuncSetAttribute(k_move_sort<T, NT, false, false, false, YP>, A, sm);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_move_sort<T, NT, false, true, false, YP>, A, sm);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_move_sort<T, NT, true, false, false, YP>, A, sm);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_move_sort<T, NT, true, true, false, YP>, A, sm);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_move_sort<T, NT, true, false, true, YP>, A, sm);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_move_sort<T, NT, true, true, true, YP>, A, sm);
    if (e == cudaSuccess)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_mag, k_move_sort<T, NT, true, false, false, YP>, NT, sm);
    if (e == cudaSuccess)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_plain, k_move_sort<T, NT, false, false, false, YP>, NT, sm);
    return e;
}

// Blocks per SM the sort-step grid is sized by (YP: the variant with the y coordinates,
// launched when some species drifts in y; it holds more shared memory).
template <typename T, int NT>
inline int sort_step_blocks_per_sm(bool mag, bool yp)
{
    int m = 0, p = 0;
    const cudaError_t e = yp ? sort_step_setup<T, NT, true>(&m, &p) : sort_step_setup<T, NT, false>(&m, &p);
    if (e != cudaSuccess) return 0;
    return mag ? m : p;
}

}  // namespace bitpic
