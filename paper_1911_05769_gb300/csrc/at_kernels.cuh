// at_kernels.cuh -- persistent weakly-synchronous AT stepper for sm_103a.
//
// One cooperative launch advances the whole 1D field by n_steps forward-Euler
// steps (arXiv 1911.05769, Sec. 3.2).  Every warp of the launch is one
// processing element (PE) of the paper: PE e owns the contiguous subdomains
// [lo, hi) and sweeps them in pass-major order.  A "tile" is one subdomain j
// over one pass of `len` consecutive levels n .. n+len (len = 1 except in
// blocked free-running mode).  For each tile the PE
//   * has already copied the subdomain's M state words into one of its
//     shared-memory stages (16-byte asynchronous copies, D tiles ahead);
//   * has already read the neighbours' delayed boundary values (levels n-k-m,
//     Eq. AT1/AT2) from the ring buffers, one tile ahead.  Every ring entry
//     carries the level it holds, so what is not there yet shows by itself and
//     is read again when the tile is reached: the blocking branch of
//     Algorithm 2.  Free running, the delay k is what the entries show: the
//     newest level the neighbour has published, at most L behind;
//   * approximates the halo values ("approximate" step of Algorithm 2, split
//     form of Sec. 5.2), applies the unchanged central stencil of order 2 or
//     4 and the Euler update `len` times on the tile held in registers
//     (neighbour values by warp shuffles), and writes the final level back in
//     place;
//   * after every level writes the new boundary values, with their level, into
//     ring slot (level mod T) (the notified put: data and notification are one
//     16-byte store).
// Halo values never come from a neighbour's state array, only from the ring,
// so each PE updates its own subdomains in place, and a PE never waits for
// another PE of its CTA except through the same entries.
//
// Blocked free-running mode (temporal blocking): a pass of len <= L+1 levels
// uses, at inner step i, the halo extrapolated with delay k0 + i from the
// levels available when the pass started (Eq. AT1/AT2 with a larger k), so
// the state is read and written once per pass instead of once per level.
//
// AT_SYNC puts a grid barrier between steps (Algorithm 1).  Every wait is
// bounded by timeout_ns; on expiry the kernel latches AT_ERR_TIMEOUT in the
// control block, raises the abort word and every PE leaves its loop (after
// its copies in flight have landed).
#pragma once

#include "at_device.cuh"

// Minimum resident CTAs per SM the stepper is compiled for (register cap).
#ifndef AT_MIN_CTAS_PER_SM
#define AT_MIN_CTAS_PER_SM 3
#endif

namespace atk {

constexpr int kWarps = 4;                         // PEs (warps) per CTA
constexpr int kThreads = 32 * kWarps;
constexpr int kRingHalf = 16;                     // bytes of a half of a ring entry: 8 of payload, 8 of level tag
constexpr int kMaxS = 3;                          // levels per halo approximation
constexpr int kStripBytes = 64;                  // blocked synchronous mode: edge strip per (subdomain, face)
constexpr int kRawEntry = 16;                     // payload of one ring entry in shared memory
constexpr int kRawFace = 64;                      // per face: kMaxS of them
constexpr int kRawBytes = 2 * kRawFace;           // one tile's delayed levels [face][m]
constexpr int kMaxM = 1024;                       // points per subdomain (one warp's tile)
constexpr int kMaxL = 16;
constexpr int kMinStages = 2;                     // stages per PE (tile in use + one ahead)

enum : int { kModeSync = 0, kModeSeeded = 1, kModeFree = 2, kModeReplay = 3 };

// Shared-memory layout of one CTA, shared by the host (launch set-up) and the
// kernel: per PE a raw-level buffer and `stages` tile buffers;
// then a table of `tab_bytes`: the forcing tables (sin/cos of the offsets in a
// subdomain, and of each PE's subdomain origins) or, for an ensemble, each
// PE's subdomain records.  M: points of a tile buffer (tile_points()).
struct SmemLayout {
    long long raw_off, stage_off, stage_bytes, tab_off, total;
};

__host__ __device__ inline long long round_up(long long x, long long a) { return (x + a - 1) / a * a; }

// Points of a tile buffer and of a forcing table for tiles of M points in
// lanes of gw whole groups (all 32 of them: lanes beyond the tile then need no
// guard) or, runs not full, of M points.
__host__ __device__ inline long long tile_points(long long M, int gw, bool full)
{
    return full ? 128LL * gw : round_up(M, 32);
}

__host__ __device__ inline SmemLayout smem_layout(long long M, int word, int stages, long long tab_bytes, bool comp = false)
{
    SmemLayout l;
    l.raw_off = 0;
    l.stage_off = round_up(l.raw_off + (long long)kWarps * kRawBytes, 128);
    l.stage_bytes = round_up(M * word, 128) * (comp ? 2 : 1);     // tile (+ its error words)
    l.tab_off = l.stage_off + (long long)kWarps * stages * l.stage_bytes;
    l.total = l.tab_off + tab_bytes;
    return l;
}

// Place of 16-byte chunk c of a tile in its stage (and of the forcing tables):
// a lane reads cpl consecutive chunks, so with cpl = 2, 4, 8 the 8 lanes that
// share a shared-memory cycle would meet in the same banks cpl at a time;
// exchanging chunks within blocks of 8 by the block's number spreads them, and
// leaves the coalesced side (consecutive lanes, consecutive chunks) conflict-free.
// An odd cpl has no conflicts, other even ones two-way ones.
struct Swizzle {
    int shift, mask;
    __host__ __device__ static constexpr Swizzle of(int cpl)
    {
        return cpl == 16 ? Swizzle{4, 7} : (cpl == 2 || cpl == 4 || cpl == 8) ? Swizzle{3, cpl - 1} : Swizzle{0, 0};
    }
    __host__ __device__ constexpr int operator()(int c) const { return c ^ ((c >> shift) & mask); }
    // byte offsets in the stage of chunk lane + 32 t (the coalesced side)
    __device__ __forceinline__ int coalesced(int lane, int t) const
    {
        return 512 * t + (((lane ^ ((lane >> shift) & mask)) << 4) ^ ((((32 * t) >> shift) & mask) << 4));
    }
};

// byte offset in the stage of chunk k of a lane that holds CPL whole chunks
template <int CPL>
__device__ __forceinline__ int lane_chunk(int lane, int k)
{
    const int lx = CPL == 16 ? lane & 7 : ((lane * CPL) >> 3) & (CPL - 1);
    return ((16 * CPL * lane) | (lx << 4)) ^ (k << 4);
}

// A ring entry holds one face's R boundary words of one level (a compensated
// state: R hi, then R lo words) in one or two halves of 16 bytes: 8 bytes of
// payload and the level's tag.  A half is written and read as one 16-byte
// access, so the words and their tag arrive together.
template <typename T, int ORDER, int PREC>
__host__ __device__ constexpr int entry_halves()
{
    return (int)sizeof(T) * (ORDER / 2) * (PREC == 2 ? 2 : 1) > 8 ? 2 : 1;
}

// Tag of a level (0, the cleared ring, is no level's).
__host__ __device__ inline unsigned long long entry_tag(long long level) { return (unsigned long long)(level + 1); }

// Ensembles: independent 1D problems of M-point subdomains laid end to end.
// One record per subdomain (built on the host, copied to shared memory by the
// PE that owns it) and one per problem instance.
struct BatchSub {
    double cA, cr;             // stencil factors of the instance (as Params::cA, cr)
    unsigned long long seed;   // AT_SEEDED seed of the instance
    int L;                     // delay bound of the instance
    int lp;                    // index of the subdomain within its instance
    int Pi;                    // subdomains of the instance
    int inst;                  // instance
    long long left, right;     // global subdomain across face 0 / 1; -1 = exact boundary
    float cA32, cr32;          // cA, cr in FP32
};
static_assert(sizeof(BatchSub) == 64, "BatchSub is four 16-byte vectors");

struct BatchInst {
    double x0, dx, dt, nu;     // grid x_i = x0 + i dx of the instance, time step, viscosity
    double ta, tc, txc;        // exact boundary values u = c - a tanh(a (x - xc - c t) / (2 nu))
    double pad_;
};
static_assert(sizeof(BatchInst) == 64, "BatchInst is 64 bytes");

// A tile of an ensemble launch: cnt consecutive subdomains s0 ..
// s0+cnt-1 of one instance, advanced together (the faces between them at
// delay 0: the neighbour's level itself).  Tiles are listed in the order the
// processing elements sweep them (instances grouped by delay bound); rec is
// the place of s0 in the list's enumeration of subdomains, which orders the
// subdomain records in shared memory.  link bit 0: the left neighbour of s0
// is the last subdomain of the previous tile of the list; bit 1: the right
// neighbour of the last subdomain is s0 of the next tile.  Stored as an int4
// (s0, rec, cnt | link << 16, 0).
struct TileInfo {
    int s0, rec, cnt, link;
};

// Ensembles in passes of several levels: the CTAs from cta[g] to cta[g + 1] own
// the tiles from tile[g] to tile[g + 1], whose instances have one pass length
// (0 groups: all CTAs own all tiles).
struct TileSplit {
    int groups;
    int cta[kMaxL + 2];
    long long tile[kMaxL + 2];
};

struct Params {
    void *u;                   // state, N words, updated in place
    unsigned char *ring;       // [T][P][2] entries (see entry_halves)
    int *ctrl;                 // control block (status, abort, diagnostics)
    unsigned long long *hist;  // [L+1] delay counts
    unsigned long long *gbar;  // grid-barrier arrival counter (AT_SYNC)
    int8_t *delays;            // [n_steps][P][2] replay input / record output
    const BatchSub *bsub;      // ensembles: [P] subdomain records (else NULL)
    const BatchInst *binst;    // ensembles: instance records (else NULL)
    const int4 *tiles;         // ensembles: the launch's tile list [ntiles] (see TileInfo)
    const int *sub_order;      // ensembles: subdomain at each place of the tile lists' enumeration [P]
    TileSplit split;
    long long ntiles;          // tiles of the launch (single domain: P, tile j = subdomain j)
    void *ur;                  // compensated state: the rounding error of every point (N words)
    unsigned char *strip;      // blocked synchronous mode: edge strips [2][P][2] of kStripBytes (pass parity)
    int strip_words;           // words per strip (R x levels per pass, rounded up to a multiple of 4)
    void *levels;              // optional copy of every level l computed: slot l mod levels_depth of N words
    long long levels_depth;    // (single-level passes only; the adjoint's recomputation)
    long long N, P, M;
    int L, T, mode, per_sub;   // L: largest delay bound (ensembles: of any instance)
    long long n_steps;
    int sb;                    // most levels per pass (temporal blocking: free mode, and the blocked
                               // synchronous mode, where k = 0 and the ghost cells are recomputed)
    unsigned long long seed;
    double cA, cB, cr;         // dt/(2dx) | dt/(12dx);  nu dt/dx^2 | nu dt/(12dx^2);  cB / cA
    double fX;                 // forcing factor: A dt (FP64 viscous term), else A dt / cA
    float cA32, cB32, cr32, fX32;   // the same in FP32 (no conversion per tile)
    double x0, dx;
    int G;                     // CTAs
    int nh;                    // halves of an entry
    int stages;                // tile buffers per PE
    int gpl;                   // groups of 4 points per lane
    int swz_shift, swz_mask;   // place of a tile's chunks in its stage (see Swizzle)
    long long smax;            // most subdomains of any PE
    int stage_bytes;           // bytes of a stage (compensated state: its second half holds the lo words)
    int tab_words;             // words of a forcing table (M, padded)
    long long raw_off, stage_off, tab_off;
    long long timeout_ns;
    int skip_publish;          // test knob: the first tile's PE stops publishing
    long long skip_step;
};

// ---------------------------------------------------------------------------
// bounded waits
// ---------------------------------------------------------------------------
static __device__ __noinline__ void raise_timeout(const Params &p, int where, long long n, long long nb)
{
    if (atomicCAS(p.ctrl + kCtrlStatus, 0, kStatusTimeout) == 0) {
        p.ctrl[kCtrlCta] = (int)blockIdx.x;
        p.ctrl[kCtrlWhere] = where;
        p.ctrl[kCtrlNb] = (int)nb;
        p.ctrl[kCtrlStep] = (int)n;
    }
    atomicExch(p.ctrl + kCtrlAbort, 1);
}

static __device__ __noinline__ bool wait_grid(const Params &p, unsigned long long target, long long n)
{
    if (ld_acquire(p.gbar) >= target) return true;
    const unsigned long long t0 = global_ns();
    for (;;) {
        __nanosleep(20);
        if (ld_acquire(p.gbar) >= target) return true;
        if (ld_relaxed(p.ctrl + kCtrlAbort)) return false;
        if ((long long)(global_ns() - t0) > p.timeout_ns) {
            raise_timeout(p, kWhereGrid, n, -1);
            return false;
        }
    }
}

// ---------------------------------------------------------------------------
// shared-memory vector access
// ---------------------------------------------------------------------------
template <typename T, int CNT>
__device__ __forceinline__ void lds(const T *s, T *v)
{
    if constexpr (sizeof(T) == 4 && CNT == 4) {
        const float4 a = *reinterpret_cast<const float4 *>(s);
        v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
    } else if constexpr (sizeof(T) == 4 && CNT == 2) {
        const float2 a = *reinterpret_cast<const float2 *>(s);
        v[0] = a.x; v[1] = a.y;
    } else if constexpr (sizeof(T) == 8 && CNT == 4) {
        const double2 a = *reinterpret_cast<const double2 *>(s);
        const double2 b = *reinterpret_cast<const double2 *>(s + 2);
        v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
    } else if constexpr (sizeof(T) == 8 && CNT == 2) {
        const double2 a = *reinterpret_cast<const double2 *>(s);
        v[0] = a.x; v[1] = a.y;
    } else {
#pragma unroll
        for (int i = 0; i < CNT; ++i) v[i] = s[i];
    }
}

template <typename T>
__device__ __forceinline__ void sts4(T *s, const T *v)
{
    if constexpr (sizeof(T) == 4) {
        *reinterpret_cast<float4 *>(s) = make_float4(v[0], v[1], v[2], v[3]);
    } else {
        *reinterpret_cast<double2 *>(s) = make_double2(v[0], v[1]);
        *reinterpret_cast<double2 *>(s + 2) = make_double2(v[2], v[3]);
    }
}

// one 16-byte chunk (4 floats or 2 doubles)
template <typename T, int CNT>
__device__ __forceinline__ void stsv(T *s, const T *v)
{
    if constexpr (sizeof(T) == 4) *reinterpret_cast<float4 *>(s) = make_float4(v[0], v[1], v[2], v[3]);
    else *reinterpret_cast<double2 *>(s) = make_double2(v[0], v[1]);
}

// 4 consecutive words to global memory (16-byte aligned), bypassing L1.
template <typename T>
__device__ __forceinline__ void stg4(T *g, const T *v)
{
    if constexpr (sizeof(T) == 4) {
        st_cg16(g, v[0], v[1], v[2], v[3]);
    } else {
        st_cg16(g, v[0], v[1]);
        st_cg16(g + 2, v[2], v[3]);
    }
}

// One ring entry: R words v (compensated state: and their lo words l) with the
// level's tag in every half (`on`: predicate).
template <typename T, int ORDER, int PREC>
__device__ __forceinline__ void st_entry(bool on, unsigned char *e, const T *v, const T *l, unsigned long long tag)
{
    constexpr int R = ORDER / 2;
    auto two = [](T a, T b) -> unsigned long long {
        return ((unsigned long long)__float_as_uint((float)b) << 32) | __float_as_uint((float)a);
    };
    if constexpr (sizeof(T) == 8) {
#pragma unroll
        for (int q = 0; q < R; ++q)
            st_tagged(on, e + q * kRingHalf, (unsigned long long)__double_as_longlong((double)v[q]), tag);
    } else if constexpr (PREC == 2 && R == 2) {
        st_tagged(on, e, two(v[0], v[1]), tag);
        st_tagged(on, e + kRingHalf, two(l[0], l[1]), tag);
    } else if constexpr (PREC == 2) {
        st_tagged(on, e, two(v[0], l[0]), tag);
    } else {
        st_tagged(on, e, two(v[0], R > 1 ? v[R - 1] : (T)0), tag);
    }
}

// Halo approximation from s delayed levels raw[m] = f^{n-k-m} (16-byte
// entries, word r of each): Lagrange extrapolation in time to level n.
// s = 2 gives (k+1) f^{n-k} - k f^{n-k-1} (Eq. AT1/AT2); s = 3 uses the
// quadratic through n-k, n-k-1, n-k-2.  k = 0 returns f^n itself.  Evaluated
// in Newton form, f0 + k d1 (+ k(k+1)/2 d2) with the backward differences
// d1 = f0 - f1, d2 = d1 - (f1 - f2): the same polynomial, but the
// differences of nearby levels are exact in floating point, so the rounding
// error stays about one ulp of f0 instead of growing with the weights
// (10, -15, 6 at k = 3).
template <typename T, int S_LEV>
__device__ __forceinline__ T approx_halo(const unsigned char *raw, int k, int r)
{
    const T r0 = reinterpret_cast<const T *>(raw)[r];
    if (k == 0) return r0;
    const T r1 = reinterpret_cast<const T *>(raw + kRawEntry)[r];
    const T d1 = r0 - r1;
    if constexpr (S_LEV == 2) {
        return r0 + (T)k * d1;
    } else {
        const T r2 = reinterpret_cast<const T *>(raw + 2 * kRawEntry)[r];
        const T d2 = d1 - (r1 - r2);
        return r0 + ((T)k * d1 + (T)(k * (k + 1) / 2) * d2);
    }
}

// Compensated state (PREC 2: a value is the pair hi + lo of FP32 words; ring
// entries hold the R hi words, then the R lo words): the halo value's hi word
// is the newest delayed level's hi word f0, and its lo word carries the rest
// of the same extrapolation in Newton form, f0 + k d1 (+ k(k+1)/2 d2 for
// s = 3), the backward differences d1, d2 formed word by word (differences of
// nearby hi words are exact), so that no part of the value is lost to the
// rounding of a single FP32 word.
template <typename T, int S_LEV, int R>
__device__ __forceinline__ T approx_halo_lo(const unsigned char *raw, int k, int r)
{
    const T *e0 = reinterpret_cast<const T *>(raw);
    const T h0 = e0[r], l0 = e0[R + r];
    if (k == 0) return l0;
    const T *e1 = reinterpret_cast<const T *>(raw + kRawEntry);
    const T h1 = e1[r], l1 = e1[R + r];
    const T d1 = (h0 - h1) + (l0 - l1);
    if constexpr (S_LEV == 2) {
        return l0 + (T)k * d1;
    } else {
        const T *e2 = reinterpret_cast<const T *>(raw + 2 * kRawEntry);
        const T h2 = e2[r], l2 = e2[R + r];
        const T d2 = ((h0 - h1) - (h1 - h2)) + ((l0 - l1) - (l1 - l2));
        return l0 + (T)k * d1 + (T)(k * (k + 1) / 2) * d2;
    }
}

// A dt sin x (scaled) of one point from the factors of its subdomain and of its
// offset: fs = f sin x_j, fc = f cos x_j, sv/cv = sin/cos of the offset.
template <typename T>
__device__ __forceinline__ T forcing_point(T fs, T fc, T sv, T cv)
{
    return fma(fc, sv, fs * cv);
}

// The forward-Euler update u += dt (-u u_x + nu u_xx) + F of a run of points,
// as u += cA (cr b - u a + F / cA): cA = dt/(2dx) | dt/(12dx), cA cr = nu
// dt/dx^2 | nu dt/(12dx^2), a and b the stencil's first and second difference,
// a = 8 (u_1 - u_-1) - (u_2 - u_-2), b = 16 (u_1 + u_-1) - (u_2 + u_-2) - 30 u
// at order 4.  The factors 1, cr, cA each ride in a fused multiply-add, so the
// increment, formed apart from u, takes 3 operations beside a and b (6 when cB
// b - cA u a + F + u is taken term by term): 10 a point at order 4, forcing
// included, 6 at order 2.  (Forming a and b from differences shared between
// points takes as many.  In FP32 it loses: there the last addition's rounding
// decides, and over runs of hundreds of steps the sums' own rounding breaks up
// its bias -- error against 64 bits 2.2e-6 against 2.9e-6 with exact differences.)
//   Compensated state: the differences word by word, first differences d_i = u_{i+1}
// - u_i and second ones e_i = d_i - d_{i-1} formed once for the points that share
// them: a = 6 (d_i + d_{i-1}) - (e_{i+1} - e_{i-1}), b = 14 e_i - (e_{i+1} + e_{i-1}).
// Those of the hi words are exact, and stay apart from those of the lo words until the
// last fused multiply-adds (joined before, the sums' roundings counted 6- and 14-fold:
// RMS error up to 1.7 times this one at order 4 and steps of 3e-8 to 1e-7).  The
// increment is formed apart from lo and meets it in one rounding, by the last factor's
// multiply-add: increments are often smaller than lo there, and added to it term by
// term they were rounded at its magnitude two or three times (up to 3 times the
// error at steps of 1e-9, 1.2 to 1.6 at 1e-8).
//
// Every operation is written as the one instruction it is, so that a point
// computed twice -- by its owner in group(), by a neighbour as a ghost cell in
// point() -- is computed the same way twice.
//
// PLAIN: the order-2 update as cB b - cA u a, 7 operations.  The unforced FP32
// single domain keeps it: its trajectories feed the FP32 gradient, which
// divides their rounding by |u(T) - target|, and stay bit for bit what they
// were before the factored form.
template <typename T, int ORDER, int PREC, bool PLAIN>
struct StencilK {
    static constexpr int R = ORDER / 2;
    static constexpr bool WINDOW = PREC != 2;   // from the values of a window
    T cA, cr, cB;
    double cB64;
    __device__ __forceinline__ StencilK(T cA_, T cr_, const Params &p)
        : cA(cA_), cr(cr_), cB((T)p.cB32), cB64(p.cB)
    {
    }

    // what a lane carries from point to point
    struct Carry {
        T w[2];                        // WINDOW: the R words left of the point
        T d0, d1, l0, l1;              // else d_{i-1}, d_i of the hi words and of the lo words (order 2: d_{i-1})
        T eh, el, e0, e1;              // e_i of the hi words, of the lo words; e_{i-1}, e_i (their sums)
    };

    // cr b - u a + F / cA
    __device__ __forceinline__ T increment(T cc, T a, T b, T F, bool forced) const
    {
        return fma(-cc, a, forced ? fma(cr, b, F) : cr * b);
    }

    // PREC 1: the viscous term in FP64
    __device__ __forceinline__ T point_v64(const T *w, T F, bool forced) const
    {
        const T cc = w[R];
        T a;
        double b64;
        if constexpr (ORDER == 2) {
            a = w[2] - w[0];
            b64 = ((double)w[2] + (double)w[0]) - 2.0 * (double)cc;
        } else {
            a = (T)8 * (w[2 * R - 1] - w[1]) - (w[2 * R] - w[0]);
            b64 = 16.0 * ((double)w[2 * R - 1] + (double)w[1]) - ((double)w[2 * R] + (double)w[0]) - 30.0 * (double)cc;
        }
        T rest = -cA * cc * a;
        if (forced) rest = rest + F;
        return (T)((double)cc + (cB64 * b64 + (double)rest));
    }

    // one point from its stencil values w[0 .. 2R] (offsets -R .. R)
    template <bool FORCED>
    __device__ __forceinline__ T point(const T *w, T F) const
    {
        const T cc = w[R];
        if constexpr (PREC == 1) {
            return point_v64(w, F, FORCED);
        } else if constexpr (PLAIN) {
            const T a = w[2] - w[0], b = (w[2] + w[0]) - (T)2 * cc;
            const T du = cB * b - cA * cc * a;
            return cc + du;
        } else if constexpr (ORDER == 2) {
            const T a = w[2] - w[0], b = fma((T)-2, cc, w[2] + w[0]);
            return fma(cA, increment(cc, a, b, F, FORCED), cc);
        } else {
            const T a = fma((T)8, w[2 * R - 1] - w[1], -(w[2 * R] - w[0]));
            const T b = fma((T)-30, cc, fma((T)16, w[2 * R - 1] + w[1], -(w[2 * R] + w[0])));
            return fma(cA, increment(cc, a, b, F, FORCED), cc);
        }
    }

    // the carry before the first point of a lane's run: lw the R words left of
    // it, c the run (lwl, cl: lo words)
    __device__ __forceinline__ void start(Carry &y, const T *lw, const T *lwl, const T *c, const T *cl) const
    {
        if constexpr (WINDOW) {
#pragma unroll
            for (int q = 0; q < R; ++q) y.w[q] = lw[q];
        } else if constexpr (ORDER == 2) {
            y.d0 = c[0] - lw[0];
            y.l0 = cl[0] - lwl[0];
        } else {
            const T dm = lw[R - 1] - lw[0], lm = lwl[R - 1] - lwl[0];
            y.d0 = c[0] - lw[R - 1];
            y.d1 = c[1] - c[0];
            y.l0 = cl[0] - lwl[R - 1];
            y.l1 = cl[1] - cl[0];
            y.e0 = (y.d0 - dm) + (y.l0 - lm);
            y.eh = y.d1 - y.d0;
            y.el = y.l1 - y.l0;
            y.e1 = y.eh + y.el;
        }
    }

    // the 4 points c of a group, in place; nx the R words right of it
    // (compensated state: cl, nxl the lo words), F their forcing
    template <bool FORCED>
    __device__ __forceinline__ void group(Carry &y, T *c, T *cl, const T *nx, const T *nxl, const T *F) const
    {
        if constexpr (WINDOW) {
            T v[4 + 2 * R];
#pragma unroll
            for (int q = 0; q < R; ++q) {
                v[q] = y.w[q];
                v[R + 4 + q] = nx[q];
                y.w[q] = c[4 - R + q];
            }
#pragma unroll
            for (int e = 0; e < 4; ++e) v[R + e] = c[e];
#pragma unroll
            for (int e = 0; e < 4; ++e) c[e] = point<FORCED>(v + e, FORCED ? F[FORCED ? e : 0] : (T)0);
        } else {
            T v[4 + R], vl[4 + R];
#pragma unroll
            for (int e = 0; e < 4 + R; ++e) {
                v[e] = e < 4 ? c[e < 4 ? e : 0] : nx[e >= 4 ? e - 4 : 0];
                vl[e] = e < 4 ? cl[e < 4 ? e : 0] : nxl[e >= 4 ? e - 4 : 0];
            }
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const T cc = v[e];
                T a, b;
                if constexpr (ORDER == 2) {
                    const T dn = v[e + 1] - cc, ln = vl[e + 1] - vl[e];
                    b = (dn - y.d0) + (ln - y.l0);
                    a = (dn + y.d0) + (ln + y.l0);
                    y.d0 = dn;
                    y.l0 = ln;
                } else {
                    const T dn = v[e + 2] - v[e + 1], ln = vl[e + 2] - vl[e + 1];
                    const T hn = dn - y.d1, kn = ln - y.l1, en = hn + kn;
                    a = fma((T)6, y.d1 + y.d0, fma((T)6, y.l1 + y.l0, -(en - y.e0)));
                    b = fma((T)14, y.eh, fma((T)14, y.el, -(en + y.e0)));
                    y.d0 = y.d1;
                    y.d1 = dn;
                    y.l0 = y.l1;
                    y.l1 = ln;
                    y.eh = hn;
                    y.el = kn;
                    y.e0 = y.e1;
                    y.e1 = en;
                }
                // two-sum of hi and (increment + lo): exact sum t + err
                const T yy = fma(cA, increment(cc, a, b, FORCED ? F[FORCED ? e : 0] : (T)0, FORCED), vl[e]);
                const T t = cc + yy;
                const T z = t - cc;
                cl[e] = (cc - (t - z)) + (yy - z);
                c[e] = t;
            }
        }
    }
};

// Synchronous algorithm: grid barrier before step `step` (1-based within the
// launch), combined per CTA.  Each warp counts itself on the CTA's shared
// counter; the warp completing the CTA's count arrives on the global counter
// and waits for all CTAs, then opens the CTA's epoch; the other warps wait
// for the epoch.  `wait` = false for the last arrival of a launch.  Bounded.
static __device__ __noinline__ bool cta_grid_sync(const Params &p, int *s_count, volatile long long *s_epoch,
                                                  long long step, bool wait)
{
    bool ok = true;
    if ((threadIdx.x & 31) == 0) {
        __threadfence();
        const int old = atomicAdd(s_count, 1);
        if ((long long)old + 1 == step * kWarps) {
            __threadfence();
            atomicAdd(p.gbar, 1ull);
            if (wait) ok = wait_grid(p, (unsigned long long)step * (unsigned long long)p.G, step);
            st_release_cta_shared(s_epoch, ok ? step : -1);
        } else if (wait) {
            const unsigned long long t0 = global_ns();
            long long ep;
            while ((ep = ld_acquire_cta_shared(s_epoch)) < step && ep >= 0) {
                if ((long long)(global_ns() - t0) > p.timeout_ns) { raise_timeout(p, kWhereGrid, step, -1); break; }
            }
            ok = (ep >= step);
        }
        __threadfence();
    }
    return __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
}

// The levels one launch advances a PE through: n0 .. n0 + n_steps, in passes
// of one level while the level is below s-1, then of sb levels (the last one
// shorter).  sb may differ between PEs (in an ensemble each PE takes the
// smallest delay bound of its subdomains): a PE's halo waits only need its
// neighbours' ring entries level by level, whatever their pass boundaries.
//
// The sweep direction alternates from pass to pass (lo..hi-1, then
// hi-1..lo, ...).  A pass of L+1 levels must start from its edge neighbours'
// level n exactly (delay 0); in a one-way sweep the first tile of a pass
// needs the left neighbour PE's last tile of the previous pass, so every PE
// waits on its neighbour at each pass start.  Alternating, each edge tile
// needs a tile its neighbour finished about a pass earlier; the tile at
// the turn is the same subdomain twice in a row, continued in registers; and
// the tiles next to it are still in the L2 cache, which is what passes of one
// level over a state about its size gain from: seeded delays, 2^25 FP32
// points, 100 levels, take 5.02 ms one way and 3.95 ms alternating (free
// delays on 2^26 points 4.27 ms before and 4.12 ms since).
//
// single: passes of one level while the level is below s-1 (the AT halos need
// s levels); the synchronous modes read level n only and have none.
struct Sweep {
    long long n0;              // level the launch starts from
    int n_steps;               // levels of the launch (the host keeps it below 2^30)
    int sb;
    int single;                // the first `single` levels take one-level passes (start-up)
};

// Position of a tile in a PE's sweep: the pass's first level n relative to n0,
// tile j (relative to the PE's first), the pass length, the direction of the
// pass, and the index of the pass within the launch.
struct Cursor {
    int n, j, len, pass;
    bool rev;
};

__device__ __forceinline__ int pass_len(const Sweep &sw, int n)
{
    const int left = sw.n_steps - n;
    return n < sw.single ? 1 : left < sw.sb ? left : sw.sb;
}

__device__ __forceinline__ int count_passes(const Sweep &sw)
{
    const int single = sw.single < sw.n_steps ? sw.single : sw.n_steps;
    return single + (sw.n_steps - single + sw.sb - 1) / sw.sb;
}

// the next tile of a sweep over tiles 0 .. S-1
__device__ __forceinline__ void advance(const Sweep &sw, Cursor &c, int S)
{
    const int end = c.rev ? 0 : S - 1;
    if (c.j != end) {
        c.j += c.rev ? -1 : 1;
    } else {
        // the next pass: back from the same tile
        c.rev = !c.rev;
        c.n += c.len;
        c.len = pass_len(sw, c.n);
        ++c.pass;
    }
}

// Exact boundary value of an ensemble instance (travelling tanh wave) at
// point `q` of the halo across face f of subdomain record b, at level lev.
template <int R>
static __device__ __noinline__ double exact_ghost64(const BatchInst *binst, const BatchSub &b, long long M, int f,
                                                    int q, long long lev)
{
    const BatchInst &bi = binst[b.inst];
    const long long gi = f ? ((long long)b.lp + 1) * M + q : (long long)b.lp * M - R + q;
    const double x = bi.x0 + (double)gi * bi.dx;
    const double t = (double)lev * bi.dt;
    return bi.tc - bi.ta * tanh(bi.ta * (x - bi.txc - bi.tc * t) / (2.0 * bi.nu));
}

template <typename T, int R>
__device__ __forceinline__ T exact_ghost(const BatchInst *binst, const BatchSub &b, long long M, int f, int q,
                                         long long lev)
{
    return (T)exact_ghost64<R>(binst, b, M, f, q, lev);
}

// The exact boundary value as a hi + lo pair of words (compensated state).
template <typename T, int R>
__device__ __forceinline__ T exact_ghost2(const BatchInst *binst, const BatchSub &b, long long M, int f, int q,
                                          long long lev, T &lo)
{
    const double g = exact_ghost64<R>(binst, b, M, f, q, lev);
    const T hi = (T)g;
    lo = (T)(g - (double)hi);
    return hi;
}

// ---------------------------------------------------------------------------
// one processing element (warp)
// ---------------------------------------------------------------------------
// Lane l keeps the gpl consecutive groups of 4 points gpl l .. gpl l + gpl - 1
// of the tile in registers for the whole pass, so that a level exchanges only
// R words with each neighbouring lane (one shuffle per word) and every other
// stencil value is the lane's own.  Lane 0 takes the left halo, the owner of
// the last group the right one.  A lane sweeps its points in order and in
// place, carrying the first and second differences from point to point.
// What bounds it is instruction issue, so that layout is the one with the fewest
// instructions: 16.8 a lane and update of the order-4 forced stencil in passes
// of 4 levels, 10 of them arithmetic.  (Interleaved runs of two groups per lane
// take four times the shuffles and a select per exchanged word, 23.8.  2^26
// points, FP32, 100 levels: 5.91 ms then, 4.27 ms so; the compensated state on
// 2^24 points 3.62 and 2.03 ms (2.06 with its exact differences kept apart); FP64
// on 2^22 points, 40 levels, bound by its FP64 pipe, 4.48 and 3.63 ms.)
//
// The tile travels through a shared-memory stage: 16-byte asynchronous copies
// in, coalesced in global memory and swizzled in the stage (see swizzle()), so
// that the lanes' reads of their consecutive chunks do not collide in the
// banks; the way back is the same stage in the other direction.  A warp's own
// copies and stores need no barrier and no proxy fence, only __syncwarp().
// A PE with one subdomain keeps it in registers for the whole launch.
//
// Halo values come from the ring entries of the neighbour's boundary words;
// an entry's halves carry the level they belong to (see st_entry), written and
// read as single 16-byte accesses, so an entry is its own notification: one
// read tells whether the level is there and brings it (a flag released after
// the entry costs the writer a fence and the reader a second trip to the L2
// cache: 16 subdomains of 256 FP64 points took 4.8 us a step that way, tiles
// written back and re-read every step, and take 2.9).  One lane per level and
// face reads them, a tile ahead; what is not there yet is read again when the
// tile is reached (bounded).
//
// In an ensemble (BATCH) a tile is cnt consecutive subdomains of one instance
// (see TileInfo; the faces between them at delay 0); the stencil factors,
// delay bound and seed come from its records in shared memory; a face whose
// record names no neighbour takes the instance's exact boundary values,
// undelayed.
//
// PREC (FP32 state only) 1: the viscous term nu dt D2(u) is formed from the
// stencil values in FP64 and added to u in FP64, rounded to FP32 once per
// update (for runs close to the diffusive stability limit).  2: compensated
// state: every point is the pair hi + lo of FP32 words (lo: array p.ur, the
// rounding error of hi); the stencil differences are formed word by word
// (differences of nearby hi words are exact, those of the lo words small),
// the halo values and ring entries carry both words, and each update adds
// the increment and lo to hi with an error-free two-sum (Knuth), keeping the
// new error as lo -- so that neither small increments nor the quantisation
// of the stored field are lost to FP32 rounding.
template <typename T, int ORDER, int GW, bool FORCED, bool FULL, bool BATCH, int PREC, bool BS>
__device__ void run_pe(const Params &p, const Sweep &sw, long long lo, int S, unsigned char *raw,
                       unsigned char *stages, const T *sj, const T *cj, const T *spt, const T *cpt,
                       const BatchSub *btab, int *s_count, volatile long long *s_epoch)
{
    constexpr int R = ORDER / 2;
    constexpr int S_LEV = ORDER / 2 + 1;
    constexpr unsigned kAll = 0xffffffffu;
    constexpr int NH = entry_halves<T, ORDER, PREC>();
    constexpr int kEnt = kRingHalf * NH;                 // bytes of a ring entry
    constexpr int CPG = (int)sizeof(T) / 4;              // 16-byte chunks per group of 4 points
    constexpr int WPC = 16 / (int)sizeof(T);             // words per chunk
    constexpr int NPT = 4 * GW;                          // points a lane holds at most
    constexpr int NCH = GW * CPG;                        // chunks a lane holds at most
    constexpr bool COMP = PREC == 2;
    constexpr bool ONE_LANE = !(FULL && GW > 1);         // a tile may lie in one lane
    constexpr bool bsync = BS;
    constexpr bool PLAIN = sizeof(T) == 4 && ORDER == 2 && PREC == 0 && !BATCH && !FORCED;
    using Stencil = StencilK<T, ORDER, PREC, PLAIN>;
    const int lane = threadIdx.x & 31;
    const int gpl = FULL ? GW : p.gpl;                   // groups per lane
    const int my_face = lane >> 4, my_m = lane & 15;     // halo work: lane 16 f + m serves face f
    // Blocked synchronous mode (AT_SYNC in passes of sb > 1 levels): every
    // delay is 0, a grid barrier precedes each pass, and a tile takes, instead
    // of the ring's per-level halo, its neighbours' edge strips of R sb points
    // at the pass's first level; the halo of each later level of the pass is
    // recomputed from them (ghost cells, the same arithmetic as the
    // neighbour's own update), so the result equals the unblocked AT_SYNC run
    // bit for bit.  Strips are written at the end of each pass (parity of the
    // pass index) and, at the launch start, from the state itself; barrier 1
    // follows that.
    // (a separate instantiation, BS: the host launches it for AT_SYNC with
    // passes of more than one level only)
    const int ep_off = bsync ? 1 : 0;                    // grid barriers before the first pass
    const bool sync_mode = p.mode == kModeSync;
    if (S <= 0) {
        // a PE without subdomains still takes part in every grid barrier
        if (sync_mode) {
            const int n_ep = count_passes(sw) + ep_off;  // arrivals of this launch
            for (int st = 1; st <= n_ep; ++st)
                if (!cta_grid_sync(p, s_count, s_epoch, st, st < n_ep)) break;
        }
        return;
    }
    // the subdomains of tile t of this PE (single domain: tile t is subdomain lo + t)
    auto tile_info = [&](int t) -> TileInfo {
        if constexpr (BATCH) {
            const int4 d = __ldg(p.tiles + lo + t);
            return TileInfo{d.x, d.y, d.z & 0xffff, d.z >> 16};
        } else {
            return TileInfo{(int)lo + t, 0, 1, 0};
        }
    };
    int rec_lo = 0;                      // place of this PE's first record
    if constexpr (BATCH) rec_lo = tile_info(0).rec;
    // the first and last subdomain records of a tile (ensembles)
    auto rec_first = [&](const TileInfo &ti) -> const BatchSub & { return btab[ti.rec - rec_lo]; };
    auto rec_last = [&](const TileInfo &ti) -> const BatchSub & { return btab[ti.rec - rec_lo + ti.cnt - 1]; };
    // whether face f of tile t is an edge of this PE's sweep: its neighbour is
    // not the adjacent tile (ensembles; the single domain: the PE's first and
    // last tile)
    auto link_edge = [&](int t, const TileInfo &ti, int f) -> bool {
        if constexpr (BATCH) return f == 0 ? !(t > 0 && (ti.link & 1)) : !(t + 1 < S && (ti.link & 2));
        else return f == 0 ? t == 0 : t == S - 1;
    };
    const int NS = p.stages;
    // tiles loaded ahead; the sweep revisits the subdomain of position i
    // after a turn 2i+1 tiles later, so at most 2 ahead
    int D = S - 1 < NS - 1 ? S - 1 : NS - 1;
    if (D > 2) D = 2;
    // groups of the tile, owner of the last one (FULL: every lane's run is
    // full, so the last group is the last of its lane)
    const int M = (int)p.M;
    int NG = M / 4;
    int lane_last = (NG - 1) / gpl, m_last = FULL ? GW - 1 : (NG - 1) - lane_last * gpl;
    const size_t tile_bytes = (size_t)M * sizeof(T);                   // one subdomain
    const size_t slot_stride = (size_t)p.P * 2 * kEnt;
    const unsigned tmask = (unsigned)p.T - 1u;
    const unsigned n0lo = (unsigned)sw.n0;
    const unsigned long long tag0 = entry_tag(sw.n0);    // tag of relative level 0
    // (test knob: the first tile's owner; in FP64 the first warp, which has a tile)
    bool stop_pub;
    if constexpr (sizeof(T) == 8) stop_pub = p.skip_publish && blockIdx.x == 0 && threadIdx.x < 32;
    else stop_pub = p.skip_publish && lo == 0;
    const T fX = sizeof(T) == 4 ? (T)p.fX32 : (T)p.fX;
    const int err_off = p.stage_bytes / 2;               // (compensated state: the error words of a tile)
    const Swizzle swz = FULL ? Swizzle::of(NCH) : Swizzle{p.swz_shift, p.swz_mask};
    // this lane's chunk k in a stage
    auto own_chunk = [&](int k) -> int { return FULL ? lane_chunk<NCH>(lane, k) : 16 * swz(gpl * CPG * lane + k); };

    // --- state tile copies: every lane its 16-byte chunks, one group per tile
    auto copy_in = [&](unsigned char *dst, const unsigned char *src, int nc) {
        src += 16 * lane;
        if (nc == 32 * NCH) {
#pragma unroll
            for (int t = 0; t < NCH; ++t) cp_async16(dst + swz.coalesced(lane, t), src + 512 * t);
        } else {
#pragma unroll
            for (int t = 0; t < NCH; ++t)
                if (lane + 32 * t < nc) cp_async16(dst + swz.coalesced(lane, t), src + 512 * t);
        }
    };
    auto issue_load = [&](int st, int t) {
        const TileInfo ti = tile_info(t);
        const int nc = (int)tile_bytes * ti.cnt / 16;
        unsigned char *dst = stages + st * p.stage_bytes;
        const size_t off = (size_t)ti.s0 * tile_bytes;
        copy_in(dst, reinterpret_cast<const unsigned char *>(p.u) + off, nc);
        if constexpr (COMP) copy_in(dst + err_off, reinterpret_cast<const unsigned char *>(p.ur) + off, nc);
        cp_async_commit();
    };

    // --- prescribed delays ----------------------------------------------------
    int kb = 0;                        // lane i: raw delay of (tile t0 + i/2, face i%2)
    unsigned kb_t0 = ~0u;
    auto raw_delay = [&](unsigned t, const Cursor &c) -> int {
        // prescribed modes draw 16 tiles' delays at once (one per lane)
        const unsigned t0 = t & ~15u;
        if (t0 != kb_t0) {
            // (n, j) of tile t0 + lane/2: its place in the sweep from that of c
            // (tile t), passes of one level, every other one reversed
            int jj = (c.rev ? S - 1 - c.j : c.j) - (int)(t - t0) + (lane >> 1), nn = c.n;
            while (jj < 0) { jj += S; --nn; }
            while (jj >= S) { jj -= S; ++nn; }
            if (((nn ^ c.n) & 1) != (c.rev ? 1 : 0)) jj = S - 1 - jj;
            int k = 0;
            if (nn >= 0 && nn < sw.n_steps) {
                // (prescribed delays: tiles of one subdomain)
                const TileInfo tj = tile_info(jj);
                if (p.mode == kModeSeeded) {
                    if constexpr (BATCH) {
                        const BatchSub &b = rec_first(tj);
                        k = seeded_delay(b.seed, sw.n0 + nn, b.lp, b.Pi, p.per_sub ? 0 : (lane & 1), b.L);
                    } else {
                        k = seeded_delay(p.seed, sw.n0 + nn, tj.s0, p.P, p.per_sub ? 0 : (lane & 1), p.L);
                    }
                } else if (p.mode == kModeReplay) {
                    k = p.delays[((long long)nn * p.P + tj.s0) * 2 + (lane & 1)];
                }
            }
            kb = k;
            kb_t0 = t0;
        }
        return __shfl_sync(kAll, kb, 2 * (int)(t - t0) + my_face);
    };

    // --- halo preparation -----------------------------------------------------
    // Lanes 16 f + m serve face f of a tile: the delay (or, free running, the
    // largest one the pass allows), and a first read of the neighbour's ring
    // entry of level n - k - m.
    unsigned long long hd[NH], ht[NH];   // the entry read: payload and level tag
    unsigned long long h_tag = 0;        // the tag wanted
    const unsigned char *h_at = nullptr; // the entry's address
    bool h_act = false;                  // this lane reads one
    int h_k = 0;                         // prescribed delay of the face (free running: 0)
    int h_kmax = 0;                      // free running: largest delay at the pass start
    int h_nb = 0;                        // the neighbour
    TileInfo hti{0, 0, 1, 0};            // the tile prepared
    T gvn = (T)0;                        // blocked synchronous mode: this lane's word of the edge strips
    auto prep = [&](unsigned t, const Cursor &c) {
        hti = tile_info(c.j);
        const int f = my_face;
        bool bnd = false, edge;
        int Lj = p.L;
        if constexpr (BATCH) {
            const BatchSub &bf = rec_first(hti);
            const long long nb = f ? rec_last(hti).right : bf.left;
            bnd = nb < 0;
            h_nb = bnd ? 0 : (int)nb;
            edge = !bnd && link_edge(c.j, hti, f);
            Lj = bf.L;
        } else {
            const int jg = hti.s0;
            h_nb = f ? (jg + 1 == (int)p.P ? 0 : jg + 1) : (jg == 0 ? (int)p.P - 1 : jg - 1);
            edge = link_edge(c.j, hti, f);
        }
        if constexpr (bsync) {
            // the neighbours' edge strips at the pass's first level: lanes
            // 0 .. G-1 the left neighbour's last G points, lanes 16 .. 16+G-1
            // the right neighbour's first
            const int G = R * c.len;
            if (!bnd && my_m < G) {
                const T *sp = reinterpret_cast<const T *>(
                    p.strip + ((size_t)((c.pass & 1) * p.P + h_nb) * 2 + (1 - f)) * kStripBytes);
                gvn = ld_cg(sp + (f ? my_m : p.strip_words - G + my_m));
            }
        } else {
            // largest delay at the start of the pass such that the last inner
            // step stays within L, and no level below 0 is ever read
            int kmax = Lj - (c.len - 1);
            if (sw.n0 + c.n < (long long)(kMaxL + S_LEV)) {
                const int ks = (int)sw.n0 + c.n - S_LEV + 1;
                kmax = ks < kmax ? ks : kmax;
            }
            kmax = kmax < 0 ? 0 : kmax;
            h_k = 0;
            if (p.mode == kModeSeeded || p.mode == kModeReplay) {
                const int kr = raw_delay(t, c);
                h_k = kr < 0 ? 0 : kr < kmax ? kr : kmax;
            }
            h_kmax = (p.mode == kModeFree && edge) ? kmax : 0;
            const int cnt = (h_k + h_kmax == 0 && c.len == 1) ? 1 : h_kmax + S_LEV;
            h_act = my_m < cnt && !bnd;
            const int d = c.n - h_k - my_m;              // relative level of this lane's entry
            h_tag = tag0 + (long long)d;
            h_at = p.ring + ((size_t)h_nb * 2 + (1 - f)) * kEnt + (size_t)((n0lo + (unsigned)d) & tmask) * slot_stride;
            ld_tagged<NH>(h_act, h_at, hd, ht);
        }
    };
    // Delay statistics: lane m counts the levels with delay m on its face
    // (cnt16: the delay 16 that no lane stands for)
    unsigned cnt_k = 0, cnt16 = 0;
    auto entry_ok = [&]() -> bool {
        bool ok = true;
#pragma unroll
        for (int h = 0; h < NH; ++h) ok = ok && ht[h] == h_tag;
        return ok;
    };
    // Reads again (bounded) the entries of the prepared tile that are not
    // there yet; free running, settles for the newest level that is there with
    // the s - 1 before it, if it is recent enough.  `first`: place of the
    // level n - k among the face's entries.  Returns false on abort.
    auto wait_entries = [&](const Cursor &c, int &k, int &first) -> bool {
        const int cnt = (h_k + h_kmax == 0 && c.len == 1) ? 1 : h_kmax + S_LEV;
        const bool face = ((__ballot_sync(kAll, h_act) >> (lane & 16)) & 0xffffu) != 0u;   // (no exact boundary)
        int base = 0;                  // offset of this lane's first entry
        const unsigned long long t0 = global_ns();
        for (int polls = 0;; ++polls) {
            const unsigned seen = (__ballot_sync(kAll, h_act && entry_ok()) >> (lane & 16)) & 0xffffu;
            bool ready = true;
            if (!face) {
                k = h_k;
            } else if (h_kmax == 0) {
                // the levels are given
                const unsigned want = (1u << cnt) - 1u;
                ready = (seen & want) == want;
                k = h_k;
            } else if (c.len == 1 && base == 0 && (seen & 1u)) {
                k = 0;                                 // level n itself
                first = 0;
            } else {
                unsigned run = seen & (seen >> 1);
                if constexpr (S_LEV == 3) run &= seen >> 2;
                run &= (2u << (h_kmax - base)) - 1u;
                ready = run != 0u;
                first = ready ? __ffs(run) - 1 : 0;
                k = base + first;
            }
            if (__all_sync(kAll, ready)) return true;
            if ((polls & 15) == 15) {
                const bool late = (long long)(global_ns() - t0) > p.timeout_ns;
                if (__any_sync(kAll, late || ld_relaxed(p.ctrl + kCtrlAbort) != 0)) {
                    // (the first lane of a face that is not there reports it; the
                    // first report stands)
                    if (!ready && my_m == 0) raise_timeout(p, kWhereFlag, sw.n0 + c.n, h_nb);
                    return false;
                }
                if (polls > 64) __nanosleep(64);
            }
            // (delay bounds above 13: the oldest levels a face may use are
            // read in turn with the newest 16)
            if (!ready && h_kmax > 0 && cnt > 16) {
                const int to = base ? 0 : cnt - 16, d = c.n - to - my_m;
                base = to;
                h_act = my_m + base < cnt;
                h_tag = tag0 + (long long)d;
                h_at = p.ring + ((size_t)h_nb * 2 + (1 - my_face)) * kEnt +
                       (size_t)((n0lo + (unsigned)d) & tmask) * slot_stride;
            }
            if (!ready) ld_tagged<NH>(h_act, h_at, hd, ht);
        }
    };
    int kcur = 0;                      // this face's delay at the pass start
    // Settles the delays of the prepared tile, counts and records them and
    // leaves the s entries of each face in `raw`.  Returns false on abort.
    auto resolve = [&](const Cursor &c) -> bool {
        int k = bsync ? 0 : h_k;
        if constexpr (!bsync) {
            int first = 0;
            // (everything read is there: the levels given, or level n itself)
            if (!__all_sync(kAll, !h_act || entry_ok())) {
                if (!wait_entries(c, k, first)) return false;
            }
            // the entries of levels n - k - m, m = 0 .. s-1, in order
            const unsigned e = (unsigned)(my_m - first);
            if (h_act && e < (unsigned)S_LEV) {
                unsigned long long *r = reinterpret_cast<unsigned long long *>(raw + my_face * kRawFace + e * kRawEntry);
#pragma unroll
                for (int h = 0; h < NH; ++h) r[h] = hd[h];
            }
        }
        // (the synchronous modes use level n itself at every level: k = 0)
        if (sync_mode) cnt_k += my_m == 0 ? (unsigned)c.len : 0u;
        else cnt_k += (unsigned)(my_m - k) < (unsigned)c.len ? 1u : 0u;
        if (p.L > 15) cnt16 += (my_m == 0 && !sync_mode && (unsigned)(16 - k) < (unsigned)c.len) ? 1u : 0u;
        // (the faces between a tile's subdomains: delay 0)
        if constexpr (BATCH) cnt_k += lane == 0 ? 2u * (unsigned)(hti.cnt - 1) * (unsigned)c.len : 0u;
        if (p.delays && p.mode != kModeReplay) {
            const int kstep = sync_mode ? 0 : 1;
            const int sf = my_face ? hti.s0 + hti.cnt - 1 : hti.s0;      // the subdomain of the face
            for (int i = 0; i < c.len; ++i) {
                int8_t *row = p.delays + (long long)(c.n + i) * p.P * 2;
                if (my_m == 0) row[(size_t)sf * 2 + my_face] = (int8_t)(k + kstep * i);
                if (BATCH && lane == 0)
                    for (int s = 0; s + 1 < hti.cnt; ++s) {
                        row[(size_t)(hti.s0 + s) * 2 + 1] = 0;
                        row[(size_t)(hti.s0 + s + 1) * 2 + 0] = 0;
                    }
            }
        }
        kcur = k;
        __syncwarp();
        return true;
    };

    // --- prologue -------------------------------------------------------------
    Cursor C{0, 0, pass_len(sw, 0), 0, false};        // tile being processed
    Cursor L = C, N = C;                              // next tile to load; tile after C
    advance(sw, N, S);
    int lead = 0;                      // tile index of L minus that of C
    int ahead = 0;                     // loads issued and not used yet
    int sl = 0;                        // stage of the next load
    int sr = 0;                        // stage of the next loaded tile to use
    unsigned char *stage = stages;     // stage of the tile last read: its way back
    // after a load: move to the next tile that is loaded (a turn tile is not:
    // it continues in registers; nor is any later tile of a PE with one
    // subdomain)
    auto load_next = [&]() {
        issue_load(sl, L.j);
        const int jj = L.j;
        advance(sw, L, S);
        ++lead;
        if (S == 1) {
            L.n = sw.n_steps;
        } else if (L.j == jj) {
            advance(sw, L, S);
            ++lead;
        }
        sl = (sl + 1 == NS) ? 0 : sl + 1;
        ++ahead;
    };
    bool ok = true;
    if constexpr (bsync) {
        // edge strips of the state at the launch's first level (parity 0),
        // then the first grid barrier
        // (every subdomain of this PE's tiles: records rec_lo .. rec_hi-1)
        const int sw4 = p.strip_words;
        const T *ust = reinterpret_cast<const T *>(p.u);
        long long nrec = S;
        if constexpr (BATCH) {
            const TileInfo tl_ = tile_info(S - 1);
            nrec = tl_.rec + tl_.cnt - rec_lo;
        }
        for (long long t = lane; t < nrec * 2 * sw4; t += 32) {
            const long long r = t / (2 * sw4);
            long long jj = lo + r;
            if constexpr (BATCH) jj = p.sub_order[rec_lo + r];
            const int f = (int)((t / sw4) & 1), wd = (int)(t % sw4);
            const long long src = jj * p.M + (f ? p.M - sw4 : 0) + wd;
            reinterpret_cast<T *>(p.strip + ((size_t)jj * 2 + f) * kStripBytes)[wd] = ust[src];
        }
        __syncwarp();
        if (!cta_grid_sync(p, s_count, s_epoch, 1, true)) ok = false;
        __syncwarp();
    }
    while (lead < D && L.n < sw.n_steps) load_next();
    int bar_pass = 0;                  // synchronous modes: the pass the grid barrier has admitted
    bool prepared = false;             // the halo of tile r has been prepared
    bool turn = false;                 // tile r continues tile r-1 in registers
    T c[NPT];                          // this lane's points
    T er[COMP ? NPT : 1];              // compensated state: carried rounding errors
    T F[FORCED ? NPT : 1];             // forcing (PREC 1: dt A sin x; else dt A sin x / cA)

    for (unsigned r = 0; C.n < sw.n_steps && ok; ++r) {
        // state copy of tile r + D (stage of tile r - 1, written back)
        if (lead <= D && L.n < sw.n_steps) load_next();
        --lead;
        // synchronous algorithm: before the first tile of a pass (a step when
        // unblocked), all PEs have finished the previous pass (grid barrier,
        // Algorithm 1)
        if (sync_mode && C.pass > bar_pass) {
            bar_pass = C.pass;
            if (!cta_grid_sync(p, s_count, s_epoch, C.pass + ep_off, true)) { ok = false; break; }
            __syncwarp();
        }
        if (!prepared) prep(r, C);
        if (!resolve(C)) { ok = false; break; }
        const TileInfo ti = hti;
        T gv = gvn;
        const int kf0 = kcur;
        // read the entries of tile r + 1 (in AT_SYNC not across the grid
        // barrier)
        prepared = N.n < sw.n_steps && !(sync_mode && N.pass != C.pass);
        if (prepared) prep(r + 1, N);
        const int n = C.n, len = C.len;                   // level at the pass start
        const int s0 = ti.s0, s1 = ti.s0 + ti.cnt - 1;    // its first and last subdomain
        T cA = sizeof(T) == 4 ? (T)p.cA32 : (T)p.cA;
        T cr = sizeof(T) == 4 ? (T)p.cr32 : (T)p.cr;
        bool bnd0 = false, bnd1 = false;
        if constexpr (BATCH) {
            const BatchSub &bf = rec_first(ti), &bl = rec_last(ti);
            if constexpr (sizeof(T) == 4) { cA = bf.cA32; cr = bf.cr32; }
            else { cA = (T)bf.cA; cr = (T)bf.cr; }
            bnd0 = bf.left < 0;
            bnd1 = bl.right < 0;
            NG = ti.cnt * M / 4;
            lane_last = (NG - 1) / gpl;
            if constexpr (!FULL) m_last = (NG - 1) - lane_last * gpl;
        }
        const bool is_first = lane == 0, is_last = lane == lane_last;
        // the state tile (a turn tile is already in registers)
        if (!turn) {
            cp_async_wait(--ahead);
            __syncwarp();
            stage = stages + sr * p.stage_bytes;
            if (++sr == NS) sr = 0;
#pragma unroll
            for (int m = 0; m < GW; ++m) {
                const bool has = FULL || (m < gpl && gpl * lane + m < NG);
#pragma unroll
                for (int h = 0; h < CPG; ++h) {
                    // (FULL: lanes beyond the tile read what the stage holds)
                    T *d = c + 4 * m + h * WPC;
                    if (has) lds<T, WPC>(reinterpret_cast<const T *>(stage + own_chunk(m * CPG + h)), d);
                    else
#pragma unroll
                        for (int e = 0; e < WPC; ++e) d[e] = (T)0;
                    if constexpr (COMP) {
                        T *de = er + 4 * m + h * WPC;
                        if (has)
                            lds<T, WPC>(reinterpret_cast<const T *>(stage + err_off + own_chunk(m * CPG + h)), de);
                        else
#pragma unroll
                            for (int e = 0; e < WPC; ++e) de[e] = (T)0;
                    }
                }
            }
            if constexpr (FORCED) {
                // A sin(x) dt = (dt A sin x_j) cos(i dx) + (dt A cos x_j) sin(i dx)
                // (the tables hold the PE's subdomains -1 .. S: entry j + 1),
                // formed once per pass and kept in registers
                const T fs = fX * spt[C.j + 1], fc = fX * cpt[C.j + 1];
#pragma unroll
                for (int m = 0; m < GW; ++m) {
                    const bool has = FULL || (m < gpl && gpl * lane + m < NG);
#pragma unroll
                    for (int h = 0; h < CPG; ++h) {
                        T sv[WPC], cv[WPC];
                        const int at = has ? own_chunk(m * CPG + h) : 0;
                        lds<T, WPC>(reinterpret_cast<const T *>(reinterpret_cast<const unsigned char *>(sj) + at), sv);
                        lds<T, WPC>(reinterpret_cast<const T *>(reinterpret_cast<const unsigned char *>(cj) + at), cv);
#pragma unroll
                        for (int e = 0; e < WPC; ++e) F[4 * m + h * WPC + e] = forcing_point(fs, fc, sv[e], cv[e]);
                    }
                }
            }
        }

        // blocked synchronous mode: ghost cells.  Lanes 0 .. G-1 hold the left
        // neighbour's points x = -G .. -1 (relative to the tile), lanes
        // 16 .. 16+G-1 the right neighbour's points M .. M+G-1, at the level
        // being advanced (G = R len; at the pass start, the strips)
        const int G = R * len;
        T gF = (T)0;                                         // this ghost point's forcing
        if constexpr (bsync && FORCED) {
            if (my_m < G) {
                const int sub = C.j + (my_face ? 2 : 0);
                const int off = my_face ? my_m : M + my_m - G;
                const int at = WPC * swz(off / WPC) + off % WPC;
                gF = forcing_point(fX * spt[sub], fX * cpt[sub], sj[at], cj[at]);
            }
        }

        // halo values of every inner level (delays k + i): lane 16 f + x, x <
        // R len, computes word x % R of level x / R once per tile; each level
        // then takes its 2R values by shuffle
        const bool hv_lanes = bsync || G <= 16;
        T hv = (T)0, hvl = (T)0;       // (hvl: lo word of a compensated state)
        if (!bsync && hv_lanes && my_m < G) {
            const int i = my_m / R, q = my_m % R;
            const unsigned char *rf = raw + my_face * kRawFace;
            if (BATCH && (my_face ? bnd1 : bnd0)) {
                const BatchSub &b = my_face ? rec_last(ti) : rec_first(ti);
                if constexpr (COMP) hv = exact_ghost2<T, R>(p.binst, b, p.M, my_face, q, sw.n0 + n + i, hvl);
                else hv = exact_ghost<T, R>(p.binst, b, p.M, my_face, q, sw.n0 + n + i);
            } else if constexpr (COMP) {
                hv = reinterpret_cast<const T *>(rf)[q];
                hvl = approx_halo_lo<T, S_LEV, R>(rf, kf0 + i, q);
            } else {
                hv = approx_halo<T, S_LEV>(rf, kf0 + i, q);
            }
        }
        const int k0cur = hv_lanes ? 0 : __shfl_sync(kAll, kf0, 0), k1cur = hv_lanes ? 0 : __shfl_sync(kAll, kf0, 16);
        // this lane's ring entry (slot 0) of the face it publishes, and the
        // faces published (the test knob stops those across the sweep's edges)
        unsigned char *const pe0 = p.ring + (is_first ? (size_t)s0 * 2 : (size_t)s1 * 2 + 1) * kEnt;
        const Stencil K(cA, cr, p);
        // one level of the tile, in place
        auto level = [&](int i) {
            const int lev = n + i + 1;                       // level being computed (relative)
            // the R words left and right of the lane's run: the neighbour
            // lanes' words, or the halo
            T lw[R], rw[R], lwl[R], rwl[R];                  // (.l: lo words of a compensated state)
            T hx[R], hxl[R];                                 // lane 0: left halo; others: right halo
            T hy[R], hyl[R];                                 // right halo of a one-lane tile
            T ownl[R], ownr[R];
            if (hv_lanes) {
                const int src_lane = is_first ? (bsync ? G - R : i * R) : (bsync ? 16 : 16 + i * R);
                const T src = bsync ? gv : hv;
#pragma unroll
                for (int q = 0; q < R; ++q) {
                    hx[q] = __shfl_sync(kAll, src, src_lane + q);
                    if constexpr (COMP) hxl[q] = __shfl_sync(kAll, hvl, src_lane + q);
                    if (ONE_LANE) {
                        hy[q] = __shfl_sync(kAll, src, (bsync ? 16 : 16 + i * R) + q);
                        if constexpr (COMP) hyl[q] = __shfl_sync(kAll, hvl, (bsync ? 16 : 16 + i * R) + q);
                    }
                }
                if constexpr (bsync && BATCH) {
                    // an ensemble's domain ends: the exact values
#pragma unroll
                    for (int q = 0; q < R; ++q) {
                        if (bnd0 && is_first)
                            hx[q] = exact_ghost<T, R>(p.binst, rec_first(ti), p.M, 0, q, sw.n0 + n + i);
                        if (bnd1 && is_last) {
                            const T g = exact_ghost<T, R>(p.binst, rec_last(ti), p.M, 1, q, sw.n0 + n + i);
                            if (ONE_LANE && is_first) hy[q] = g;
                            else hx[q] = g;
                        }
                    }
                }
            } else {
                // (long passes: R len > 16) the face's value, level by level
#pragma unroll
                for (int q = 0; q < R; ++q) {
                    auto val = [&](int f, T &l) -> T {
                        const unsigned char *rf = raw + f * kRawFace;
                        const int kf = (f ? k1cur : k0cur) + i;
                        l = (T)0;
                        if (BATCH && (f ? bnd1 : bnd0)) {
                            const BatchSub &b = f ? rec_last(ti) : rec_first(ti);
                            if constexpr (COMP) return exact_ghost2<T, R>(p.binst, b, p.M, f, q, sw.n0 + n + i, l);
                            else return exact_ghost<T, R>(p.binst, b, p.M, f, q, sw.n0 + n + i);
                        }
                        if constexpr (COMP) {
                            l = approx_halo_lo<T, S_LEV, R>(rf, kf, q);
                            return reinterpret_cast<const T *>(rf)[q];
                        } else {
                            return approx_halo<T, S_LEV>(rf, kf, q);
                        }
                    };
                    hx[q] = val(is_first ? 0 : 1, hxl[q]);
                    if (ONE_LANE) hy[q] = val(1, hyl[q]);
                }
            }
            // (runs that are not full: the last word of a lane's run is in
            // slot gpl - 1, and the last group may be in an earlier slot)
            T tail[R], taill[R];
#pragma unroll
            for (int q = 0; q < R; ++q) {
                tail[q] = c[NPT - R + q];
                if constexpr (COMP) taill[q] = er[NPT - R + q];
                if constexpr (!FULL) {
#pragma unroll
                    for (int m = 0; m + 1 < GW; ++m)
                        if (m == gpl - 1) {
                            tail[q] = c[4 * m + 4 - R + q];
                            if constexpr (COMP) taill[q] = er[4 * m + 4 - R + q];
                        }
                }
            }
            if constexpr (bsync) {
                // the tile's own edge words, for the ghost cells below
#pragma unroll
                for (int q = 0; q < R; ++q) {
                    T el = tail[q];
                    if constexpr (!FULL) {
#pragma unroll
                        for (int m = 0; m < GW; ++m) el = (m == m_last) ? c[4 * m + 4 - R + q] : el;
                    }
                    ownl[q] = __shfl_sync(kAll, c[q], 0);
                    ownr[q] = __shfl_sync(kAll, el, lane_last);
                }
            }
#pragma unroll
            for (int q = 0; q < R; ++q) {
                lw[q] = __shfl_up_sync(kAll, tail[q], 1);
                rw[q] = __shfl_down_sync(kAll, c[q], 1);
                lw[q] = is_first ? hx[q] : lw[q];
                if constexpr (COMP) {
                    lwl[q] = __shfl_up_sync(kAll, taill[q], 1);
                    rwl[q] = __shfl_down_sync(kAll, er[q], 1);
                    lwl[q] = is_first ? hxl[q] : lwl[q];
                }
                if (ONE_LANE) {
                    hx[q] = is_first ? hy[q] : hx[q];
                    if constexpr (COMP) hxl[q] = is_first ? hyl[q] : hxl[q];
                }
                if constexpr (FULL) {
                    rw[q] = is_last ? hx[q] : rw[q];
                    if constexpr (COMP) rwl[q] = is_last ? hxl[q] : rwl[q];
                }
            }
            if constexpr (bsync) {
                if (i + 1 < len) {
                    // the ghost cells of level n+i+1 from level n+i: ghost
                    // lanes and the tile's own edge words (not yet updated)
                    const bool left = lane < 16;
                    const int xo = left ? lane - G : lane - 16;      // x, or x - M on the right
                    T w[2 * R + 1];
#pragma unroll
                    for (int jj = -R; jj <= R; ++jj) {
                        const T gq = __shfl_sync(kAll, gv, (lane + jj) & 31);
                        const int y = xo + jj;
                        T v;
                        if (left) v = (y < 0) ? gq : ((R == 1 || y == 0) ? ownl[0] : ownl[R - 1]);
                        else v = (y >= 0) ? gq : ((R == 1 || y == -1) ? ownr[R - 1] : ownr[0]);
                        w[jj + R] = v;
                    }
                    gv = K.template point<FORCED>(w, gF);
                }
            }
            // the lane's points, left to right
            typename Stencil::Carry cy;
            K.start(cy, lw, lwl, c, er);
            T rb[R], rbl[R];                                 // new last words of the tile (its owner's)
#pragma unroll
            for (int m = 0; m < GW; ++m) {
                if (!FULL && m >= gpl) break;
                T nx[R], nxl[R];                             // the words right of the group
#pragma unroll
                for (int q = 0; q < R; ++q) {
                    nx[q] = m + 1 < GW ? c[4 * (m + 1 < GW ? m + 1 : m) + q] : rw[q];
                    if constexpr (COMP) nxl[q] = m + 1 < GW ? er[4 * (m + 1 < GW ? m + 1 : m) + q] : rwl[q];
                }
                if (!FULL && m >= m_last) {
#pragma unroll
                    for (int q = 0; q < R; ++q) {
                        if (m == gpl - 1) {
                            nx[q] = rw[q];
                            if constexpr (COMP) nxl[q] = rwl[q];
                        }
                        if (m == m_last) {
                            nx[q] = is_last ? hx[q] : nx[q];
                            if constexpr (COMP) nxl[q] = is_last ? hxl[q] : nxl[q];
                        }
                    }
                }
                K.template group<FORCED>(cy, c + 4 * m, COMP ? er + 4 * m : er, nx, nxl, FORCED ? F + 4 * m : F);
                if (FULL ? m == GW - 1 : m == m_last) {
#pragma unroll
                    for (int q = 0; q < R; ++q) {
                        rb[q] = c[4 * m + 4 - R + q];
                        if constexpr (COMP) rbl[q] = er[4 * m + 4 - R + q];
                    }
                }
            }
            // publish the new boundary values: face 0 by lane 0, face 1 by
            // the owner of the last group
            const size_t slot = (size_t)((n0lo + (unsigned)lev) & tmask) * slot_stride;
            const unsigned long long tag = tag0 + (unsigned)lev;
            bool pub0 = true, pub1 = true;
            if (stop_pub && sw.n0 + lev > p.skip_step) {
                pub0 = !link_edge(C.j, ti, 0);
                pub1 = !link_edge(C.j, ti, 1);
            }
            {
                T w[R], wl[R];             // word by word: no runtime choice between arrays
#pragma unroll
                for (int q = 0; q < R; ++q) {
                    w[q] = is_first ? c[q] : rb[q];
                    if constexpr (COMP) wl[q] = is_first ? er[q] : rbl[q];
                }
                st_entry<T, ORDER, PREC>((is_first && pub0) || (is_last && !is_first && pub1), pe0 + slot, w, wl, tag);
                // (a one-lane tile: lane 0 publishes both faces)
                if (ONE_LANE)
                    st_entry<T, ORDER, PREC>(is_first && is_last && pub1, p.ring + ((size_t)s1 * 2 + 1) * kEnt + slot, rb,
                                             rbl, tag);
            }
            if constexpr (BATCH && FULL) {
                // the faces between the subdomains of a multi-subdomain tile
                // (a subdomain is M / (4 GW) whole lanes): ring entries only of
                // the launch's last L + s levels -- no tile of this launch
                // reads them, and a later launch with other tiles reads back
                // to its first level - L - s + 1 at most
                if (ti.cnt > 1 && lev > sw.n_steps - (p.L + S_LEV)) {
                    const int lps = M / NPT, sidx = lane / lps, place = lane - sidx * lps;
                    unsigned char *const e = p.ring + slot + ((size_t)(s0 + sidx) * 2) * kEnt;
                    T w[R], wl[R];
#pragma unroll
                    for (int q = 0; q < R; ++q) { w[q] = c[NPT - R + q]; wl[q] = COMP ? er[COMP ? NPT - R + q : 0] : (T)0; }
                    st_entry<T, ORDER, PREC>(place == 0 && sidx >= 1 && sidx < ti.cnt, e, c, er, tag);
                    st_entry<T, ORDER, PREC>(place == lps - 1 && sidx + 1 < ti.cnt, e + kEnt, w, wl, tag);
                }
            }
        };
        for (int i = 0; i < len; ++i) level(i);
        if constexpr (bsync) {
            // edge strips of the pass's last level for the next pass
            const int gq = p.strip_words / 4;
            const size_t par_off = (size_t)((C.pass + 1) & 1) * p.P;
            T *st0 = reinterpret_cast<T *>(p.strip + ((par_off + s0) * 2 + 0) * kStripBytes);
            T *st1 = reinterpret_cast<T *>(p.strip + ((par_off + s1) * 2 + 1) * kStripBytes);
            // (read after the next grid barrier: the warp barrier at the end
            // of this tile and the fence of the arrival order them before it)
#pragma unroll
            for (int m = 0; m < GW; ++m) {
                const int g = gpl * lane + m;
                if (!FULL && m >= gpl) continue;
                if (g < gq) stg4<T>(st0 + 4 * g, c + 4 * m);
                if (g >= NG - gq && g < NG) stg4<T>(st1 + 4 * (g - (NG - gq)), c + 4 * m);
            }
        }
        // before a turn, and with one subdomain, the words stay in registers
        const bool keep = N.j == C.j && N.n < sw.n_steps;
        if (!keep || p.levels) {
            // back through the tile's stage to coalesced 16-byte stores
            // (lanes beyond a FULL tile write chunks nobody reads)
#pragma unroll
            for (int m = 0; m < GW; ++m) {
                if (FULL || (m < gpl && gpl * lane + m < NG)) {
#pragma unroll
                    for (int h = 0; h < CPG; ++h) {
                        stsv<T, WPC>(reinterpret_cast<T *>(stage + own_chunk(m * CPG + h)), c + 4 * m + h * WPC);
                        if constexpr (COMP)
                            stsv<T, WPC>(reinterpret_cast<T *>(stage + err_off + own_chunk(m * CPG + h)),
                                         er + 4 * m + h * WPC);
                    }
                }
            }
            __syncwarp();
            const int nc = (int)tile_bytes * ti.cnt / 16;
            auto copy_out = [&](const unsigned char *src, unsigned char *dst) {
                dst += 16 * lane;
                if (nc == 32 * NCH) {
#pragma unroll
                    for (int t = 0; t < NCH; ++t)
                        st_cg16(dst + 512 * t, *reinterpret_cast<const uint4 *>(src + swz.coalesced(lane, t)));
                } else {
#pragma unroll
                    for (int t = 0; t < NCH; ++t)
                        if (lane + 32 * t < nc)
                            st_cg16(dst + 512 * t, *reinterpret_cast<const uint4 *>(src + swz.coalesced(lane, t)));
                }
            };
            const size_t off = (size_t)s0 * tile_bytes;
            if (!keep) {
                copy_out(stage, reinterpret_cast<unsigned char *>(p.u) + off);
                if constexpr (COMP) copy_out(stage + err_off, reinterpret_cast<unsigned char *>(p.ur) + off);
            }
            if (p.levels)
                copy_out(stage, reinterpret_cast<unsigned char *>(p.levels) +
                                    (size_t)((sw.n0 + n + len) % p.levels_depth) * (size_t)p.N * sizeof(T) + off);
        }
        // orders this tile's stores (and the raw entries' reads) before the
        // other lanes' next copies of it
        __syncwarp();
        turn = N.j == C.j;
        C = N;
        advance(sw, N, S);
    }
    // synchronous algorithm: the last pass's arrival at the grid barrier
    if (ok && sync_mode) cta_grid_sync(p, s_count, s_epoch, count_passes(sw) + ep_off, false);
    // let every copy in flight land before the warp leaves
    cp_async_wait(0);
    __syncwarp();
    if (my_m <= p.L && cnt_k) atomicAdd(p.hist + my_m, (unsigned long long)cnt_k);
    if (cnt16) atomicAdd(p.hist + 16, (unsigned long long)cnt16);
}

// ---------------------------------------------------------------------------
// the persistent kernel
// ---------------------------------------------------------------------------
// (a compensated state in runs of one and two groups a lane, and of four at order 2
// unforced: the registers that three CTAs an SM leave, or four, are a few short of
// what the compiler would take: 4800 subdomains of 256 points, order 4, 5.0 us a
// seeded level, 6.1 with a CTA less)
constexpr int stepper_min_ctas(int order, int gw, bool forced, bool batch, int prec)
{
    if (prec != 2) return AT_MIN_CTAS_PER_SM;
    return gw == 1 && !forced && !batch ? 4 : gw <= 2 || (gw == 4 && order == 2 && !forced && !batch) ? 3 : AT_MIN_CTAS_PER_SM;
}

template <typename T, int ORDER, int GW, bool FORCED, bool FULL, bool BATCH, int PREC, bool BS>
__global__ void __launch_bounds__(kThreads, stepper_min_ctas(ORDER, GW, FORCED, BATCH, PREC)) at_stepper(const Params p)
{
    extern __shared__ __align__(128) unsigned char smem[];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // this warp's tiles (an ensemble: of its CTA's group)
    int g0 = 0, g1 = p.G;
    long long t0 = 0, t1 = p.ntiles;
    if constexpr (BATCH) {
        for (int g = 0; g < p.split.groups; ++g) {
            if ((int)blockIdx.x < p.split.cta[g]) break;
            g0 = p.split.cta[g]; g1 = p.split.cta[g + 1];
            t0 = p.split.tile[g]; t1 = p.split.tile[g + 1];
        }
    }
    // (fewer tiles than warps: FP64 spreads them over the CTAs, whose SMs' pipes set its
    // pace; FP32 fills the last CTAs with them, whose neighbours are then near.  100
    // subdomains of 256 points in passes of 4: FP32 0.45 us a level on 25 SMs, 0.54 on
    // 100; FP64, 600 of 1000: 23.8 us a level on 75 SMs, 12.8 on 152.)
    const long long G = g1 - g0, g = (int)blockIdx.x - g0;
    const ItemRange own = sizeof(T) == 8 ? cta_items(t1 - t0, G, kWarps, g, w) : item_range(t1 - t0, G * kWarps, g * kWarps + w);
    const long long lo = t0 + own.lo, hi = t0 + own.hi;
    const long long S = hi - lo;
    unsigned char *raw = smem + p.raw_off + (size_t)w * kRawBytes;
    unsigned char *stages = smem + p.stage_off + (size_t)w * p.stages * p.stage_bytes;
    T *tab = reinterpret_cast<T *>(smem + p.tab_off);
    T *sj = tab, *cj = tab + p.tab_words;
    T *spt = tab + 2 * p.tab_words + (size_t)w * 2 * (p.smax + 2), *cpt = spt + p.smax + 2;
    BatchSub *btab = reinterpret_cast<BatchSub *>(smem + p.tab_off) + (size_t)w * p.smax;
    // time level of the state, advanced at the end of the previous launch
    Sweep sw;
    sw.n0 = *reinterpret_cast<const volatile long long *>(p.ctrl + kCtrlN0);
    sw.n_steps = (int)p.n_steps;
    sw.sb = p.sb;
    sw.single = (p.mode != kModeSync && sw.n0 < ORDER / 2) ? ORDER / 2 - (int)sw.n0 : 0;

    __shared__ int s_count;                   // grid-barrier arrivals of this CTA's warps
    __shared__ long long s_epoch;             // last grid barrier this CTA passed
    if (threadIdx.x == 0) { s_count = 0; s_epoch = 0; }
    // (a CTA without subdomains forms no tables: 8 us of an SM's FP64 pipe at M = 1024)
    if (FORCED && __syncthreads_or(S > 0)) {
        // sin/cos of the offsets j dx within a subdomain and of the subdomain
        // origins x0 + p M dx (FP64), so that A sin(x_i) needs two FMAs
        for (long long i = threadIdx.x; i < p.M; i += blockDim.x) {
            double sv, cv;
            sincos((double)i * p.dx, &sv, &cv);
            constexpr int WPC = 16 / (int)sizeof(T);
            const Swizzle swz{p.swz_shift, p.swz_mask};
            const int tp = WPC * swz((int)i / WPC) + (int)i % WPC;
            sj[tp] = (T)sv;
            cj[tp] = (T)cv;
        }
        // entry i: subdomain lo - 1 + i (wrapped), i = 0 .. S + 1
        for (long long i = lane; i < S + 2; i += 32) {
            long long q = lo - 1 + i;
            if (q < 0) q += p.P;
            if (q >= p.P) q -= p.P;
            double sv, cv;
            sincos(p.x0 + (double)(q * p.M) * p.dx, &sv, &cv);
            spt[i] = (T)sv;
            cpt[i] = (T)cv;
        }
    }
    if constexpr (BATCH) {
        // this PE's subdomain records, in the order of its tiles; passes no
        // longer than the smallest delay bound among them allows
        // (k0 + len - 1 <= L), except in the synchronous modes
        long long r_lo = 0, r_hi = 0;
        if (S > 0) {
            const int4 a = p.tiles[lo], b = p.tiles[hi - 1];
            r_lo = a.y;
            r_hi = (long long)b.y + (b.z & 0xffff);
        }
        uint4 *dst = reinterpret_cast<uint4 *>(btab);
        constexpr int kVec = (int)(sizeof(BatchSub) / sizeof(uint4));
        for (long long i = lane; i < (r_hi - r_lo) * kVec; i += 32)
            dst[i] = reinterpret_cast<const uint4 *>(p.bsub + p.sub_order[r_lo + i / kVec])[i % kVec];
        int lmin = kMaxL;
        for (long long i = lane; i < r_hi - r_lo; i += 32) lmin = min(lmin, p.bsub[p.sub_order[r_lo + i]].L);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) lmin = min(lmin, __shfl_xor_sync(0xffffffffu, lmin, o));
        if (p.mode != kModeSync && sw.sb > lmin + 1) sw.sb = lmin + 1;
    }
    __syncthreads();
    run_pe<T, ORDER, GW, FORCED, FULL, BATCH, PREC, BS>(p, sw, lo, (int)S, raw, stages, sj, cj, spt, cpt, btab, &s_count,
                                                       &s_epoch);
    // the last CTA to finish advances the level of the state and rearms the
    // grid barrier for the next launch (every CTA has read the level by now)
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        if (atomicAdd(p.ctrl + kCtrlDone, 1) == p.G - 1) {
            *reinterpret_cast<volatile long long *>(p.ctrl + kCtrlN0) = sw.n0 + p.n_steps;
            *reinterpret_cast<volatile int *>(p.ctrl + kCtrlDone) = 0;
            *reinterpret_cast<volatile unsigned long long *>(p.gbar) = 0ull;
            __threadfence();
        }
    }
}

// ---------------------------------------------------------------------------
// state (re)initialisation: level-0 boundary values into ring slot 0 (the host
// has cleared the ring)
// ---------------------------------------------------------------------------
// Ring entry of R words at u (a compensated state starts with lo words of 0).
template <typename T, int R>
__device__ __forceinline__ void put_entry(const Params &p, unsigned char *e, const T *u, long long level)
{
    const T v[2] = {u[0], R > 1 ? u[R - 1] : (T)0}, l[2] = {(T)0, (T)0};
    if constexpr (sizeof(T) == 4 && R == 2) {
        if (p.nh == 2) { st_entry<T, 2 * R, 2>(true, e, v, l, entry_tag(level)); return; }
    }
    st_entry<T, 2 * R, 0>(true, e, v, l, entry_tag(level));
}

template <typename T, int R>
__global__ void at_init(const Params p)
{
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long j = (long long)blockIdx.x * blockDim.x + threadIdx.x; j < p.P; j += stride) {
        const T *u = reinterpret_cast<const T *>(p.u) + j * p.M;
        unsigned char *e = p.ring + (size_t)j * 2 * kRingHalf * p.nh;
        put_entry<T, R>(p, e, u, 0);
        put_entry<T, R>(p, e + kRingHalf * p.nh, u + p.M - R, 0);
    }
    if (blockIdx.x == 0) {
        if (threadIdx.x < kCtrlWords) p.ctrl[threadIdx.x] = 0;
        if (threadIdx.x <= p.L) p.hist[threadIdx.x] = 0ull;
        if (threadIdx.x == 0) *p.gbar = 0ull;
    }
}

// ---------------------------------------------------------------------------
// restart from stored levels: ring slots of levels lo_level .. level from the
// full fields levels[l mod depth] (the host has cleared the ring), the control
// block cleared with the state's level set to `level`
// ---------------------------------------------------------------------------
template <typename T, int R>
__global__ void at_restore(const Params p, const T *levels, long long depth, long long lo_level, long long level)
{
    const long long nl = level - lo_level + 1;
    const long long stride = (long long)gridDim.x * blockDim.x;
    const size_t ent = (size_t)kRingHalf * p.nh;
    for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < p.P * nl; t += stride) {
        const long long j = t % p.P, l = lo_level + t / p.P;
        const T *u = levels + (size_t)(l % depth) * (size_t)p.N + (size_t)j * p.M;
        unsigned char *e = p.ring + ((size_t)(l & (p.T - 1)) * p.P + j) * 2 * ent;
        put_entry<T, R>(p, e, u, l);
        put_entry<T, R>(p, e + ent, u + p.M - R, l);
    }
    if (blockIdx.x == 0) {
        if (threadIdx.x < kCtrlWords) p.ctrl[threadIdx.x] = 0;
        __syncthreads();
        if (threadIdx.x == 0) {
            *reinterpret_cast<long long *>(p.ctrl + kCtrlN0) = level;
            *p.gbar = 0ull;
        }
    }
}

}  // namespace atk

// ---------------------------------------------------------------------------
// kernel selection (each translation unit instantiates one word size and
// either the single-domain or the ensemble kernels)
// ---------------------------------------------------------------------------
namespace atk {

template <typename T, int ORDER, bool FORCED, bool FULL, bool BATCH, int PREC, bool BS>
void *stepper_gw(int gw)
{
    switch (gw) {
    case 1: return (void *)at_stepper<T, ORDER, 1, FORCED, FULL, BATCH, PREC, BS>;
    case 2: return (void *)at_stepper<T, ORDER, 2, FORCED, FULL, BATCH, PREC, BS>;
    case 4: return (void *)at_stepper<T, ORDER, 4, FORCED, FULL, BATCH, PREC, BS>;
    default: return (void *)at_stepper<T, ORDER, 8, FORCED, FULL, BATCH, PREC, BS>;
    }
}

template <typename T, int ORDER, bool FORCED, bool BATCH, int PREC, bool BS>
void *stepper_full(int gw, bool full)
{
    return full ? stepper_gw<T, ORDER, FORCED, true, BATCH, PREC, BS>(gw)
                : stepper_gw<T, ORDER, FORCED, false, BATCH, PREC, BS>(gw);
}

// Stepper for stencil order 2|4, gw groups of 4 points per lane (1, 2, 4 or
// 8), with or without forcing (single domain only), full tiles (M = 128 gw)
// or not; PREC 1: FP64 viscous accumulation, 2: compensated state; BS: the
// blocked synchronous mode (AT_SYNC in passes of more than one level).
template <typename T, bool BATCH, int PREC = 0, bool BS = false>
void *stepper_kernel(int order, int gw, bool forced, bool full)
{
    if constexpr (BATCH) {
        return order == 2 ? stepper_full<T, 2, false, true, PREC, BS>(gw, full)
                          : stepper_full<T, 4, false, true, PREC, BS>(gw, full);
    } else {
        if (order == 2)
            return forced ? stepper_full<T, 2, true, false, PREC, BS>(gw, full)
                          : stepper_full<T, 2, false, false, PREC, BS>(gw, full);
        return forced ? stepper_full<T, 4, true, false, PREC, BS>(gw, full)
                      : stepper_full<T, 4, false, false, PREC, BS>(gw, full);
    }
}

}  // namespace atk
