// at_adjoint.cuh -- discrete adjoint of the AT time step (reverse mode).
//
// One step takes lambda^{n+1} = dJ/du^{n+1} to lambda^n = dJ/du^n for a
// scalar J of the final level, given the stored level u^n, the levels the
// delayed halos of level n were extrapolated from, and the delays of level n.
// One cooperative launch takes the steps of a whole checkpoint interval,
// n_hi - 1 down to n_lo, with a grid barrier (bounded) between steps.
//
// The forward step (Sec. 3.2, Eq. BS, AT halos of Eq. AT1/AT2 in split form)
// writes u^{n+1}_i = v_0 + cB b(v) - cA v_0 a(v) (+ forcing, independent of u
// and nu), with a = sum_j alpha_j v_j, b = sum_j beta_j v_j over the stencil
// values v_j (j = -R..R) of point i.  Each v_j is u^n at a point of the same
// subdomain, or across a subdomain face with delay k the extrapolation
// sum_m w_m(k) u^{n-k-m} of the neighbour's point.  So
//     d u^{n+1}_i / d v_j = [j = 0] (1 - cA a) + cB beta_j - cA v_0 alpha_j,
//     d u^{n+1}_i / d nu  = (cB / nu) b.
// lambda^n_i gathers, over every point r whose stencil reads u^n_i at level n
// (the point itself, its neighbours in the subdomain, and a neighbouring
// subdomain's boundary points when that face's delay is 0), the term
// lambda^{n+1}_r d u^{n+1}_r / d v_{i-r}.  Reads of older levels (k + m >= 1)
// are scattered into a pending ring [slot][P][2][R] by the one thread that owns
// the reading face (one writer per slot entry and step) and collected, then
// cleared, when the sweep reaches that level (no atomics there); dJ/dnu is
// summed per block in FP64 and added into the block's own slot (one add per
// block and launch, so the sum's order is fixed).  Blocks walk the subdomains, 4 points per thread; the
// word offsets of the levels read are computed on the host.
#pragma once

#include "at_kernels.cuh"

namespace atk {

constexpr int kAdjMaxLevels = 20;   // levels n .. n-L-s+1 a step reads (L <= 16, s <= 3)

struct AdjParams {
    const void *levels;        // full fields of the stored levels, N words each: level l in slot l mod Dl
    long long Dl;
    void *lam_a, *lam_b;       // lambda, N words each: lambda^{n_hi} in lam_a, then alternating
    void *pend;                // [Tp][P][2][R] words: adjoint of boundary values at older levels
    double *dnu_part;          // running FP64 sums of dJ/dnu, one per block (at_adjoint_warp: per subdomain)
    const int8_t *delays;      // delays of level n at delays[(n - k_level) * P * 2 + p * 2 + face]
    long long k_level;         // level of the delays' first row
    long long N, P, M;
    int L, Tp;                 // Tp: a power of two
    double cA, cB, dtdx2;      // as the stepper's; dtdx2 = cB / nu
    float cAf, cBf, dtdx2f;    // the same in FP32 (FP32 kernels convert nothing per point)
    long long n_hi, n_lo;      // this launch: lambda^{n_hi} -> lambda^{n_lo}, n_hi > n_lo
    unsigned long long *bar;   // grid-barrier arrivals, zero at the launch
    int *ctrl;                 // the solver's control block (status, abort word)
    long long timeout_ns;      // bound of each wait
    // one subdomain per warp (at_adjoint_warp; lambda in lam_a only)
    unsigned char *msg;        // messages between neighbours [kAdjMsgSlots][P][2], zero at the first launch
    int gpl, swz_shift, swz_mask, stage_bytes;   // tile layout, as the stepper's
    long long stop_below;      // test knob: subdomain 0 leaves out intervals that start at or below it (0: none)
};

template <int ORDER>
struct Coeffs;
template <>
struct Coeffs<2> {
    static __device__ __forceinline__ int alpha(int j) { return j; }                 // a = v1 - v-1
    static __device__ __forceinline__ int beta(int j) { return j == 0 ? -2 : 1; }    // b = v1 + v-1 - 2 v0
};
template <>
struct Coeffs<4> {
    // a = 8 (v1 - v-1) - (v2 - v-2), b = 16 (v1 + v-1) - (v2 + v-2) - 30 v0
    static __device__ __forceinline__ int alpha(int j) { return j == 0 ? 0 : (j == 1 ? 8 : j == -1 ? -8 : j == 2 ? -1 : 1); }
    static __device__ __forceinline__ int beta(int j) { return j == 0 ? -30 : (j == 1 || j == -1) ? 16 : -1; }
};

// Per-step view of the stored levels and the adjoint fields, with 32-bit
// indices within a level (the host checks N < 2^31); off[q] is the word
// offset of level n - q in the stored levels (in shared memory).
template <typename T, int ORDER>
struct AdjStep {
    static constexpr int R = ORDER / 2;
    static constexpr int S_LEV = ORDER / 2 + 1;
    const AdjParams &a;
    long long n;               // level of the lambda being computed
    const long long *off;
    const T *lev;              // stored levels
    const T *un;               // level n
    const T *lam;              // lambda^{n+1}
    int M, P;
    T cA, cB;

    __device__ AdjStep(const AdjParams &p, long long n_, const long long *off_, const T *lam_)
        : a(p), n(n_), off(off_), lev(reinterpret_cast<const T *>(p.levels)),
          un(reinterpret_cast<const T *>(p.levels) + off_[0]), lam(lam_), M((int)p.M), P((int)p.P)
    {
        if constexpr (sizeof(T) == 4) { cA = p.cAf; cB = p.cBf; }
        else { cA = (T)p.cA; cB = (T)p.cB; }
    }

    // delay of face f of subdomain p at level n (the forward run's, read from
    // the recomputation's record or the replayed array), clamped as the
    // forward run clamps it (no level below 0, at most L)
    __device__ int delay(int p, int f) const
    {
        int k = a.delays[((size_t)(n - a.k_level) * a.P + p) * 2 + f];
        long long kmax = n - S_LEV + 1;
        if (kmax < 0) kmax = 0;
        if (kmax > a.L) kmax = a.L;
        if (k > kmax) k = (int)kmax;
        if (k < 0) k = 0;
        return k;
    }

    // halo value of point src extrapolated with delay k (same operations as
    // the stepper's halo approximation: Newton form)
    __device__ T halo(int src, int k) const
    {
        const T r0 = lev[off[k] + src];
        if (k == 0) return r0;
        const T r1 = lev[off[k + 1] + src];
        const T d1 = r0 - r1;
        if constexpr (S_LEV == 2) {
            return r0 + (T)k * d1;
        } else {
            const T r2 = lev[off[k + 2] + src];
            const T d2 = d1 - (r1 - r2);
            return r0 + ((T)k * d1 + (T)(k * (k + 1) / 2) * d2);
        }
    }

    __device__ int left(int p) const { return p == 0 ? P - 1 : p - 1; }
    __device__ int right(int p) const { return p == P - 1 ? 0 : p + 1; }

    // stencil values v[0..2R] at level n of point loc of subdomain p, whose
    // faces have delays k0, k1
    __device__ void values(int p, int loc, int k0, int k1, T *v) const
    {
#pragma unroll
        for (int j = -R; j <= R; ++j) {
            const int lj = loc + j;
            if (lj < 0) v[j + R] = halo(left(p) * M + M + lj, k0);
            else if (lj >= M) v[j + R] = halo(right(p) * M + (lj - M), k1);
            else v[j + R] = un[p * M + lj];
        }
    }

    // lambda^{n+1}_r d u^{n+1}_r / d v_j, given the values v of point r
    __device__ T gbar(int r, int j, const T *v) const
    {
        T av = (T)0;
#pragma unroll
        for (int q = -R; q <= R; ++q) av += (T)Coeffs<ORDER>::alpha(q) * v[q + R];
        T d = cB * (T)Coeffs<ORDER>::beta(j) - cA * v[R] * (T)Coeffs<ORDER>::alpha(j);
        if (j == 0) d += (T)1 - cA * av;
        return lam[r] * d;
    }

    __device__ T *pend(long long l, int p, int side, int r) const
    {
        return reinterpret_cast<T *>(a.pend) + (((size_t)(l & (a.Tp - 1)) * a.P + p) * 2 + side) * R + r;
    }
};

// Block (x, y) handles the chunk of points y*C .. y*C+C-1 (C = 1024: a thread
// takes 4 points, 256 apart) of subdomains x, x + gridDim.x, ...  Each point
// first computes the 2R+1 terms it contributes to the adjoint of its stencil
// values (c_j = lambda^{n+1}_r d u^{n+1}_r / d v_j) into shared memory; each
// point then gathers the terms of its readers from there.
constexpr int kAdjThreads = 256;
constexpr int kAdjPts = 4;                            // points per thread
constexpr int kAdjChunk = kAdjThreads * kAdjPts;      // points per block and subdomain

// One step, lambda^{n+1} (lam_in) -> lambda^n (lam_out), by this block;
// returns the block's FP64 contribution to dJ/dnu (thread 0).
template <typename T, int ORDER>
__device__ double adjoint_level(const AdjParams &a, long long n, const long long *s_off, const T *lam_in, T *lam_out,
                                T (*s_c)[kAdjChunk], T *red)
{
    constexpr int R = ORDER / 2;
    constexpr int S_LEV = ORDER / 2 + 1;
    const AdjStep<T, ORDER> A(a, n, s_off, lam_in);
    T nu_acc = (T)0;          // this thread's sum of lambda^{n+1}_i b_i
    const T dtdx2 = sizeof(T) == 4 ? (T)a.dtdx2f : (T)a.dtdx2;
    const int tid = threadIdx.x, lane = tid & 31;
    const int M = A.M;
    const int chunk_lo = blockIdx.y * kAdjChunk;
    for (int p = blockIdx.x; p < A.P; p += gridDim.x) {
        const int pl = A.left(p), pr = A.right(p);
        // loads that need no delay first (lambda^{n+1}; the pending words
        // addressed to this level), so that their latency overlaps the delays'
        T gl[kAdjPts], pw[kAdjPts];
#pragma unroll
        for (int kp = 0; kp < kAdjPts; ++kp) {
            const int loc = chunk_lo + tid + kp * kAdjThreads;
            gl[kp] = loc < M ? A.lam[p * M + loc] : (T)0;
            pw[kp] = loc < R ? *A.pend(n, p, 0, loc) : (loc >= M - R && loc < M) ? *A.pend(n, p, 1, loc - (M - R)) : (T)0;
        }
        // delays (lanes 0..3, then shared across the warp): this subdomain's
        // faces 0, 1; the left neighbour's face 1; the right neighbour's face 0
        int kk = 0;
        if (lane < 4) kk = A.delay(lane < 2 ? p : (lane == 2 ? pl : pr), lane < 2 ? lane : (lane == 2 ? 1 : 0));
        const int k0 = __shfl_sync(0xffffffffu, kk, 0), k1 = __shfl_sync(0xffffffffu, kk, 1);
        const int kl1 = __shfl_sync(0xffffffffu, kk, 2), kr0 = __shfl_sync(0xffffffffu, kk, 3);
        if (p != (int)blockIdx.x) __syncthreads();   // the previous subdomain's terms have been read
#pragma unroll
        for (int kp = 0; kp < kAdjPts; ++kp) {
            const int off = tid + kp * kAdjThreads, loc = chunk_lo + off;
            if (loc >= M) continue;
            T v[2 * R + 1];
            A.values(p, loc, k0, k1, v);
            T av = (T)0, bv = (T)0;
#pragma unroll
            for (int q = -R; q <= R; ++q) {
                av += (T)Coeffs<ORDER>::alpha(q) * v[q + R];
                bv += (T)Coeffs<ORDER>::beta(q) * v[q + R];
            }
            const T g = gl[kp];
#pragma unroll
            for (int j = -R; j <= R; ++j) {
                T d = A.cB * (T)Coeffs<ORDER>::beta(j) - A.cA * v[R] * (T)Coeffs<ORDER>::alpha(j);
                if (j == 0) d += (T)1 - A.cA * av;
                s_c[j + R][off] = g * d;
            }
            nu_acc += g * bv;
        }
        __syncthreads();
#pragma unroll
        for (int kp = 0; kp < kAdjPts; ++kp) {
            const int off = tid + kp * kAdjThreads, loc = chunk_lo + off;
            if (loc >= M) continue;
            const int i = p * M + loc;
            T v[2 * R + 1];
            T acc = (T)0;
            // readers r = i + d whose value j = -d is u^n_i
#pragma unroll
            for (int d = -R; d <= R; ++d) {
                const int rl = loc + d;
                if (rl >= 0 && rl < M) {
                    if (rl >= chunk_lo && rl < chunk_lo + kAdjChunk) {
                        acc += s_c[-d + R][off + d];
                    } else {
                        A.values(p, rl, k0, k1, v);
                        acc += A.gbar(i + d, -d, v);
                    }
                } else if (rl < 0) {
                    // the left neighbour's last points read u^n_i across their
                    // face 1; only an undelayed read lands on level n (with
                    // M >= 2R their stencils do not reach their own face 0)
                    if (kl1 == 0) {
                        A.values(pl, M + rl, -1, kl1, v);
                        acc += A.gbar(pl * M + M + rl, -d, v);
                    }
                } else if (kr0 == 0) {
                    A.values(pr, rl - M, kr0, -1, v);
                    acc += A.gbar(pr * M + (rl - M), -d, v);
                }
            }
            // delayed reads from later steps addressed to level n (loaded above)
            if (loc < R) {
                acc += pw[kp];
                *A.pend(n, p, 0, loc) = (T)0;
            } else if (loc >= M - R) {
                acc += pw[kp];
                *A.pend(n, p, 1, loc - (M - R)) = (T)0;
            }
            lam_out[i] = acc;

            // this subdomain's delayed reads across a face, scattered to older
            // levels of the neighbour's boundary values (one thread per face;
            // its readers are in its own chunk: the last chunk holds >= 4 points)
            if (loc == 0 || loc == M - 1) {
                const int f = loc == 0 ? 0 : 1;
                const int k = f == 0 ? k0 : k1;
                const int q = f == 0 ? pl : pr;
                T w[S_LEV];
                if constexpr (S_LEV == 2) {
                    w[0] = (T)(k + 1);
                    w[1] = (T)(-k);
                } else {
                    w[0] = (T)((k + 1) * (k + 2) / 2);
                    w[1] = (T)(-k * (k + 2));
                    w[2] = (T)(k * (k + 1) / 2);
                }
                // per source point of q: the sum of its readers' terms (source:
                // point M + t + j of q across face 0, j - t - 1 across face 1)
                T src[R];
#pragma unroll
                for (int r = 0; r < R; ++r) src[r] = (T)0;
#pragma unroll
                for (int t = 0; t < R; ++t) {
                    const int rt = f == 0 ? off + t : off - t;         // reader's place in the chunk
#pragma unroll
                    for (int j = -R; j <= R; ++j) {
                        const bool crosses = f == 0 ? (j <= -t - 1) : (j >= t + 1);
                        if (!crosses) continue;
                        src[f == 0 ? R + t + j : j - t - 1] += s_c[j + R][rt];
                    }
                }
                // older levels n-k-m of those points: all loads, then all stores
                const int side = f == 0 ? 1 : 0;
                T old[S_LEV][R];
#pragma unroll
                for (int m = 0; m < S_LEV; ++m)
#pragma unroll
                    for (int r = 0; r < R; ++r)
                        old[m][r] = (k + m == 0 || w[m] == (T)0) ? (T)0 : *A.pend(n - k - m, q, side, r);
#pragma unroll
                for (int m = 0; m < S_LEV; ++m) {
                    if (k + m == 0 || w[m] == (T)0) continue;     // level n: gathered above
#pragma unroll
                    for (int r = 0; r < R; ++r) *A.pend(n - k - m, q, side, r) = old[m][r] + w[m] * src[r];
                }
            }
        }
    }
    // dJ/dnu of this block: warp sums in the state's precision, then the
    // block's FP64 sum (one FP64 add per warp: FP64 is slow here)
    for (int o = 16; o > 0; o >>= 1) nu_acc += __shfl_xor_sync(0xffffffffu, nu_acc, o);
    if (lane == 0) red[tid >> 5] = nu_acc;
    __syncthreads();
    double sum = 0.0;
    if (tid == 0)
        for (int w = 0; w < kAdjThreads / 32; ++w) sum += (double)red[w] * (double)dtdx2;
    return sum;
}

// Grid barrier between the steps of an interval: every block arrives once
// per step (thread 0, after a block barrier and a fence) and waits for all;
// bounded by timeout_ns, after which the status and abort words are set and
// every block leaves.  Returns false on abort.
static __device__ __noinline__ bool adjoint_grid_sync(const AdjParams &a, unsigned long long target, long long n,
                                               int *s_ok)
{
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        atomicAdd(a.bar, 1ull);
        bool ok = true;
        if (ld_acquire(a.bar) < target) {
            const unsigned long long t0 = global_ns();
            for (;;) {
                __nanosleep(32);
                if (ld_acquire(a.bar) >= target) break;
                if (ld_relaxed(a.ctrl + kCtrlAbort)) { ok = false; break; }
                if ((long long)(global_ns() - t0) > a.timeout_ns) {
                    if (atomicCAS(a.ctrl + kCtrlStatus, 0, kStatusTimeout) == 0) {
                        a.ctrl[kCtrlCta] = (int)(blockIdx.y * gridDim.x + blockIdx.x);
                        a.ctrl[kCtrlWhere] = kWhereAdjoint;
                        a.ctrl[kCtrlNb] = -1;
                        a.ctrl[kCtrlStep] = (int)n;
                    }
                    atomicExch(a.ctrl + kCtrlAbort, 1);
                    ok = false;
                    break;
                }
            }
        }
        __threadfence();
        *s_ok = ok ? 1 : 0;
    }
    __syncthreads();
    return *s_ok != 0;
}

// The steps n_hi - 1 .. n_lo of one checkpoint interval in one cooperative
// launch (every block resident): lambda^{n_hi} in lam_a, lambda^{n_lo} in
// lam_a or lam_b after an even or odd number of steps.  Each block adds its
// dJ/dnu contribution of every step into its own FP64 running total, in the
// order of the steps.
template <typename T, int ORDER>
__global__ void __launch_bounds__(kAdjThreads, ORDER == 2 ? 7 : 3) at_adjoint_interval(const AdjParams a)
{
    constexpr int R = ORDER / 2;
    __shared__ T s_c[2 * R + 1][kAdjChunk];
    __shared__ T red[kAdjThreads / 32];
    __shared__ long long s_off[kAdjMaxLevels];
    __shared__ int s_ok;
    const int tid = threadIdx.x;
    unsigned long long arrivals = 0;
    const unsigned long long nblocks = (unsigned long long)gridDim.x * gridDim.y;
    for (long long n = a.n_hi - 1, it = 0; n >= a.n_lo; --n, ++it) {
        // word offsets of the levels n, n-1, ..., n-L-s+1 in the stored ring
        if (tid < kAdjMaxLevels) s_off[tid] = (n - tid >= 0) ? ((n - tid) % a.Dl) * a.N : 0;
        __syncthreads();
        const T *lam_in = reinterpret_cast<const T *>((it & 1) ? a.lam_b : a.lam_a);
        T *lam_out = reinterpret_cast<T *>((it & 1) ? a.lam_a : a.lam_b);
        const double sum = adjoint_level<T, ORDER>(a, n, s_off, lam_in, lam_out, s_c, red);
        // one add per block and step into the block's own running total: a
        // reduction without return (no load on the block's critical path)
        if (tid == 0) atomicAdd(a.dnu_part + (size_t)blockIdx.y * gridDim.x + blockIdx.x, sum);
        if (n > a.n_lo) {
            arrivals += nblocks;
            if (!adjoint_grid_sync(a, arrivals, n, &s_ok)) return;
        }
    }
}

// ---------------------------------------------------------------------------
// The interval kernel for one subdomain per warp (every subdomain's warp
// resident).  A level of at_adjoint_interval is a chain of a grid barrier, a
// block barrier and dependent global round trips (9.2 us a level of 2^20 points
// in 1024 subdomains when a block keeps its lambda in registers and prefetches
// what it can).  Here a warp keeps its subdomain's lambda in registers for the
// whole interval, in the stepper's lane-major layout, and the only thing it
// hears from its neighbours is one message per face and level:
//   * the adjoint of its halo values at level n (src: R words, from lambda^{n+1}
//     and u^n at its own edge points) goes out at the start of the level, as one
//     16-byte access with the level's tag (see st_entry in at_kernels.cuh);
//   * a warp that receives the message of level n adds w_m(k) src to its own
//     pending words of level n - k - m, k the neighbour's delay (prescribed, so
//     known to both sides): the pending ring is private, in shared memory;
//   * level n waits for the neighbours' messages of level n only where their
//     delay is 0, else for those of level n + 1 (one level of slack).
// The stored levels do not depend on lambda: the subdomain's tile comes in
// through a swizzled stage two levels ahead, the words its halos are
// extrapolated from one level ahead, the delays eight levels at a time.
// Same terms as at_adjoint_interval; the pending words are added last.
// 2^20 points in 1024 subdomains of 1024, FP32, order 2: 9.25 us a level then,
// 2.2 us so (6.7 warps per SM, so a level's latency, not its 27 instructions a
// point, sets the pace); forward and backward over 200 levels 3.32 and 1.88 ms.

// Shared memory of a warp: `stages` tiles, the halo levels, the pending words.
__host__ __device__ inline long long adjoint_warp_smem(long long stage_bytes, int stages, int R, int word, int Tp)
{
    return stages * stage_bytes + round_up(kRawBytes, 128) + round_up(2LL * Tp * R * word, 128);
}
constexpr int kAdjStages = 3;
constexpr int kAdjMsgSlots = 8;      // levels of messages kept (a neighbour is at most 2 levels away)

template <typename T, int ORDER, int GW, bool FULL>
__global__ void __launch_bounds__(kThreads, sizeof(T) == 4 ? 3 : 2) at_adjoint_warp(const AdjParams a)
{
    constexpr int R = ORDER / 2;
    constexpr int S_LEV = ORDER / 2 + 1;
    constexpr unsigned kAll = 0xffffffffu;
    constexpr int NH = entry_halves<T, ORDER, 0>();
    constexpr int kEnt = kRingHalf * NH;
    constexpr int CPG = (int)sizeof(T) / 4, WPC = 16 / (int)sizeof(T), NPT = 4 * GW, NCH = GW * CPG;
    extern __shared__ __align__(128) unsigned char smem[];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int my_face = lane >> 4, my_m = lane & 15;
    const int P = (int)a.P, M = (int)a.M;
    const long long e = (long long)blockIdx.x * kWarps + w, E = (long long)gridDim.x * kWarps;
    const int p = (int)(e * P / E);
    if ((e + 1) * P / E == p) return;                    // (no subdomain)
    if (p == 0 && a.n_hi <= a.stop_below) return;
    const int nb = my_face ? (p == P - 1 ? 0 : p + 1) : (p == 0 ? P - 1 : p - 1);   // across this lane's face
    unsigned char *base = smem + (size_t)w * adjoint_warp_smem(a.stage_bytes, kAdjStages, R, (int)sizeof(T), a.Tp);
    unsigned char *raw = base + kAdjStages * a.stage_bytes;
    T *pend = reinterpret_cast<T *>(raw + round_up(kRawBytes, 128));              // [Tp][2][R]
    const int gpl = FULL ? GW : a.gpl;
    const int NG = M / 4, lane_last = (NG - 1) / gpl, m_last = FULL ? GW - 1 : (NG - 1) - lane_last * gpl;
    const bool is_first = lane == 0, is_last = lane == lane_last;
    const Swizzle swz = FULL ? Swizzle::of(NCH) : Swizzle{a.swz_shift, a.swz_mask};
    auto own_chunk = [&](int k) -> int { return FULL ? lane_chunk<NCH>(lane, k) : 16 * swz(gpl * CPG * lane + k); };
    const T cA = sizeof(T) == 4 ? (T)a.cAf : (T)a.cA, cB = sizeof(T) == 4 ? (T)a.cBf : (T)a.cB;
    const T *lev = reinterpret_cast<const T *>(a.levels);
    const int Dl = (int)a.Dl;
    const int n_lev = (int)(a.n_hi - a.n_lo);
    const unsigned pmask = (unsigned)a.Tp - 1u;

    // the pending words of this subdomain
    T *pend_g = reinterpret_cast<T *>(a.pend);
    for (int i = lane; i < 2 * a.Tp * R; i += 32) {
        const int t = i / (2 * R), r = i - t * 2 * R;
        pend[i] = pend_g[((size_t)t * P + p) * 2 * R + r];
    }
    // lambda^{n_hi}
    T lam[NPT];
    T *lg = reinterpret_cast<T *>(a.lam_a) + (size_t)p * M;
#pragma unroll
    for (int m = 0; m < GW; ++m) {
        const int g = gpl * lane + m;
        const bool live = m < gpl && g < NG;
#pragma unroll
        for (int q = 0; q < 4; ++q) lam[4 * m + q] = live ? lg[4 * g + q] : (T)0;
    }
    // slot of level l of the stored levels, l = n_hi - 1 - i
    const int slot_hi = (int)((a.n_hi - 1) % a.Dl);
    auto level_slot = [&](int back) -> int {            // back: levels below n_hi - 1
        int s = slot_hi - back % Dl;
        return s < 0 ? s + Dl : s;
    };
    // --- the tile of level n_hi - 1 - i into its stage
    const int nc = (int)((size_t)M * sizeof(T) / 16);
    auto load_tile = [&](int i) {
        if (i < n_lev) {
            unsigned char *dst = base + (i % kAdjStages) * a.stage_bytes;
            const unsigned char *src =
                reinterpret_cast<const unsigned char *>(lev + (size_t)level_slot(i) * a.N + (size_t)p * M) + 16 * lane;
#pragma unroll
            for (int t = 0; t < NCH; ++t)
                if (lane + 32 * t < nc) cp_async16(dst + swz.coalesced(lane, t), src + 512 * t);
        }
        cp_async_commit();
    };
    // --- delays: lane 4 i + b holds byte b of level n_hi - 1 - (t0 + i): the left
    // neighbour's face 1, this subdomain's faces 0 and 1, the right neighbour's face 0
    auto load_delays = [&](int t0) -> int {
        const long long i = t0 + (lane >> 2);
        if (i >= n_lev) return 0;
        const int b = lane & 3;
        const long long at = b == 0 ? (p == 0 ? 2LL * P - 1 : 2LL * p - 1)
                                    : b == 3 ? (p == P - 1 ? 0 : 2LL * p + 2) : 2LL * p + b - 1;
        const long long n = a.n_hi - 1 - i;
        int k = a.delays[(n - a.k_level) * 2 * P + at];
        // (clamped as the forward run clamps it)
        long long kmax = n - S_LEV + 1;
        kmax = kmax < 0 ? 0 : kmax > a.L ? a.L : kmax;
        return k > kmax ? (int)kmax : k < 0 ? 0 : k;
    };
    int kb = load_delays(0), kb_next = load_delays(8);
    auto delay = [&](int i, int b) -> int {               // of level n_hi - 1 - i, in the current batch
        return __shfl_sync(kAll, kb, 4 * (i & 7) + b);
    };
    // --- the words this face's halo of level i is extrapolated from: lane m < s
    // reads level n - k - m
    T hw[R];
    auto load_halo = [&](int i, int k) {
        if (my_m < S_LEV && (my_m == 0 || k != 0)) {
            const T *src = lev + (size_t)level_slot(i + k + my_m) * a.N + (size_t)nb * M + (my_face ? 0 : M - R);
#pragma unroll
            for (int q = 0; q < R; ++q) hw[q] = ld_cg(src + q);
        }
    };
    // --- messages: the neighbour's facing one of level i
    const unsigned char *msg_in = a.msg + ((size_t)nb * 2 + (1 - my_face)) * kEnt;
    unsigned char *msg_out = a.msg + (size_t)p * 2 * kEnt;
    const size_t msg_stride = (size_t)P * 2 * kEnt;
    unsigned long long md[NH], mt[NH];
    auto msg_tag = [&](int i) { return entry_tag(a.n_hi - 1 - i); };
    auto read_msg = [&](bool on, int i) {
        ld_tagged<NH>(on, msg_in + (size_t)((unsigned)(a.n_hi - 1 - i) & (kAdjMsgSlots - 1)) * msg_stride, md, mt);
    };
    auto msg_there = [&](int i) -> bool {
        bool ok = true;
#pragma unroll
        for (int h = 0; h < NH; ++h) ok = ok && mt[h] == msg_tag(i);
        return ok;
    };
    // adds the message of level i (this face's neighbour had delay k there) to
    // the pending words: lane m < s the level n - k - m
    auto apply_msg = [&](bool on, int i, int k) {
        if (on && my_m < S_LEV) {
            T wt;
            if constexpr (S_LEV == 2) wt = my_m == 0 ? (T)(k + 1) : (T)(-k);
            else wt = my_m == 0 ? (T)((k + 1) * (k + 2) / 2) : my_m == 1 ? (T)(-k * (k + 2)) : (T)(k * (k + 1) / 2);
            if (wt != (T)0) {
                T *d = pend + ((size_t)((unsigned)(a.n_hi - 1 - i - k - my_m) & pmask) * 2 + my_face) * R;
                T s[R];
                if constexpr (sizeof(T) == 8) {
#pragma unroll
                    for (int q = 0; q < R; ++q) s[q] = (T)__longlong_as_double((long long)md[q < NH ? q : 0]);
                } else {
#pragma unroll
                    for (int q = 0; q < R; ++q) s[q] = (T)__uint_as_float((unsigned)(md[0] >> (32 * q)));
                }
#pragma unroll
                for (int q = 0; q < R; ++q) d[q] += wt * s[q];
            }
        }
        __syncwarp();
    };
    // Receives the message of level i where `want` (bounded wait); returns
    // false on abort.  (md, mt: a read of it, perhaps too early)
    auto receive = [&](bool want, int i, int k) -> bool {
        if (!__all_sync(kAll, !want || msg_there(i))) {
            const unsigned long long t0 = global_ns();
            for (int polls = 0;; ++polls) {
                const bool miss = want && !msg_there(i);
                if (miss) read_msg(true, i);
                if (__all_sync(kAll, !want || msg_there(i))) break;
                if ((polls & 15) == 15) {
                    const bool late = (long long)(global_ns() - t0) > a.timeout_ns;
                    if (__any_sync(kAll, late || ld_relaxed(a.ctrl + kCtrlAbort) != 0)) {
                        // (any lane that misses it reports it: each reads for itself;
                        // the first report stands)
                        if (miss) {
                            if (atomicCAS(a.ctrl + kCtrlStatus, 0, kStatusTimeout) == 0) {
                                a.ctrl[kCtrlCta] = (int)blockIdx.x;
                                a.ctrl[kCtrlWhere] = kWhereAdjoint;
                                a.ctrl[kCtrlNb] = nb;
                                a.ctrl[kCtrlStep] = (int)(a.n_hi - 1 - i);
                            }
                            atomicExch(a.ctrl + kCtrlAbort, 1);
                        }
                        return false;
                    }
                    if (polls > 64) __nanosleep(64);
                }
            }
        }
        apply_msg(want, i, k);
        return true;
    };

    load_tile(0);
    load_tile(1);
    load_halo(0, delay(0, 1 + my_face));
    double nu_sum = 0.0;
    bool late_msg = false;              // this face's message of the level before is still to come
    int k_late = 0;                     // the neighbour's delay there
    bool ok = true;
    for (int i = 0; i < n_lev; ++i) {
        const long long n = a.n_hi - 1 - i;
        if (i > 0 && (i & 7) == 0) {
            kb = kb_next;
            kb_next = load_delays(i + 8);
        }
        const int k_own = delay(i, 1 + my_face);         // of this face
        const int k_nb = delay(i, my_face ? 3 : 0);      // of the neighbour's facing face
        // --- u^n: tile and halos
        load_tile(i + 2);
        if (my_m < S_LEV) {
            T *r = reinterpret_cast<T *>(raw + my_face * kRawFace + my_m * kRawEntry);
#pragma unroll
            for (int q = 0; q < R; ++q) r[q] = hw[q];
        }
        cp_async_wait(2);
        __syncwarp();
        T hv = (T)0;
        if (my_m < R) hv = approx_halo<T, S_LEV>(raw + my_face * kRawFace, k_own, my_m);
        const unsigned char *stage = base + (i % kAdjStages) * a.stage_bytes;
        T u[NPT];
#pragma unroll
        for (int m = 0; m < GW; ++m) {
            // (FULL: the stage has room for the lanes beyond the tile)
            const bool has = FULL || (m < gpl && gpl * lane + m < NG);
#pragma unroll
            for (int h = 0; h < CPG; ++h) {
                T *d = u + 4 * m + h * WPC;
                if (has) lds<T, WPC>(reinterpret_cast<const T *>(stage + own_chunk(m * CPG + h)), d);
                else
#pragma unroll
                    for (int q = 0; q < WPC; ++q) d[q] = (T)0;
            }
        }
        // --- the words of u and lambda at the run's edges
        T tu[R], tl[R];                                  // last words of the lane's run
        T eu[R], el[R];                                  // last words of the tile (its owner's)
#pragma unroll
        for (int q = 0; q < R; ++q) {
            tu[q] = eu[q] = u[NPT - R + q];
            tl[q] = el[q] = lam[NPT - R + q];
            if constexpr (!FULL) {
#pragma unroll
                for (int m = 0; m < GW; ++m) {
                    if (m == gpl - 1) { tu[q] = u[4 * m + 4 - R + q]; tl[q] = lam[4 * m + 4 - R + q]; }
                    if (m == m_last) { eu[q] = u[4 * m + 4 - R + q]; el[q] = lam[4 * m + 4 - R + q]; }
                }
            }
        }
        // --- the adjoint of this subdomain's halo values at level n, out to the
        // neighbours: c_j = lambda (cB beta_j - cA u alpha_j) of the points next
        // to each face
        {
            T s0[R], s1[R];
            auto c = [&](T l, T uu, int j) -> T {
                return l * (cB * (T)Coeffs<ORDER>::beta(j) - cA * uu * (T)Coeffs<ORDER>::alpha(j));
            };
            if constexpr (R == 1) {
                s0[0] = c(lam[0], u[0], -1);
                s1[0] = c(el[0], eu[0], 1);
            } else {
                s0[0] = c(lam[0], u[0], -2);
                s0[R - 1] = c(lam[0], u[0], -1) + c(lam[1], u[1], -2);
                s1[0] = c(el[R - 1], eu[R - 1], 1) + c(el[0], eu[0], 2);
                s1[R - 1] = c(el[R - 1], eu[R - 1], 2);
            }
            unsigned char *o = msg_out + (size_t)((unsigned)n & (kAdjMsgSlots - 1)) * msg_stride;
            st_entry<T, ORDER, 0>(is_first, o, s0, s0, msg_tag(i));
            st_entry<T, ORDER, 0>(is_last, o + kEnt, s1, s1, msg_tag(i));
        }
        // --- the message of the level before, where the neighbour's delay let
        // it come later; a first read of this level's
        if (__any_sync(kAll, late_msg)) {
            read_msg(late_msg, i - 1);
            if (!receive(late_msg, i - 1, k_late)) { ok = false; break; }
        }
        read_msg(true, i);
        if (i + 1 < n_lev) {
            const int kx = __shfl_sync(kAll, ((i + 1) & 7) == 0 ? kb_next : kb, 4 * ((i + 1) & 7) + 1 + my_face);
            load_halo(i + 1, kx);
        }
        // --- lambda^n inside the subdomain
        T ul[R], ur[R], ll[R], lr[R], hr[R];
#pragma unroll
        for (int q = 0; q < R; ++q) {
            const T h = __shfl_sync(kAll, hv, (is_first ? 0 : 16) + q);   // lane 0: left halo; others: right halo
            hr[q] = __shfl_sync(kAll, hv, 16 + q);
            ul[q] = __shfl_up_sync(kAll, tu[q], 1);
            ur[q] = __shfl_down_sync(kAll, u[q], 1);
            ll[q] = __shfl_up_sync(kAll, tl[q], 1);
            lr[q] = __shfl_down_sync(kAll, lam[q], 1);
            ul[q] = is_first ? h : ul[q];
            ll[q] = is_first ? (T)0 : ll[q];
            if constexpr (FULL) {
                ur[q] = is_last ? hr[q] : ur[q];
                lr[q] = is_last ? (T)0 : lr[q];
            }
        }
        T nu_acc = (T)0;
#pragma unroll
        for (int m = 0; m < GW; ++m) {
            if (!FULL && m >= gpl) break;
            // u and lambda^{n+1} of the group and R points on either side
            T U[4 + 2 * R], G[4 + 2 * R];
#pragma unroll
            for (int q = 0; q < R; ++q) {
                U[q] = ul[q];
                G[q] = ll[q];
                U[R + 4 + q] = m + 1 < GW ? u[4 * (m + 1 < GW ? m + 1 : m) + q] : ur[q];
                G[R + 4 + q] = m + 1 < GW ? lam[4 * (m + 1 < GW ? m + 1 : m) + q] : lr[q];
                if constexpr (!FULL) {
                    if (m >= m_last) {
                        if (m == gpl - 1) { U[R + 4 + q] = ur[q]; G[R + 4 + q] = lr[q]; }
                        if (m == m_last && is_last) { U[R + 4 + q] = hr[q]; G[R + 4 + q] = (T)0; }
                    }
                }
                ul[q] = u[4 * m + 4 - R + q];
                ll[q] = lam[4 * m + 4 - R + q];
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) { U[R + q] = u[4 * m + q]; G[R + q] = lam[4 * m + q]; }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                T av = (T)0, bv = (T)0;
#pragma unroll
                for (int j = -R; j <= R; ++j) {
                    if (j != 0) av += (T)Coeffs<ORDER>::alpha(j) * U[R + q + j];
                    bv += (T)Coeffs<ORDER>::beta(j) * U[R + q + j];
                }
                T acc = (T)0;
#pragma unroll
                for (int d = -R; d <= R; ++d) {          // reader q + d, whose value j = -d this point is
                    const int x = R + q + d;
                    T t = cB * (T)Coeffs<ORDER>::beta(-d);
                    if (d != 0) t -= cA * U[x] * (T)Coeffs<ORDER>::alpha(-d);
                    else t += (T)1 - cA * av;
                    acc += G[x] * t;
                }
                // (points beyond the tile stay 0)
                const bool live = FULL || gpl * lane + m < NG;
                if constexpr (!FULL) acc = live ? acc : (T)0;
                nu_acc += live ? G[R + q] * bv : (T)0;
                lam[4 * m + q] = acc;
            }
        }
        nu_sum += lane <= lane_last ? (double)nu_acc : 0.0;
        // --- this level's messages: where the neighbour's delay is 0, and
        // where they are there already; then the pending words of level n
        {
            const bool here = msg_there(i);
            const bool now = k_nb == 0 || here;
            const unsigned bal = __ballot_sync(kAll, now);
            // (one decision per face)
            const bool want = ((bal >> (lane & 16)) & 0xffffu) == 0xffffu || k_nb == 0;
            if (!receive(want, i, k_nb)) { ok = false; break; }
            late_msg = !want;
            k_late = k_nb;
        }
        {
            T *pw = pend + (size_t)((unsigned)n & pmask) * 2 * R;
            T p0[R], p1[R];
#pragma unroll
            for (int q = 0; q < R; ++q) { p0[q] = pw[q]; p1[q] = pw[R + q]; }
            __syncwarp();
            if (lane < 2 * R) pw[lane] = (T)0;
            __syncwarp();
#pragma unroll
            for (int q = 0; q < R; ++q) {
                if (is_first) lam[q] += p0[q];
#pragma unroll
                for (int m = 0; m < GW; ++m)
                    if (FULL ? m == GW - 1 : m == m_last)
                        if (is_last) lam[4 * m + 4 - R + q] += p1[q];
            }
        }
    }
    // the last level's messages belong to the pending words of the levels below
    if (ok && __any_sync(kAll, late_msg)) {
        read_msg(late_msg, n_lev - 1);
        receive(late_msg, n_lev - 1, k_late);
    }
    cp_async_wait(0);
    __syncwarp();
    if (!ok) return;
#pragma unroll
    for (int m = 0; m < GW; ++m) {
        const int g = gpl * lane + m;
        // (word by word: the caller's array may start at any word)
        if (m < gpl && g < NG)
#pragma unroll
            for (int q = 0; q < 4; ++q) lg[4 * g + q] = lam[4 * m + q];
    }
    for (int i = lane; i < 2 * a.Tp * R; i += 32) {
        const int t = i / (2 * R), r = i - t * 2 * R;
        pend_g[((size_t)t * P + p) * 2 * R + r] = pend[i];
    }
    for (int o = 16; o > 0; o >>= 1) nu_sum += __shfl_xor_sync(kAll, nu_sum, o);
    if (lane == 0) a.dnu_part[p] += nu_sum * a.dtdx2;
}

}  // namespace atk
