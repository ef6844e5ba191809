// at_resident.cuh -- the 1D stepper with one subdomain per CTA and prescribed
// delays (AT_SEEDED, AT_REPLAY), for launches whose CTAs can hold every
// subdomain at once.
//
// There the whole state lives in registers and a launch is a chain of
// hand-overs: level n of a subdomain needs the neighbours' level n (delay 0) or
// older ones, so what counts is the time from a neighbour's boundary value to
// this one's, not throughput.  The general stepper gives such a subdomain one
// warp, which spends some 400 integer and control instructions a level on
// tiles, passes and cursors, and with FP64 state one SM partition's share of the
// FP64 pipe, 73 cycles an instruction (2.9 us a level of 16 subdomains of 256
// points).  Here the points are spread over up to 8 warps (PPT a thread: 1 to
// 128 points, else about M / 128), on all four partitions, and a level is: check
// the ring entries read ahead and extrapolate them with shuffles (the warps that
// own a face), exchange R words between neighbouring warps through shared memory
// (one CTA barrier) and between lanes by shuffles, compute, publish, read ahead.
// Same update, entries, tags and delay statistics as at_stepper, bit for bit; the
// two may follow each other on one solver.
//
// A step of 16 subdomains of 256 FP64 points, order 2: 2.83 us in the general
// stepper, 1.99 with one lean warp a subdomain, 1.34 so; of 64 points, order 4,
// forced: 3.0 and 1.5; 1024 subdomains of 1024 FP32 points, every level stored:
// 1.95 and 1.3.
#pragma once

#include "at_kernels.cuh"

namespace atk {

// points per thread of the resident stepper for subdomains of M points (a
// multiple of 4, at most 1024): 1, 2, 4 or 8, at most 128 threads where the count
// divides M, else 4 and at most 255
__host__ __device__ inline int resident_points(long long M)
{
    int ppt = 1;
    while (ppt * 128 < M) ppt <<= 1;
    return M % ppt == 0 ? ppt : 4;
}
__host__ __device__ inline int resident_threads(long long M)
{
    return (int)((M / resident_points(M) + 31) / 32 * 32);
}

// CL: up to kMaxCluster subdomains, the CTAs one cluster.  A boundary value goes
// straight into the shared memory of the CTA that reads it, and the ring in global
// memory takes only the levels a later launch may read: what a level waits for is
// then one store across the SMs instead of a store to the L2 cache and the loads
// that find it there.  An entry is two 8-byte words, each half of the payload with
// 32 bits of tag, so that each is whole by itself.  16 subdomains of 256 FP64
// points, order 2, 1000 levels: 1421 us through the L2 cache, 1140 so; of 64 points,
// order 4, forced, 120 levels: 207 and 187.
constexpr int kMaxCluster = 16;
constexpr int kClusterSlots = 64;          // ring_slots(kMaxL, kMaxS)

__device__ __forceinline__ void cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}

// shared-memory address of this CTA's `addr` in CTA `rank` of the cluster
__device__ __forceinline__ unsigned cluster_addr(unsigned addr, int rank)
{
    unsigned r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}

__device__ __forceinline__ void st_half(unsigned addr, unsigned long long payload, unsigned tag)
{
    const unsigned long long t = (unsigned long long)tag << 32;
    asm volatile("st.relaxed.cluster.shared::cluster.v2.u64 [%0], {%1, %2};"
                 ::"r"(addr), "l"(t | (payload & 0xffffffffull)), "l"(t | (payload >> 32)) : "memory");
}

// (tag 0, no level's: off, or the two words of different levels)
__device__ __forceinline__ void ld_half(bool on, unsigned addr, unsigned long long *payload, unsigned long long *tag)
{
    unsigned long long a = 0, b = 0;
    if (on)
        asm volatile("ld.relaxed.cluster.shared::cta.v2.u64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "r"(addr) : "memory");
    *payload = (a & 0xffffffffull) | (b << 32);
    *tag = (a >> 32) == (b >> 32) ? a >> 32 : 0;
}

template <typename T, int ORDER, int PPT, bool FORCED, bool CL>
__global__ void __launch_bounds__(256) at_resident(const Params p)
{
    constexpr int R = ORDER / 2;
    constexpr int S_LEV = ORDER / 2 + 1;
    constexpr unsigned kAll = 0xffffffffu;
    constexpr int NH = entry_halves<T, ORDER, 0>();
    constexpr int kEnt = kRingHalf * NH;
    constexpr bool PLAIN = sizeof(T) == 4 && ORDER == 2 && !FORCED;     // (as the general stepper)
    __shared__ T s_edge[2][8][2][R];           // [level parity][warp][first | last R words]
    // level whose wait ran out.  (With a mere flag, a warp past a level's barrier could
    // set it for the next level before a slower warp has read it for this one; that
    // warp would leave a barrier early, for the last ones, which are not bounded.)
    __shared__ int s_abort;
    __shared__ T s_kt[kMaxL + 1][2];           // k and k (k + 1) / 2 in the state's type
    __shared__ ulonglong2 s_ring[CL ? kClusterSlots * 2 * NH : 1];      // [slot][face][half]: the neighbours' words
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int M = (int)p.M, P = (int)p.P, NTH = M / PPT, n_warps = (NTH + 31) / 32;
    const int pj = (int)blockIdx.x;
    const long long n0 = *reinterpret_cast<const volatile long long *>(p.ctrl + kCtrlN0);
    const int n_steps = (int)p.n_steps;
    const bool w_first = w == 0, w_last = w == n_warps - 1, live = tid < NTH;
    const int ll = w_last ? (NTH - 1) & 31 : 31;                         // last lane with points
    // halo work: lane 16 f + 4 q + m reads word q of level n - k - m across face
    // f, in the warp that owns the face
    const int f = lane >> 4, hq = (lane >> 2) & 3, hm = lane & 3;
    const bool h_own = (f == 0 ? w_first : w_last) && hq < R && hm < S_LEV;
    const int nb = f ? (pj + 1 == P ? 0 : pj + 1) : (pj == 0 ? P - 1 : pj - 1);
    const unsigned tmask = (unsigned)p.T - 1u, slot_stride = (unsigned)(P * 2 * kEnt);
    const unsigned n0lo = (unsigned)n0;
    const unsigned char *ring_in = p.ring + (size_t)(nb * 2 + (1 - f)) * kEnt + (NH == 2 ? hq * kRingHalf : 0);
    unsigned char *ring_out = p.ring + (size_t)pj * 2 * kEnt;
    // (CL: tags count from 64, the oldest level read is n0 - L - s + 1)
    const unsigned long long tag0 = CL ? 64ull : entry_tag(n0);
    const unsigned ring_sm = smem_addr(s_ring);
    const unsigned half_in = ring_sm + (unsigned)(f * NH + (NH == 2 ? hq : 0)) * 16u;
    // this CTA's entries in the neighbours' shared memory, at slot 0: face 0 of this
    // subdomain is across face 1 of the left one
    const unsigned out0 = CL ? cluster_addr(ring_sm + 16u * NH, pj == 0 ? P - 1 : pj - 1) : 0u;
    const unsigned out1 = CL ? cluster_addr(ring_sm, pj + 1 == P ? 0 : pj + 1) : 0u;
    const T cA = sizeof(T) == 4 ? (T)p.cA32 : (T)p.cA, cr = sizeof(T) == 4 ? (T)p.cr32 : (T)p.cr;
    const StencilK<T, ORDER, 0, PLAIN> K(cA, cr, p);

    // the state, and the forcing of this thread's points
    T v[PPT], F[FORCED ? PPT : 1];
    T *ug = reinterpret_cast<T *>(p.u) + (size_t)pj * M + tid * PPT;
#pragma unroll
    for (int i = 0; i < PPT; ++i) v[i] = live ? ug[i] : (T)0;
    if constexpr (FORCED) {
        // (as the general stepper forms it: FP64 sin/cos of the offset and of the
        // subdomain's origin, rounded to the state's words)
        double so, co;
        sincos(p.x0 + (double)((long long)pj * M) * p.dx, &so, &co);
        const T fX = sizeof(T) == 4 ? (T)p.fX32 : (T)p.fX;
        const T fs = fX * (T)so, fc = fX * (T)co;
#pragma unroll
        for (int i = 0; i < PPT; ++i) {
            double sv, cv;
            sincos((double)(tid * PPT + i) * p.dx, &sv, &cv);
            F[i] = forcing_point(fs, fc, (T)sv, (T)cv);
        }
    }
    if (tid <= kMaxL) {
        s_kt[tid][0] = (T)tid;
        s_kt[tid][1] = (T)(tid * (tid + 1) / 2);
    }
    if (tid == 0) s_abort = 0x7fffffff;
    if constexpr (CL) {
        // the levels a halo may use that are there already, from the global ring
        // (unread ones empty), before any neighbour stores into this one
        for (int i = tid; i < kClusterSlots * 2 * NH; i += (int)blockDim.x) s_ring[i] = make_ulonglong2(0, 0);
        __syncthreads();
        for (int i = tid; i < (p.L + S_LEV) * 2 * NH; i += (int)blockDim.x) {
            const int back = i / (2 * NH), fi = (i / NH) & 1, half = i % NH;
            const int from = fi ? (pj + 1 == P ? 0 : pj + 1) : (pj == 0 ? P - 1 : pj - 1);
            const unsigned slot = (n0lo - (unsigned)back) & tmask;
            unsigned long long pay, tag;
            ld_tagged<1>(true, p.ring + (size_t)slot * slot_stride + (size_t)(from * 2 + (1 - fi)) * kEnt + half * kRingHalf,
                         &pay, &tag);
            if (back <= n0 && tag == entry_tag(n0 - back))
                st_half(ring_sm + ((slot * 2u + (unsigned)fi) * NH + (unsigned)half) * 16u, pay, (unsigned)(tag0 - back));
        }
        cluster_sync();
    }

    // --- prescribed delays, 16 levels at a time: lane 2 i + face, level i of the batch
    auto draw = [&](int i0) -> int {
        const int i = i0 + (lane >> 1);
        int k = 0;
        if (i < n_steps) {
            const long long n = n0 + i;
            if (p.mode == kModeSeeded) k = seeded_delay(p.seed, n, pj, p.P, p.per_sub ? 0 : (lane & 1), p.L);
            else k = p.delays[((long long)i * P + pj) * 2 + (lane & 1)];
            // (no level below 0 is read, at most L)
            const long long ks = n - S_LEV + 1;
            const int kmax = ks < 0 ? 0 : ks < p.L ? (int)ks : p.L;
            k = k < 0 ? 0 : k < kmax ? k : kmax;
        }
        return k;
    };
    int kb = 0, kb_next = 0;
    unsigned cnt_k = 0, cnt16 = 0;        // levels with delay hc (and 16) on this face
    const int hc = lane & 15;
    unsigned long long hd = 0, ht = 0, h_tag = 0;
    const unsigned char *h_at = ring_in;
    unsigned h_half = half_in;
    bool h_act = false;
    int h_k = 0;
    auto read_ahead = [&](int i, int k) {
        h_k = k;
        h_act = h_own && (hm == 0 || k != 0);
        const int d = i - k - hm;
        h_tag = tag0 + (long long)d;
        const unsigned slot = (n0lo + (unsigned)d) & tmask;
        if constexpr (CL) {
            h_half = half_in + slot * (2u * NH * 16u);
            ld_half(h_act, h_half, &hd, &ht);
        } else {
            h_at = ring_in + slot * slot_stride;
            ld_tagged<1>(h_act, h_at, &hd, &ht);
        }
    };
    auto wait_entries = [&](int i) -> bool {
        const unsigned long long t0 = global_ns();
        for (int polls = 0;; ++polls) {
            const bool miss = h_act && ht != h_tag;
            if constexpr (CL) {
                if (miss) ld_half(true, h_half, &hd, &ht);
            } else {
                if (miss) ld_tagged<1>(true, h_at, &hd, &ht);
            }
            if (__all_sync(kAll, !h_act || ht == h_tag)) return true;
            if ((polls & 15) == 15) {
                const bool late = (long long)(global_ns() - t0) > p.timeout_ns;
                if (__any_sync(kAll, late || ld_relaxed(p.ctrl + kCtrlAbort) != 0)) {
                    // (any lane that misses its words reports it: the newest
                    // level may be there and another's half be missing; the first
                    // report stands)
                    if (miss) raise_timeout(p, kWhereFlag, n0 + i, nb);
                    return false;
                }
                if (polls > 256) __nanosleep(64);
            }
        }
    };
    // the words other warps need: the first and last R of this warp's run
    auto put_edges = [&](int par) {
        if constexpr (PPT >= R) {
#pragma unroll
            for (int q = 0; q < R; ++q) {
                if (lane == 0) s_edge[par][w][0][q] = v[q];
                if (lane == ll) s_edge[par][w][1][q] = v[PPT - R + q];
            }
        } else {
            if (lane < R) s_edge[par][w][0][lane] = v[0];
            if (lane > ll - R && lane <= ll) s_edge[par][w][1][lane - (ll - R + 1)] = v[0];
        }
    };
    const bool edge_warp = w_first || w_last;
    if (edge_warp) {
        kb = draw(0);
        read_ahead(0, __shfl_sync(kAll, kb, f));
    }
    if (n_warps > 1) put_edges(0);
    __syncthreads();
    // (test knob: CTA 0 takes no part in a launch that goes beyond level skip_step)
    bool ok = !(p.skip_publish && pj == 0 && n0 + n_steps > p.skip_step);
    if (ok)
    for (int i = 0; i < n_steps; ++i) {
        const int par = i & 1;
        // the R words left and right of the warp's run
        T lw[R], rw[R];
        if (edge_warp) {
            // the next batch of delays, a few levels before it is needed
            if ((i & 15) == 8) kb_next = draw((i & ~15) + 16);
            const int k = h_k;
            if (!__all_sync(kAll, !h_act || ht == h_tag)) {
                if (!wait_entries(i)) { ok = false; if (lane == 0) *reinterpret_cast<volatile int *>(&s_abort) = i; }
            }
            if (f == 0 ? w_first : w_last) {
                cnt_k += hc == k ? 1u : 0u;
                if (p.L > 15) cnt16 += (hc == 0 && k == 16) ? 1u : 0u;
                if (p.delays && p.mode == kModeSeeded && hc == 0)
                    p.delays[((long long)i * P + pj) * 2 + f] = (int8_t)k;
            }
            // the halo words (Newton form, see approx_halo), in lanes 16 f + 4 q
            T r0;
            if constexpr (sizeof(T) == 8) r0 = (T)__longlong_as_double((long long)hd);
            else r0 = (T)__uint_as_float((unsigned)(hd >> (32 * (hq & 1))));
            const T r1 = __shfl_down_sync(kAll, r0, 1), d1 = r0 - r1;
            T h;
            if constexpr (S_LEV == 2) {
                h = r0 + s_kt[k][0] * d1;
            } else {
                const T r2 = __shfl_down_sync(kAll, r0, 2);
                const T d2 = d1 - (r1 - r2);
                h = r0 + (s_kt[k][0] * d1 + s_kt[k][1] * d2);
            }
            h = k == 0 ? r0 : h;
#pragma unroll
            for (int q = 0; q < R; ++q) {
                lw[q] = __shfl_sync(kAll, h, 4 * q);
                rw[q] = __shfl_sync(kAll, h, 16 + 4 * q);
            }
        }
        if (n_warps > 1) {
            __syncthreads();
            if (*reinterpret_cast<volatile int *>(&s_abort) <= i) { ok = false; break; }
#pragma unroll
            for (int q = 0; q < R; ++q) {
                if (!w_first) lw[q] = s_edge[par][w - 1][1][q];
                if (!w_last) rw[q] = s_edge[par][w + 1][0][q];
            }
        } else if (!ok) {
            break;
        }
        // the window: R words left, the thread's points, R words right
        T W[PPT + 2 * R];
        if constexpr (PPT >= R) {
#pragma unroll
            for (int q = 0; q < R; ++q) {
                const T l = __shfl_up_sync(kAll, v[PPT - R + q], 1), r = __shfl_down_sync(kAll, v[q], 1);
                W[q] = lane == 0 ? lw[q] : l;
                W[R + PPT + q] = lane == ll ? rw[q] : r;
            }
        } else {
            // (one point a thread, R = 2)
            const T l1 = __shfl_up_sync(kAll, v[0], 1), l2 = __shfl_up_sync(kAll, v[0], 2);
            const T r1 = __shfl_down_sync(kAll, v[0], 1), r2 = __shfl_down_sync(kAll, v[0], 2);
            W[0] = lane == 0 ? lw[0] : lane == 1 ? lw[R - 1] : l2;
            W[R - 1] = lane == 0 ? lw[R - 1] : l1;
            W[R + 1] = lane == ll ? rw[0] : r1;
            W[2 * R] = lane == ll ? rw[R - 1] : lane == ll - 1 ? rw[0] : r2;
        }
#pragma unroll
        for (int q = 0; q < PPT; ++q) W[R + q] = v[q];
#pragma unroll
        for (int q = 0; q < PPT; ++q) v[q] = K.template point<FORCED>(W + q, FORCED ? F[FORCED ? q : 0] : (T)0);
        // the new boundary values, out to the neighbours
        if (edge_warp) {
            const unsigned slot = (n0lo + (unsigned)i + 1u) & tmask;
            const unsigned off = slot * slot_stride;
            const unsigned long long tag = entry_tag(n0) + (unsigned)(i + 1);
            // (CL: the global ring takes the launch's last levels)
            const bool glob = !CL || i + 1 > n_steps - (p.L + S_LEV);
            if constexpr (CL) {
                auto send = [&](unsigned to, const T *o) {
                    to += slot * (2u * NH * 16u);
                    if constexpr (sizeof(T) == 8) {
#pragma unroll
                        for (int q = 0; q < R; ++q)
                            st_half(to + 16u * q, (unsigned long long)__double_as_longlong((double)o[q]), 64u + i + 1u);
                    } else {
                        st_half(to, ((unsigned long long)__float_as_uint((float)(R > 1 ? o[R - 1] : (T)0)) << 32) |
                                        __float_as_uint((float)o[0]), 64u + i + 1u);
                    }
                };
                T o[R];
                if constexpr (PPT >= R) {
#pragma unroll
                    for (int q = 0; q < R; ++q) o[q] = v[q];
                    if (tid == 0) send(out0, o);
#pragma unroll
                    for (int q = 0; q < R; ++q) o[q] = v[PPT - R + q];
                    if (tid == NTH - 1) send(out1, o);
                } else {
                    o[0] = v[0];
                    o[R - 1] = __shfl_down_sync(kAll, v[0], 1);
                    if (tid == 0) send(out0, o);
                    if (tid == NTH - 2) send(out1, o);
                }
            }
            T o[R];
            if constexpr (PPT >= R) {
#pragma unroll
                for (int q = 0; q < R; ++q) o[q] = v[q];
                st_entry<T, ORDER, 0>(glob && tid == 0, ring_out + off, o, o, tag);
#pragma unroll
                for (int q = 0; q < R; ++q) o[q] = v[PPT - R + q];
                st_entry<T, ORDER, 0>(glob && tid == NTH - 1, ring_out + kEnt + off, o, o, tag);
            } else {
                o[0] = v[0];
                o[R - 1] = __shfl_down_sync(kAll, v[0], 1);
                st_entry<T, ORDER, 0>(glob && tid == 0, ring_out + off, o, o, tag);
                st_entry<T, ORDER, 0>(glob && tid == NTH - 2, ring_out + kEnt + off, o, o, tag);
            }
            if ((i & 15) == 15) kb = kb_next;
            const int k_next = __shfl_sync(kAll, kb, 2 * ((i + 1) & 15) + f);
            if (i + 1 < n_steps) read_ahead(i + 1, k_next);
        }
        if (n_warps > 1) put_edges(par ^ 1);
        if (p.levels && live) {
            // every level to its slot of the caller's array
            T *lg = reinterpret_cast<T *>(p.levels) + (size_t)((n0 + i + 1) % p.levels_depth) * (size_t)p.N +
                    (size_t)pj * M + tid * PPT;
            if constexpr (PPT >= 4) {
#pragma unroll
                for (int q = 0; q < PPT; q += 4) stg4<T>(lg + q, v + q);
            } else {
#pragma unroll
                for (int q = 0; q < PPT; ++q) lg[q] = v[q];
            }
        }
    }
    if (live && ok) {
#pragma unroll
        for (int i = 0; i < PPT; ++i) ug[i] = v[i];
    }
    if (hc <= p.L && cnt_k) atomicAdd(p.hist + hc, (unsigned long long)cnt_k);
    if (cnt16) atomicAdd(p.hist + 16, (unsigned long long)cnt16);
    // (no CTA leaves while a neighbour may still store into its shared memory)
    if constexpr (CL) cluster_sync();
    // the last CTA to finish advances the level of the state
    __syncthreads();
    if (tid == 0) {
        __threadfence();
        if (atomicAdd(p.ctrl + kCtrlDone, 1) == p.G - 1) {
            *reinterpret_cast<volatile long long *>(p.ctrl + kCtrlN0) = n0 + p.n_steps;
            *reinterpret_cast<volatile int *>(p.ctrl + kCtrlDone) = 0;
            __threadfence();
        }
    }
}

}  // namespace atk
