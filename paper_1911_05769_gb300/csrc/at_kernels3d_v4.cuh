// at_kernels3d_v4.cuh -- the 3D stepper of at_kernels3d.cuh (scalar equation or
// system, one level per pass, every delay mode) for FP32 subdomains whose rows
// are a power of two of 4-point groups: the shapes nearly every run has.
//
// The scheme is that of at_stepper3d; what differs is what a plane costs.  That
// kernel is bound by instruction issue, and most of its instructions are
// addresses: 606 lane instructions per point of the 5-field system on 16^3
// subdomains, 97 of them arithmetic.  Here
//   * a thread owns TC groups of 4 consecutive x columns in every field, for
//     any plane size: 16-byte shared loads, x neighbours by shuffles; a 16 x 16
//     plane takes a CTA of 64 threads, so that four to eight CTAs share an SM
//     and one's tile start overlaps the others' planes;
//   * shared memory is addressed by 32-bit byte offsets kept per thread, a
//     field's plane by one stride;
//   * the new x and y face values of a tile go into the halo words the same
//     thread has just read, and from there to the ring in 16-byte rows by the
//     whole team after the tile (no scattered stores in the plane loop); the z
//     faces are rows already and go straight between ring and registers;
//   * six lanes settle the six faces' delays at once, and all threads stage the
//     halos, every field of two faces in flight together, while the last warp
//     releases the previous tile's flags;
//   * the planes of a column alternate between two register slots known at
//     compile time, and only the first and last plane test for the z faces.
// The arithmetic is at_stepper3d's, operation by operation.
//
// A processing element is a team of NT threads; scalar CTAs hold 256 / NT teams
// (planes of 1024 points: one of 128; long columns fewer, as their halos fit),
// each with its own subdomains, shared memory and named barrier, the system's CTAs one (their shared memory is what
// limits them, and it comes in smaller pieces so).
//
// Pass times before and after (at_stepper3d, this kernel): 5-field system on
// 256^3 points in 16^3 subdomains, 16 levels, 7.98 and 4.6 ms (62.5 bytes a
// point and level: 2.47 ms at the measured copy bandwidth); scalar equation on 384
// x 256 x 288 points in 32^3 subdomains, 40 seeded levels, 3.74 and 2.79 ms
// (10.25 bytes: 1.71 ms).  What is left is the tile start: the halos' loads wait
// for the flags, and the CTAs of an SM only partly cover for each other.
#pragma once

#include "at_kernels3d.cuh"

namespace atk {

// resident CTAs per SM compiled for: the scalar equation 512 threads' worth;
// the system, whose threads hold every field's window, 256
constexpr int v4_min_ctas(int nf, int nt) { return nf == 1 ? 512 / nt : nt <= 64 ? 256 / nt : nt == 128 ? 2 : 1; }

// Free running, a face whose neighbour lags (by at most L) gets this long to bring
// level n itself before the delay is taken (at.h says so; at_stepper3d and the
// blocked kernel take what is there at once).  A team ahead of its neighbours stays
// nearer to them by it.  Mean delay, relative error against delay 0 and time a level,
// without the wait, with 10 and with 20 us (in brackets the kernel before this one,
// which had none):
//   5 fields of 256^3 in 16^3, 16 levels  0.091 2.8e-6 263 us  0.019 1.3e-6 248  0.011 8.5e-7 250  (0.030 1.2e-6 458)
//   256^3 in 16^3, 24 levels              0.104 4.5e-6  55     0.041 2.6e-6  59  0.003 5.1e-7  58  (0.102 2.9e-6 211)
//   512^3 in 32^3, 24 levels              0.053 3.0e-7 262     0.025 2.8e-7 266  0.013 2.2e-7 266  (0.097 3.9e-7 333)
// (barrier per level: 268, 58 and 249 us).  So it pays in time for several fields and
// costs the scalar equation 2 to 6 %, for delays a tenth to a quarter as large.
constexpr long long kGraceNs = 20000;

// grid barrier before level `step` (1-based within the launch), one arrival per
// team that has subdomains (npe of them); bounded.  Returns false on abort.
// (The flag may be tested behind the last barrier here: a synchronous run sets it
// again only behind the tile's next one.)
template <typename Sync>
__device__ bool team_grid_sync(const Params3 &p, long long step, long long npe, int ttid, volatile int *s_flag, Sync sync)
{
    sync();
    if (ttid == 0) {
        __threadfence();
        atomicAdd(p.gbar, 1ull);
        const unsigned long long target = (unsigned long long)step * (unsigned long long)npe;
        const unsigned long long t0 = global_ns();
        while (ld_acquire(p.gbar) < target) {
            if (ld_relaxed(p.ctrl + kCtrlAbort)) { *s_flag = -1; break; }
            if ((long long)(global_ns() - t0) > p.timeout_ns) { raise_timeout3(p, kWhereGrid, step, -1); *s_flag = -1; break; }
        }
        __threadfence();
    }
    sync();
    return *s_flag != -1;
}

// Shared memory of a team: stage barriers and counters, delay counters, the
// faces' delays and the abort word, the halos of the x and y faces (z halos go
// straight to registers), plane stages.
struct Smem3v4 {
    long long hist_off, face_off, halo_at[4], top_off, stage_off, plane_bytes, total;
};

__host__ __device__ inline Smem3v4 smem3v4_layout(int m0, int m1, int m2, int stages, int nf)
{
    Smem3v4 l;
    l.hist_off = 24LL * stages;                      // full[stages], empty[stages], two ints per stage
    l.face_off = round_up(l.hist_off + 4LL * (kMaxL + 1), 16);
    long long at = round_up(l.face_off + 32, 128);
    for (int f = 0; f < 4; ++f) {
        l.halo_at[f] = at;
        at = round_up(at + 4LL * nf * (f < 2 ? m1 : m0) * m2, 16);
    }
    l.top_off = round_up(at, 128);                   // several fields: the halo above the tile
    l.plane_bytes = round_up(4LL * nf * m0 * m1, 128);   // a plane of every field
    l.stage_off = l.top_off + (nf > 1 ? l.plane_bytes : 0);
    l.total = round_up(l.stage_off + stages * l.plane_bytes, 128);
    return l;
}

template <int NF, bool SYS, int NT, int TC, bool ISO, int TEAMS, int CTAS = v4_min_ctas(NF, NT * TEAMS)>
__global__ void __launch_bounds__(NT * TEAMS, CTAS)
    at_stepper3d_v4(const Params3 p, const __grid_constant__ CUtensorMap tmap)
{
    using T = float;
    constexpr int VW = 4;
    constexpr int kWarps3 = NT / 32;
    extern __shared__ __align__(128) unsigned char smem_cta[];
    const Smem3v4 sl = smem3v4_layout(p.m0, p.m1, p.m2, p.stages, NF);
    const int team = TEAMS == 1 ? 0 : (int)threadIdx.x / NT;
    unsigned char *smem = smem_cta + team * (int)sl.total;
    // barrier of this team's threads
    auto sync = [&]() {
        if constexpr (TEAMS == 1) __syncthreads();
        else asm volatile("bar.sync %0, %1;" ::"r"(team + 1), "n"(NT) : "memory");
    };
    // the same, and whether `x` holds for any of them: the whole team leaves or
    // stays together (a word tested after a plain barrier may have been set
    // since by a thread that is already past it)
    auto any = [&](bool x) -> bool {
        if constexpr (TEAMS == 1) {
            return __syncthreads_or(x) != 0;
        } else {
            int r;
            asm volatile("{\n\t.reg .pred a, b;\n\tsetp.ne.s32 a, %1, 0;\n\t"
                         "barrier.cta.red.or.pred b, %2, %3, a;\n\tselp.s32 %0, 1, 0, b;\n\t}"
                         : "=r"(r) : "r"((int)x), "r"(team + 1), "n"(NT) : "memory");
            return r != 0;
        }
    };
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem);
    unsigned *hist = reinterpret_cast<unsigned *>(smem + sl.hist_off);
    volatile int *s_k = reinterpret_cast<volatile int *>(smem + sl.face_off);   // the faces' delays
    int *s_flag = reinterpret_cast<int *>(smem + sl.face_off + 24);             // barrier / abort word
    const int m0 = p.m0, m1 = p.m1, m2 = p.m2, NS = p.stages;
    const int PW = m0 * m1;
    // byte offsets of the halo planes, byte strides of a field in them and in a stage
    const int o_x0 = (int)sl.halo_at[0], o_x1 = (int)sl.halo_at[1], o_y0 = (int)sl.halo_at[2],
              o_y1 = (int)sl.halo_at[3];
    const int bx = 4 * m1 * m2, by = 4 * m0 * m2, bp = 4 * PW;
    const int o_top = (int)sl.top_off, o_stage = (int)sl.stage_off, pbytes = (int)sl.plane_bytes;
    const unsigned tx_bytes = (unsigned)(NF * bp);                           // one box: a plane of every field

    const int tid = (int)threadIdx.x - team * NT, lane = tid & 31, warp = tid >> 5;   // within the team
    const long long npes = (long long)p.G * TEAMS;
    const ItemRange own = cta_items(p.P, p.G, TEAMS, blockIdx.x, team);
    const long long lo = own.lo, hi = own.hi;
    const long long S = hi - lo;
    const long long lev0 = *reinterpret_cast<const volatile long long *>(p.ctrl + kCtrlN0);
    const long long Q = p.n_steps * S * m2;                                  // planes this team sweeps
    const T cA0 = p.cA32[0], cA1 = p.cA32[1], cA2 = p.cA32[2];
    const long long field_words = p.n0 * p.n1 * p.n2, plane_words = p.n0 * p.n1;
    const size_t fstride = (size_t)p.face_words;                             // a field of a ring entry
    const unsigned uP0 = (unsigned)p.P0, uP01 = (unsigned)(p.P0 * p.P1);

    constexpr bool LAST_WARP = NF == 1;
    int *s_fills = reinterpret_cast<int *>(bars + 2 * NS), *s_done = s_fills + NS;   // planes issued, warps done
    if (tid < NS) {
        mbar_init(&bars[tid], 1);
        if (!LAST_WARP) mbar_init(&bars[NS + tid], kWarps3);
        s_fills[tid] = 0;
        s_done[tid] = 0;
    }
    if (tid == 0) { mbar_fence_init(); *s_flag = 0; }
    for (int i = tid; i <= kMaxL; i += NT) hist[i] = 0u;
    sync();

    auto tile_coords = [&](long long sub, int *x, int *y, int *z) {
        const unsigned us = (unsigned)sub, q2 = us / uP01, r = us - q2 * uP01, q1 = r / uP0, q0 = r - q1 * uP0;
        *x = (int)(q0 * m0); *y = (int)(q1 * m1); *z = (int)(q2 * m2);
    };
    auto issue_plane = [&](int st, int x0, int y0, int z0) {
        mbar_arrive_expect_tx(&bars[st], tx_bytes);
        tensor_load_4d(smem + o_stage + st * pbytes, &tmap, x0, y0, z0, 0, &bars[st]);
        s_fills[st] += 1;
    };
    int tx0, ty0, tz0, nx0, ny0, nz0;    // the current tile's first point, the next tile's
    tile_coords(lo, &tx0, &ty0, &tz0);
    tile_coords(lo + 1 >= hi ? lo : lo + 1, &nx0, &ny0, &nz0);

    // this thread's groups (a row of GR <= 32 groups lies in one warp).  Threads
    // beyond the plane take group 0's addresses and store nothing.
    const int GR = m0 / VW;
    int cb[TC], cxb[TC], cyb[TC], goff[TC];      // bytes in a plane, of x, of y; words in a plane of u
    bool cv[TC], fx0[TC], fx1[TC], fy0[TC], fy1[TC], wx0[TC], wx1[TC], wy0[TC], wy1[TC];
#pragma unroll
    for (int q = 0; q < TC; ++q) {
        const int g = tid + NT * q;
        cv[q] = g < PW / VW;
        const int x = cv[q] ? (g % GR) * VW : 0, y = cv[q] ? g / GR : 0;
        cb[q] = 4 * (y * m0 + x);
        cxb[q] = 4 * x;
        cyb[q] = 4 * y;
        goff[q] = y * (int)p.n0 + x;
        fx0[q] = x == 0; fx1[q] = x + VW == m0; fy0[q] = y == 0; fy1[q] = y == m1 - 1;
        // (face words are read by any thread, written by the group's owner)
        wx0[q] = fx0[q] && cv[q]; wx1[q] = fx1[q] && cv[q]; wy0[q] = fy0[q] && cv[q]; wy1[q] = fy1[q] && cv[q];
    }
    // a group that is first and last of its row takes both x halos
    const bool both_x = GR == 1;
    // planes z - 1 and z of this thread's columns while plane z is computed:
    // plane z in slot z & 1 (UNROLL; else 0), plane z - 1 in the other; the
    // halo above the tile
    // (UNROLL: in registers; else in shared memory)
    constexpr bool UNROLL = NF == 1;
    T W[2][NF][TC][VW], above_top[UNROLL ? NF : 1][TC][VW];

    if (tid == 0)
        for (int st = 0; st < NS && st < Q; ++st) issue_plane(st, tx0, ty0, tz0 + st);
    int gs = 0;                              // stage and fill parity of the current plane
    unsigned gp = 0;
    // every lane tests the stage's barrier; a wait that runs out is recorded in
    // s_flag, on which the team acts as one at the next barrier of a tile start
    auto wait_plane = [&](int st, unsigned par) -> bool {
        bool good = mbar_try_wait(&bars[st], par);
        if (!good) {
            good = wait_stage3(p, &bars[st], par);
            if (!good) atomicExch(s_flag, -1);
        }
        return __all_sync(0xffffffffu, good);
    };
    auto sm = [&](int off) -> T * { return reinterpret_cast<T *>(smem + off); };

    bool ok = true;
    long long lv = lev0, sub = lo;
    long long prev_sub = -1, prev_new = 0;   // the tile whose faces are still to be published
    const long long n_tiles = p.n_steps * S;
    // the x and y faces of tile (sub, new level) from the halo words to the ring
    auto faces_out = [&](long long s, long long l) {
        T *rb = ring_entry<T>(p, l, s, 0);
#pragma unroll
        for (int f = 0; f < 4; ++f) {
            const int nw = f < 2 ? m1 * m2 : m0 * m2;
            const T *h = sm(f == 0 ? o_x0 : f == 1 ? o_x1 : f == 2 ? o_y0 : o_y1);
            T *r = rb + (size_t)f * fstride * NF;
            if ((nw & 3) == 0) {
#pragma unroll 2
                for (int i = 4 * tid; i < nw; i += 4 * NT) {
                    T v[NF][4];
#pragma unroll
                    for (int fld = 0; fld < NF; ++fld) lds<T, 4>(h + fld * nw + i, v[fld]);
#pragma unroll
                    for (int fld = 0; fld < NF; ++fld) stv<T, 4>(r + fld * fstride + i, v[fld]);
                }
            } else {
                for (int i = tid; i < nw; i += NT)
                    for (int fld = 0; fld < NF; ++fld) r[fld * fstride + i] = h[fld * nw + i];
            }
        }
    };
    // flags of the published faces (lanes 0..5 of the last warp)
    auto release = [&](long long s, long long l) {
        if (warp == kWarps3 - 1 && lane < 6 && !(p.skip_publish && blockIdx.x == 0 && l > p.skip_step)) {
            __threadfence();
            st_relaxed(p.flag + s * 6 + lane, (unsigned long long)l);
        }
    };
    for (long long t = 0; t < n_tiles; ++t) {
        // ---- tile start: the previous tile's faces to the ring, grid barrier
        // (synchronous mode), delays, halos
        if (any(*reinterpret_cast<volatile int *>(s_flag) == -1)) { ok = false; break; }
        // (released before this tile waits for other teams' flags)
        if (prev_sub >= 0) {
            faces_out(prev_sub, prev_new);
            sync();
            release(prev_sub, prev_new);
        }
        if (p.mode == kModeSync && sub == lo && lv > lev0) {
            if (!team_grid_sync(p, lv - lev0, p.P < npes ? p.P : npes, tid, s_flag, sync)) { ok = false; break; }
        }
        const unsigned us = (unsigned)sub, us2 = us / uP01, usr = us - us2 * uP01, us1 = usr / uP0;
        const long long s0 = usr - us1 * uP0, s1 = us1, s2 = us2;
        if (tid < 6) {
            const int f = tid;
            const long long q = face_neighbour(p, s0, s1, s2, f);
            long long k = 0;
            bool good = true;
            long long kmax = lv - 2 + 1;           // s = 2 levels per extrapolation
            if (kmax < 0) kmax = 0;
            if (kmax > p.L) kmax = p.L;
            if (p.mode == kModeSeeded) {
                const unsigned long long ctr = ((unsigned long long)lv * (unsigned long long)p.P +
                                                (unsigned long long)sub) * 6ull + (unsigned long long)f;
                k = (long long)(((splitmix64(p.seed, ctr) >> 32) * (unsigned long long)(p.L + 1)) >> 32);
            } else if (p.mode == kModeReplay) {
                k = p.delays[((size_t)(lv - lev0) * p.P + sub) * 6 + f];
            }
            if (k > kmax) k = kmax;
            if (k < 0) k = 0;
            if (p.mode != kModeSync) {
                const unsigned long long *fl = p.flag + q * 6 + (f ^ 1);
                const long long need = (p.mode == kModeFree) ? lv - kmax : lv - k;
                unsigned long long seen = ld_acquire(fl);
                if ((long long)seen < need && !wait_flag3(p, fl, need, &seen, lv, q)) good = false;
                if (p.mode == kModeFree && (long long)seen < lv && good) {
                    const unsigned long long t0 = global_ns();
                    do seen = ld_acquire(fl);
                    while ((long long)seen < lv && (long long)(global_ns() - t0) < kGraceNs);
                }
                if (good && p.mode == kModeFree) k = lv - ((long long)seen < lv ? (long long)seen : lv);
            }
            if (good) {
                atomicAdd(&hist[k], 1u);
                if (p.delays && p.mode != kModeReplay)
                    p.delays[((size_t)(lv - lev0) * p.P + sub) * 6 + f] = (int8_t)k;
            } else {
                atomicExch(s_flag, -1);
            }
            s_k[f] = (int)k;
            __threadfence();
        }
        if (any(*reinterpret_cast<volatile int *>(s_flag) == -1)) { ok = false; break; }
        // halos, (k+1) f0 - k f1 in Newton form f0 + k (f0 - f1): the z faces of
        // this thread's columns into registers, the x and y faces into shared
        // memory; the loads of two faces in flight together
        {
            auto entry = [&](int f, int kk, int back) -> const T * {
                return ring_entry<T>(p, lv - kk - back, face_neighbour(p, s0, s1, s2, f), f ^ 1);
            };
            const int k4 = s_k[4], k5 = s_k[5];
            T n4[NF][TC][VW], n5[NF][TC][VW], h5[NF][TC][VW];
            const T *e4 = entry(4, k4, 0), *d4 = entry(4, k4, 1), *e5 = entry(5, k5, 0), *d5 = entry(5, k5, 1);
#pragma unroll
            for (int f = 0; f < NF; ++f)
#pragma unroll
                for (int q = 0; q < TC; ++q) {
                    lds<T, VW>(e4 + f * fstride + cb[q] / 4, W[1][f][q]);        // (16-byte global loads)
                    lds<T, VW>(e5 + f * fstride + cb[q] / 4, h5[f][q]);
                    if (k4 != 0) lds<T, VW>(d4 + f * fstride + cb[q] / 4, n4[f][q]);
                    if (k5 != 0) lds<T, VW>(d5 + f * fstride + cb[q] / 4, n5[f][q]);
                }
            auto finish_z = [&]() {
#pragma unroll
                for (int f = 0; f < NF; ++f)
#pragma unroll
                    for (int q = 0; q < TC; ++q) {
#pragma unroll
                        for (int e = 0; e < VW; ++e) {
                            const T a = W[1][f][q][e], b = h5[f][q][e];
                            if (k4 != 0) W[1][f][q][e] = a + (T)k4 * (a - n4[f][q][e]);
                            h5[f][q][e] = k5 != 0 ? b + (T)k5 * (b - n5[f][q][e]) : b;
                            if constexpr (UNROLL) above_top[f][q][e] = h5[f][q][e];
                        }
                        if (!UNROLL && cv[q]) sts4<T>(sm(o_top + f * bp + cb[q]), h5[f][q]);
                    }
            };
            if constexpr (!UNROLL) finish_z();
            constexpr int FB = NF <= 3 ? 2 : 1;     // faces in flight together
#pragma unroll 1
            for (int fa = 0; fa < 4; fa += FB) {
                const int nw = fa < 2 ? m1 * m2 : m0 * m2;
                const T *ea[FB], *da[FB];
                int ka[FB];
                T *ha[FB];
#pragma unroll
                for (int h = 0; h < FB; ++h) {
                    const int f = fa + h;
                    ka[h] = s_k[f];
                    ea[h] = entry(f, ka[h], 0);
                    da[h] = entry(f, ka[h], 1);
                    ha[h] = sm(f == 0 ? o_x0 : f == 1 ? o_x1 : f == 2 ? o_y0 : o_y1);
                }
                if ((nw & 3) == 0) {
#pragma unroll(NF == 1 ? 2 : 1)
                    for (int i = 4 * tid; i < nw; i += 4 * NT) {
                        T va[FB][NF][4], wa[FB][NF][4];
#pragma unroll
                        for (int h = 0; h < FB; ++h)
#pragma unroll
                            for (int f = 0; f < NF; ++f) {
                                lds<T, 4>(ea[h] + f * fstride + i, va[h][f]);
                                if (ka[h] != 0) lds<T, 4>(da[h] + f * fstride + i, wa[h][f]);
                            }
#pragma unroll
                        for (int h = 0; h < FB; ++h)
#pragma unroll
                            for (int f = 0; f < NF; ++f) {
                                if (ka[h] != 0) {
#pragma unroll
                                    for (int e = 0; e < 4; ++e)
                                        va[h][f][e] = va[h][f][e] + (T)ka[h] * (va[h][f][e] - wa[h][f][e]);
                                }
                                sts4<T>(ha[h] + f * nw + i, va[h][f]);
                            }
                    }
                } else {
                    for (int i = tid; i < nw; i += NT)
                        for (int h = 0; h < FB; ++h)
                            for (int f = 0; f < NF; ++f) {
                                const T a = ea[h][f * fstride + i];
                                ha[h][f * nw + i] = ka[h] == 0 ? a : a + (T)ka[h] * (a - da[h][f * fstride + i]);
                            }
                }
            }
            if constexpr (UNROLL) finish_z();
        }
        sync();
        // plane 0
        if (!wait_plane(gs, gp)) ok = false;
#pragma unroll
        for (int f = 0; f < NF; ++f)
#pragma unroll
            for (int q = 0; q < TC; ++q) lds<T, VW>(sm(o_stage + gs * pbytes + f * bp + cb[q]), W[0][f][q]);
        T *up = reinterpret_cast<T *>(p.u) + ((long long)tz0 * plane_words + (long long)ty0 * p.n0 + tx0);
        T *const rz = ring_entry<T>(p, lv + 1, sub, 4);       // the z faces' ring entries (4, then 5)
        // ---- the planes of the tile; warps run independently (stage barriers
        // only).  Each warp counts itself done with a stage, which is refilled
        // by the last warp (LAST_WARP), or by thread 0 a plane later: 2.83
        // against 3.04 ms for the scalar equation's four warps (40 levels of 384
        // x 256 x 288 points, seeded), the other way round for the system's two.
        const bool more = t + 1 < n_tiles;
        auto refill = [&](int st, unsigned par, int z) -> bool {     // the stage that held plane z
            if (z + NS >= m2 && !more) return true;
            if (!mbar_try_wait(&bars[NS + st], par) && !wait_stage3(p, &bars[NS + st], par)) {
                atomicExch(s_flag, -1);
                return false;
            }
            if (z + NS < m2) issue_plane(st, tx0, ty0, tz0 + z + NS);
            else issue_plane(st, nx0, ny0, nz0 + z + NS - m2);
            return true;
        };
        int ps = 0;                              // the last plane's stage and parity
        unsigned pp = 0;
        // shared-memory addresses that move by a plane: the y halos' row and
        // the x halos' column of this thread's groups
        int hy[TC], hx[TC];
#pragma unroll
        for (int q = 0; q < TC; ++q) {
            hy[q] = (fy0[q] ? o_y0 : o_y1) + cxb[q];
            hx[q] = (fx0[q] ? o_x0 : o_x1) + cyb[q];
        }
        T *ug[TC];
#pragma unroll
        for (int q = 0; q < TC; ++q) ug[q] = up + goff[q];
        // one plane.  PAR: z & 1 (slots of the window); EDGE: it may be the
        // tile's first or last one
        auto plane = [&](auto PAR, auto EDGE, int z) -> bool {
            constexpr int C = UNROLL ? decltype(PAR)::value : 0, B = C ^ 1;
            constexpr bool edge = decltype(EDGE)::value != 0;
            const bool top = edge && z == m2 - 1;
            const int sg = gs, sg1 = gs + 1 == NS ? 0 : gs + 1;
            const unsigned gp1 = sg1 == 0 ? gp ^ 1u : gp;
            if (!top && !wait_plane(sg1, gp1)) return false;
            if (!LAST_WARP && warp == 0 && z > 0) {
                const int r = lane == 0 ? (refill(ps, pp, z - 1) ? 1 : 0) : 0;
                if (!__shfl_sync(0xffffffffu, r, 0)) return false;
            }
            const int st = o_stage + sg * pbytes, sn = o_stage + sg1 * pbytes;
            int ao[TC], ym_a[TC], yp_a[TC], xa[TC];
            T Uv[TC][VW], Vv[TC][VW], Wv[TC][VW];        // advecting velocity, level n (the system)
#pragma unroll
            for (int q = 0; q < TC; ++q) {
                ao[q] = (!UNROLL && top ? o_top : sn) + cb[q];
                ym_a[q] = fy0[q] ? hy[q] : st + cb[q] - 4 * m0;
                yp_a[q] = fy1[q] ? hy[q] : st + cb[q] + 4 * m0;
                xa[q] = hx[q];
#pragma unroll
                for (int e = 0; e < VW; ++e) {
                    Uv[q][e] = SYS ? W[C][0][q][e] : (T)0;
                    Vv[q][e] = SYS ? W[C][1 % NF][q][e] : (T)0;
                    Wv[q][e] = SYS ? W[C][2 % NF][q][e] : (T)0;
                }
            }
#pragma unroll
            for (int f = 0; f < NF; ++f) {
                const T b0 = p.cBf32[SYS ? f : 0][0];
                [[maybe_unused]] const T b1 = p.cBf32[SYS ? f : 0][1], b2 = p.cBf32[SYS ? f : 0][2];
                T ab[TC][VW], ym[TC][VW], yp[TC][VW], xl[TC], xr[TC];
#pragma unroll
                for (int q = 0; q < TC; ++q) {
                    if (UNROLL && top) {
#pragma unroll
                        for (int e = 0; e < VW; ++e) ab[q][e] = above_top[UNROLL ? f : 0][q][e];
                    } else {
                        lds<T, VW>(sm(ao[q]), ab[q]);
                    }
                    lds<T, VW>(sm(ym_a[q]), ym[q]);
                    lds<T, VW>(sm(yp_a[q]), yp[q]);
                    xl[q] = __shfl_up_sync(0xffffffffu, W[C][f][q][VW - 1], 1);
                    xr[q] = __shfl_down_sync(0xffffffffu, W[C][f][q][0], 1);
                    if (fx0[q]) xl[q] = *sm(xa[q]);
                    if (fx1[q]) xr[q] = *sm(xa[q] + (both_x ? o_x1 - o_x0 : 0));
                }
#pragma unroll
                for (int q = 0; q < TC; ++q) {
                    T un[VW];
#pragma unroll
                    for (int e = 0; e < VW; ++e) {
                        const T cc = W[C][f][q][e], below = W[B][f][q][e], above = ab[q][e];
                        const T xm = e == 0 ? xl[q] : W[C][f][q][e > 0 ? e - 1 : 0];
                        const T xp = e == VW - 1 ? xr[q] : W[C][f][q][e + 1 < VW ? e + 1 : e];
                        if constexpr (ISO) {
                            const T sum = ((xp + xm) + (yp[q][e] + ym[q][e])) + (above + below);
                            const T dif = ((xp - xm) + (yp[q][e] - ym[q][e])) + (above - below);
                            un[e] = cc + (b0 * (sum - (T)6 * cc) - cc * (cA0 * dif));
                        } else {
                            const T d2 = b0 * ((xp + xm) - (T)2 * cc) + b1 * ((yp[q][e] + ym[q][e]) - (T)2 * cc) +
                                         b2 * ((above + below) - (T)2 * cc);
                            if constexpr (SYS) {
                                const T adv = cA0 * Uv[q][e] * (xp - xm) + cA1 * Vv[q][e] * (yp[q][e] - ym[q][e]) +
                                              cA2 * Wv[q][e] * (above - below);
                                un[e] = cc + (d2 - adv);
                            } else {
                                const T d1 = cA0 * (xp - xm) + cA1 * (yp[q][e] - ym[q][e]) + cA2 * (above - below);
                                un[e] = cc + (d2 - cc * d1);
                            }
                        }
                    }
                    if (cv[q]) stv<T, VW>(ug[q] + f * field_words, un);
                    // the new x and y face values into the halo words just read,
                    // the z faces to the ring
                    if (wx0[q]) *sm(xa[q]) = un[0];
                    if (wx1[q]) *sm(xa[q] + (both_x ? o_x1 - o_x0 : 0)) = un[VW - 1];
                    if (wy0[q]) sts4<T>(sm(ym_a[q]), un);
                    if (wy1[q]) sts4<T>(sm(yp_a[q]), un);
                    if constexpr (edge) {
                        if (cv[q] && (z == 0 || top))
                            stv<T, VW>(rz + (top ? fstride * NF : (size_t)0) + f * fstride + cb[q] / 4, un);
                    }
#pragma unroll
                    for (int e = 0; e < VW; ++e) {
                        if constexpr (UNROLL) {
                            W[B][f][q][e] = ab[q][e];
                        } else {
                            W[1][f][q][e] = W[0][f][q][e];
                            W[0][f][q][e] = ab[q][e];
                        }
                    }
                    if (NF > 1) {
                        ao[q] += bp;
                        ym_a[q] += fy0[q] ? by : bp;
                        yp_a[q] += fy1[q] ? by : bp;
                        xa[q] += bx;
                    }
                }
            }
#pragma unroll
            for (int q = 0; q < TC; ++q) {
                ug[q] += plane_words;
                hy[q] += 4 * m0;
                hx[q] += 4 * m1;
            }
            // the next read of a plane written here is a bulk copy (async
            // proxy) at the next level: with two or more subdomains per team it
            // is issued after this tile ends, so one proxy fence per tile
            // covers every plane; with one subdomain, fence every plane
            if (top || S == 1) fence_proxy_async_global();
            __syncwarp();
            // done with stage sg (plane z - 1 read it as the plane above)
            if (lane == 0) {
                if constexpr (LAST_WARP) {
                    __threadfence_block();
                    if (kWarps3 == 1 || atomicAdd(&s_done[sg], 1) == kWarps3 - 1) {
                        s_done[sg] = 0;
                        __threadfence_block();
                        if (z + NS < m2) issue_plane(sg, tx0, ty0, tz0 + z + NS);
                        else if (more) issue_plane(sg, nx0, ny0, nz0 + z + NS - m2);
                    }
                } else {
                    mbar_arrive(&bars[NS + sg]);
                }
            }
            ps = sg;
            pp = gp;
            gs = sg1;
            gp = gp1;
            return true;
        };
        if constexpr (UNROLL) {
            ok = ok && plane(IntC<0>{}, IntC<1>{}, 0);
            int z = 1;
            for (; z + 1 < m2 - 1 && ok; z += 2) {
                ok = plane(IntC<1>{}, IntC<0>{}, z);
                ok = ok && plane(IntC<0>{}, IntC<0>{}, z + 1);
            }
            if (z < m2 - 1 && ok) {
                ok = plane(IntC<1>{}, IntC<0>{}, z);
                ok = ok && plane(IntC<0>{}, IntC<1>{}, z + 1);
            } else if (ok) {
                ok = plane(IntC<1>{}, IntC<1>{}, z);
            }
        } else {
            // (several fields: one copy of the plane's code, or it does not fit
            // the instruction cache)
            for (int z = 0; z < m2 && ok; ++z) ok = plane(IntC<0>{}, IntC<1>{}, z);
        }
        if (!LAST_WARP && tid == 0 && ok && !refill(ps, pp, m2 - 1)) ok = false;
        prev_sub = sub;
        prev_new = lv + 1;
        if (++sub == hi) { sub = lo; ++lv; }
        tx0 = nx0; ty0 = ny0; tz0 = nz0;
        tile_coords(sub + 1 == hi ? lo : sub + 1, &nx0, &ny0, &nz0);
    }
    if (any(*reinterpret_cast<volatile int *>(s_flag) == -1)) ok = false;
    if (ok && prev_sub >= 0) {
        faces_out(prev_sub, prev_new);
        sync();
        release(prev_sub, prev_new);
    }
    // let the copies in flight land before leaving (the latest fill of each
    // stage completes the phase of parity (fills of the stage - 1) & 1)
    if (tid == 0) {
        for (int st = 0; st < NS; ++st) {
            if (s_fills[st] == 0) continue;
            const unsigned par = (unsigned)((s_fills[st] - 1) & 1);
            const unsigned long long t0 = global_ns();
            while (!mbar_try_wait(&bars[st], par) && (long long)(global_ns() - t0) < p.timeout_ns) {
            }
        }
    }
    sync();
    for (int i = tid; i <= p.L && i <= kMaxL; i += NT)
        if (hist[i]) atomicAdd(p.hist + i, (unsigned long long)hist[i]);
    // the last CTA to finish advances the level and rearms the grid barrier
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        if (atomicAdd(p.ctrl + kCtrlDone, 1) == p.G - 1) {
            *reinterpret_cast<volatile long long *>(p.ctrl + kCtrlN0) = lev0 + p.n_steps;
            *reinterpret_cast<volatile int *>(p.ctrl + kCtrlDone) = 0;
            *reinterpret_cast<volatile unsigned long long *>(p.gbar) = 0ull;
            __threadfence();
        }
    }
}

}  // namespace atk
