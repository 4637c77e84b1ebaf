// K4, open boundaries: the FP64 force sums with the pair terms of all but the
// closest sources in two-part FP32 arithmetic (grav_df.cuh).  One target per
// thread; two stages of packed tiles, each released warp by warp (no block
// barrier between tiles); the running FP64 sums (hi, lo) of each target in
// shared memory.
//
// What bounds it: issue and the FP32 pipe's latency (about 320 lane operations a
// pair in dependent chains, 12 warps an SM by registers: issue slots 43% busy, 1.81
// instructions a clock); the FP64 unit, 23% busy, has the per-tile conversions and
// carries, about 160 FP64 instructions per warp and tile, and the listed pairs.
#pragma once

#include "grav_df.cuh"
#include "grav_eval.cuh"

namespace grav {

// slots of the two-part sums
enum { DA = 0, DJ1 = 3, DJ2 = 6, DT = 9, DP = 15, kDfSums = 16 };

template <int NT, int S, bool POT>
struct DfSmem {
    static constexpr int NC = POT ? kNCPot : kNC;
    static constexpr int kStages = 2;
    float stage[kStages][df_words<S>()];
    double sum[NC][2][NT];         // running sums (hi, lo) of each target
    uint64_t bar[kStages];
    int done[kStages];             // warps finished with the tile in each stage
    unsigned issued[kStages];      // copies issued into each stage
    int abort_flag;
    long long ticket;
};

// The sums of one pair of sources given its separations and inverse powers.
template <bool POT>
__device__ __forceinline__ void df_accumulate(DfSum (&sm)[kDfSums], const DfWindows &w, const DfInv &inv,
                                              const float2 d[3], const float2 e[3], const float2 vh[3],
                                              const float2 vl[3], float2 mh, float2 ml)
{
    float2 y3h, y3l, fh, fl, gh, gl;
    df_inv3(inv, y3h, y3l);
    df_mul(mh, ml, y3h, y3l, fh, fl);
    df_times_inv2(inv, fh, fl, gh, gl);
    const float2 CA = dup2(w.a), CT = dup2(w.t), CJ = dup2(w.j);
    const float2 CA2 = dup2(df_second(w.a)), CT2 = dup2(df_second(w.t)), CJ2 = dup2(df_second(w.j));
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        df_add_product(sm[DA + c], CA, CA2, fh, fl, d[c], e[c]);
        df_add_product(sm[DJ1 + c], CJ, CJ2, fh, fl, vh[c], vl[c]);
    }
    float2 dvh, dvl;
    df_dot3(d, e, vh, vl, dvh, dvl);
    float2 xh, xl;
    df_mul(gh, gl, d[0], e[0], xh, xl);
    df_add_product(sm[DT + 0], CT, CT2, xh, xl, d[0], e[0]);
    df_add_product(sm[DT + 3], CT, CT2, xh, xl, d[1], e[1]);
    df_add_product(sm[DT + 4], CT, CT2, xh, xl, d[2], e[2]);
    df_add_product(sm[DJ2 + 0], CJ, CJ2, xh, xl, dvh, dvl);
    df_mul(gh, gl, d[1], e[1], xh, xl);
    df_add_product(sm[DT + 1], CT, CT2, xh, xl, d[1], e[1]);
    df_add_product(sm[DT + 5], CT, CT2, xh, xl, d[2], e[2]);
    df_add_product(sm[DJ2 + 1], CJ, CJ2, xh, xl, dvh, dvl);
    df_mul(gh, gl, d[2], e[2], xh, xl);
    df_add_product(sm[DT + 2], CT, CT2, xh, xl, d[2], e[2]);
    df_add_product(sm[DJ2 + 2], CJ, CJ2, xh, xl, dvh, dvl);
    if (POT) {
        // r^-1 = y (1 + t/2 + 3/8 t^2)
        float2 yh = inv.y;
        float2 yl = __fmul2_rn(__ffma2_rn(inv.t, __ffma2_rn(dup2(0.375f), inv.t, dup2(0.5f)),
                                          __fmul2_rn(dup2(0.5f), inv.s)), yh);
        df_norm(yh, yl);
        df_add_product(sm[DP], dup2(w.p), dup2(df_second(w.p)), mh, ml, yh, yl);
    }
}

// One sub-block of 32 sources (16 records at P).  LIST: pairs closer than thr2
// (squared, units of L) are listed and left out of the sums (list(j), j < 32);
// otherwise no pair is that close.
template <bool POT, bool LIST, typename Add>
__device__ __forceinline__ void df_sub_loop(const float4 *__restrict__ P, const DfTarget &tg,
                                            const DfWindows &w, float thr2, DfSum (&sums)[kDfSums],
                                            Add &&list)
{
#pragma unroll 1
    for (int k0 = 0; k0 < kDfSub / 2; k0 += kDfCarry) {
#pragma unroll 1
        for (int k = k0; k < k0 + kDfCarry; ++k) {
            const float4 *r = P + 7 * k;
            const float4 q0 = r[0], q1 = r[1], q2 = r[2];
            float2 d[3], e[3];
            df_diff(make_float2(q0.x, q0.y), make_float2(q1.z, q1.w), -tg.h[0], -tg.l[0], -tg.l2[0], d[0],
                    e[0]);
            df_diff(make_float2(q0.z, q0.w), make_float2(q2.x, q2.y), -tg.h[1], -tg.l[1], -tg.l2[1], d[1],
                    e[1]);
            df_diff(make_float2(q1.x, q1.y), make_float2(q2.z, q2.w), -tg.h[2], -tg.l[2], -tg.l2[2], d[2],
                    e[2]);
            float2 r2h, r2l, sq;
            df_square3(d, e, r2h, r2l, sq);
            const float4 q3 = r[3], q4 = r[4], q5 = r[5], q6 = r[6];
            float2 mh = make_float2(q6.x, q6.y), ml = make_float2(q6.z, q6.w);
            if (LIST && !(fminf(r2h.x, r2h.y) >= thr2)) {
                // (listed, or padding: no mass at distance 1 instead)
                if (!(r2h.x >= thr2)) {
                    if (mh.x != 0.0f) list(2 * k);
                    mh.x = ml.x = r2l.x = sq.x = 0.0f;
                    r2h.x = 1.0f;
                }
                if (!(r2h.y >= thr2)) {
                    if (mh.y != 0.0f) list(2 * k + 1);
                    mh.y = ml.y = r2l.y = sq.y = 0.0f;
                    r2h.y = 1.0f;
                }
            }
            const DfInv inv = df_inverse(r2h, r2l, sq);
            const float2 vh[3] = {make_float2(q3.x, q3.y), make_float2(q3.z, q3.w), make_float2(q4.x, q4.y)};
            const float2 vl[3] = {make_float2(q4.z, q4.w), make_float2(q5.x, q5.y), make_float2(q5.z, q5.w)};
            df_accumulate<POT>(sums, w, inv, d, e, vh, vl, mh, ml);
        }
#pragma unroll
        for (int c = 0; c < kDfSums - (POT ? 0 : 1); ++c)
            df_carry(sums[c], dup2(df_second(c < DJ1 ? w.a : c < DT ? w.j : c < DP ? w.t : w.p)));
    }
}

// One pair in FP64, the cubic spline inside h.  LISTED: the Newtonian inverse
// powers are corrected for the rounding of rsqrt (t = 1 - r^2 y^2, as in the
// two-part loop), since these few pairs carry most of a target's rounding.
template <bool POT, bool LISTED>
__device__ __forceinline__ void df_pair_terms(double r2, double m, double h2, double hinv, double hinv3,
                                              double hinv5, double &mf, double &mg, double &mp)
{
    const double ri = rsqrt(r2);
    const double ri2 = ri * ri;
    mp = m * ri;
    mf = mp * ri2;
    if (LISTED) {
        const double t = fma(-r2, fma(ri, ri, -ri2), fma(-r2, ri2, 1.0));
        mf = fma(mf, 1.5 * t, mf);
        mg = mf * ri2;
        mg = fma(mg, t, mg);
        if (POT) mp = fma(mp, 0.5 * t, mp);
    } else {
        mg = mf * ri2;
    }
    if (less_bits(r2, h2)) {
        double F, Gp, P;
        spline_kernel<double>(sqrt(r2) * hinv, F, Gp, P);
        mf = m * F * hinv3;
        mg = m * Gp * hinv5;
        mp = m * P * hinv;
    }
}

// The listed pairs of target i, added to its running sums.
template <bool POT>
__device__ __noinline__ void df_flush(const double *__restrict__ pos, const double *__restrict__ vel,
                                      const double *__restrict__ mass, double h, int64_t i,
                                      const int32_t *list, int cnt, double *sum, int stride)
{
    double acc[kNCPot];
#pragma unroll
    for (int c = 0; c < kNCPot; ++c) acc[c] = 0.0;
    const double xi[3] = {pos[3 * i], pos[3 * i + 1], pos[3 * i + 2]};
    const double vi[3] = {vel[3 * i], vel[3 * i + 1], vel[3 * i + 2]};
    const double h2 = h * h, hinv = 1.0 / h;
    const double hinv3 = hinv * hinv * hinv, hinv5 = hinv3 * hinv * hinv;
    for (int k = 0; k < cnt; ++k) {
        const int64_t j = list[k];
        const double dx = pos[3 * j] - xi[0], dy = pos[3 * j + 1] - xi[1], dz = pos[3 * j + 2] - xi[2];
        double mf, mg, mp;
        df_pair_terms<POT, true>(fma(dx, dx, fma(dy, dy, dz * dz)), mass[j], h2, hinv, hinv3, hinv5, mf, mg, mp);
        accumulate_d<POT>(acc, dx, dy, dz, vel[3 * j] - vi[0], vel[3 * j + 1] - vi[1],
                          vel[3 * j + 2] - vi[2], mf, mg, mp);
    }
#pragma unroll
    for (int c = 0; c < (POT ? kNCPot : kNC); ++c) {
        double hi = sum[2 * c * stride], lo = sum[(2 * c + 1) * stride];
        two_sum_ordered(hi, lo, acc[c]);
        sum[2 * c * stride] = hi;
        sum[(2 * c + 1) * stride] = lo;
    }
}

// The marked sources of the sub-block at element `first` in FP64 from the
// caller's arrays: heavy sources, sub-blocks inside the softening, tiles out of the
// two-part ranges.  Each lane loads one source, its velocity relative to the
// tile's, and hands it round: the FP64 unit bounds this loop, and subtracting the
// tile's velocity and comparing r^2 and h^2 in FP64 for every pair, and dividing
// by h for every sub-block, cost a tenth (16384 elements, all pairs here: 21.3 ms,
// now 19.0; eval_f64_kernel 19.2).
// REL: `cv` is the target's own velocity, and each pair takes the difference: the
// loose sub-blocks hold a target's closest pairs, which carry its jerk, and a smooth
// flow cancels in the sums over a tile's velocities (turbulent cloud of 6794 elements,
// rms error of the jerk 5.1e-15 that way, 6.3e-16 this way, for three subtractions a
// pair: 65536 elements in random order 302 -> 326 ms).
template <bool POT, bool REL>
__device__ __forceinline__ void df_fp64_loop(const EvalArgs &a, const double cv[3], int64_t first,
                                             uint32_t marks, const double xi[3], int64_t ti, const DfSoftening &h,
                                             double acc[kNCPot])
{
    const DfMarked s(marks, ti - first);
    const int64_t own = first + s.own;
    double x[3], v[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        x[c] = a.pos[3 * own + c];
        v[c] = REL ? a.vel[3 * own + c] : a.vel[3 * own + c] - cv[c];
    }
    const double m = a.mass[own];
#pragma unroll 4
    for (int k = 0; k < s.count; ++k) {
        const double dx = __shfl_sync(0xffffffffu, x[0], k) - xi[0], dy = __shfl_sync(0xffffffffu, x[1], k) - xi[1],
                     dz = __shfl_sync(0xffffffffu, x[2], k) - xi[2];
        double mf, mg, mp;
        df_pair_terms<POT, false>(fma(dx, dx, fma(dy, dy, dz * dz)), __shfl_sync(0xffffffffu, m, k), h.h2, h.hinv,
                                  h.hinv3, h.hinv5, mf, mg, mp);
        if (k == s.self) {
            mf = 0.0;
            mg = 0.0;
            mp = 0.0;
        }
        double u[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            u[c] = __shfl_sync(0xffffffffu, v[c], k);
            if (REL) u[c] -= cv[c];
        }
        accumulate_d<POT>(acc, dx, dy, dz, u[0], u[1], u[2], mf, mg, mp);
    }
}

template <int NT, int S, bool POT>
__device__ __forceinline__ bool df_item(const EvalArgs &a, DfSmem<NT, S, POT> &sm, Ring &ring,
                                        const ItemSpec &it)
{
    constexpr int NSTAGE = DfSmem<NT, S, POT>::kStages;
    constexpr int NC = DfSmem<NT, S, POT>::NC;
    const char *src = static_cast<const char *>(a.src);
    const int t_begin = it.t_begin, t_end = it.t_end;

    const int64_t i = item_target(it, it.slot0 + threadIdx.x, a.flags);
    double xi[3] = {0, 0, 0}, vi[3] = {0, 0, 0};
    if (i >= 0) {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            xi[c] = a.pos[3 * i + c];
            vi[c] = a.vel[3 * i + c];
        }
    }
    double *sum = &sm.sum[0][0][threadIdx.x];
#pragma unroll
    for (int c = 0; c < 2 * NC; ++c) sum[c * NT] = 0.0;
    if (threadIdx.x == 0) {
        for (int s = 0; s < NSTAGE; ++s) {
            const int t = t_begin + s;
            if (t < t_end) {
                tma_load_1d(sm.stage[s], src + t * df_stride<S>(), df_bytes<S>(), &sm.bar[s]);
                sm.issued[s] += 1u;
            }
        }
    }
    const bool live = i >= 0;
    const bool warp_live = __any_sync(0xffffffffu, live);
    int32_t list[kDfList];
    int cnt = 0;

    for (int t = t_begin; t < t_end; ++t) {
        const int s = (t - t_begin) % NSTAGE;
        const bool got = mbar_wait_warp(&sm.bar[s], (ring.parity >> s) & 1u, a.flags);
        if (got)
            ring.parity ^= 1u << s;
        else
            atomicExch(&sm.abort_flag, 1);
        if (warp_live && got) {
            const TileGeom g = a.geo[t];
            const float *tile = sm.stage[s];
            const DfHead head = *reinterpret_cast<const DfHead *>(tile);
            DfTarget tg;
            DfClass k;
            const int el = head.el, n_sub = (head.count + kDfSub - 1) / kDfSub;
            if (head.ok) {
                const double il = df_offset(head, g.c, xi, tg);
                k = df_classify<S, true>(tile, head, tg, live, a.h, il);
            } else {
                k.direct = (1u << n_sub) - 1u;
                k.loose = 0;
            }
            const double vr[3] = {vi[0] - (double)g.cv[0], vi[1] - (double)g.cv[1],
                                  vi[2] - (double)g.cv[2]};
            double acc[kNCPot];
#pragma unroll
            for (int c = 0; c < kNCPot; ++c) acc[c] = 0.0;
            const int n_df = n_sub - __popc(k.direct);
            if (n_df > 0) {
                DfSum sums[kDfSums];
#pragma unroll
                for (int c = 0; c < kDfSums; ++c) sums[c] = DfSum{0u, 0u, make_float2(0.0f, 0.0f)};
                const DfWindows w = df_windows(k.rmin2);
                const float4 *P = reinterpret_cast<const float4 *>(tile + df_records<S>());
                for (int q = 0; q < n_sub; ++q) {
                    if ((k.direct >> q) & 1u) continue;
                    if ((k.close >> q) & 1u) {
                        if (__any_sync(0xffffffffu, cnt > kDfList - kDfSub)) {
                            if (cnt > 0) df_flush<POT>(a.pos, a.vel, a.mass, a.h, i, list, cnt, sum, NT);
                            cnt = 0;
                            __syncwarp();
                        }
                        const int64_t j0 = g.first + kDfSub * q;
                        auto add = [&](int j) {
                            if (live && j0 + j != i) list[cnt++] = (int32_t)(j0 + j);
                        };
                        df_sub_loop<POT, true>(P + 7 * (kDfSub / 2) * q, tg, w,
                                               df_radius2(k, df_diagonal2(tile + kDfHeader + 6 * q)), sums,
                                               add);
                    } else {
                        df_sub_loop<POT, false>(P + 7 * (kDfSub / 2) * q, tg, w, 0.0f, sums, [](int) {});
                    }
                }
                // FP64 sums of the tile, back in the caller's units
                const uint32_t n1 = kDfSub * n_df, n2 = n1 + n1 / kDfCarry;
                auto value = [&](int c, float C, double unit) { return df_value(sums[c], C, n1, n2, unit); };
                const double M = head.munit;
                const double ua = __dmul_rn(M, pow2d(-2 * el)), ut = __dmul_rn(M, pow2d(-3 * el)),
                             uj = __dmul_rn(ut, pow2d(head.ev));
                // the squares of the separations' low parts, which r^-3 takes
                // into account and the remaining r^-2 does not: in the diagonal
                // products they cancel against the missing e^2 of d^2, off the
                // diagonal their mean is left (e uniform within half a unit of
                // d, mantissas uniform: 2^-46 / 24 of r^2)
                const double uo = __dmul_rn(ut, 1.0 - 0x1p-46 / 24.0);
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    acc[A0 + c] = value(DA + c, w.a, ua);
                    acc[J10 + c] = value(DJ1 + c, w.j, uj);
                    acc[J20 + c] = value(DJ2 + c, w.j, uj);
                }
#pragma unroll
                for (int c = 0; c < 6; ++c) acc[TXX + c] = value(DT + c, w.t, c < 3 ? ut : uo);
                if (POT) acc[PSUM] = value(DP, w.p, __dmul_rn(M, pow2d(-el)));
                // beyond the softening m f = m g' r^2
                acc[FSUM] = __dadd_rn(__dadd_rn(acc[TXX], acc[TYY]), acc[TZZ]);
            }
            const bool any = df_any_fp64<S>(tile, k.direct, n_sub);
            if (any && (k.direct != k.loose || df_any_fp64<S>(tile, 0u, n_sub))) {
                const DfSoftening h(a.h);
                const double cv[3] = {(double)g.cv[0], (double)g.cv[1], (double)g.cv[2]};
                for (int q = 0; q < n_sub; ++q) {
                    const uint32_t marks = df_fp64_sources<S>(tile, k.direct, q, min(kDfSub, head.count - kDfSub * q));
                    if (marks && !((k.loose >> q) & 1u))
                        df_fp64_loop<POT, false>(a, cv, g.first + (int64_t)kDfSub * q, marks, xi, i, h, acc);
                }
            }
            target_velocity_d(acc, vr);
            if (k.loose) {                       // (with the target's velocity in every pair)
                const DfSoftening h(a.h);
                for (int q = 0; q < n_sub; ++q)
                    if ((k.loose >> q) & 1u)
                        df_fp64_loop<POT, true>(a, vi, g.first + (int64_t)kDfSub * q,
                                                0xffffffffu >> (kDfSub - min(kDfSub, head.count - kDfSub * q)), xi, i, h,
                                                acc);
            }
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                double hi = sum[2 * c * NT], lo2 = sum[(2 * c + 1) * NT];
                two_sum_ordered(hi, lo2, acc[c]);
                sum[2 * c * NT] = hi;
                sum[(2 * c + 1) * NT] = lo2;
            }
        }
        // this warp is done reading stage s; the last warp refills it
        __syncwarp();
        if ((threadIdx.x & 31) == 0) {
            __threadfence_block();
            const int prev = atomicAdd(&sm.done[s], 1);
            if (prev == NT / 32 - 1) {
                sm.done[s] = 0;
                __threadfence_block();
                if (t + NSTAGE < t_end && !*(volatile int *)&sm.abort_flag) {
                    fence_proxy_async_smem();
                    tma_load_1d(sm.stage[s], src + (t + NSTAGE) * df_stride<S>(), df_bytes<S>(), &sm.bar[s]);
                    sm.issued[s] += 1u;
                }
            }
        }
        __syncwarp();
        if (__any_sync(0xffffffffu, *(volatile int *)&sm.abort_flag)) break;
    }
    // warps leave the tile loop at different times: a uniform status
    __syncthreads();
    if (cnt > 0) df_flush<POT>(a.pos, a.vel, a.mass, a.h, i, list, cnt, sum, NT);
    if (live || it.split > 1) {
        double total[kNCPot];
#pragma unroll
        for (int c = 0; c < kNCPot; ++c)
            total[c] = c < NC ? __dadd_rn(sum[2 * c * NT], sum[(2 * c + 1) * NT]) : 0.0;
        if (it.split == 1)
            write_target<POT, false>(a, i, total);
        else if (warp_live)
            write_partial<NC>(a, it.sp, it.rows, it.slot0 + threadIdx.x, total);
    }
    return !sm.abort_flag;
}

template <int NT, int S, bool POT>
__global__ void __launch_bounds__(NT, 384 / NT)
eval_df_kernel(const EvalArgs a)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    auto &sm = *reinterpret_cast<DfSmem<NT, S, POT> *>(smem_raw);
    init_mixed_ring(sm);
    Ring ring{0u, 0u};
    const int64_t n_act = active_count(a);
    const int64_t n_tb = (n_act + NT - 1) / NT;
    const int split = choose_split(n_tb, a.n_tiles, a.grid, a.max_split, a.part_cap_rows, NT);
    const int64_t items = n_tb * split;
    for (int64_t item = blockIdx.x; item < items; item += gridDim.x) {
        const uint32_t tb = (uint32_t)item / (uint32_t)split;
        const int sp = (int)((uint32_t)item - tb * (uint32_t)split);
        ItemSpec it;
        it.idx = a.idx;
        it.slot0 = (int64_t)tb * NT;
        it.slot_end = n_act;
        it.elem_lo = 0;
        it.elem_hi = a.n_src;
        it.t_begin = chunk_begin(sp, a.n_tiles, split);
        it.t_end = chunk_begin(sp + 1, a.n_tiles, split);
        it.sp = sp;
        it.split = split;
        it.rows = n_tb * NT;
        it.tile0 = 0;
        it.pad = 0;
        if (!df_item<NT, S, POT>(a, sm, ring, it)) break;
        __syncthreads();
    }
    drain_mixed_ring(sm, ring, a.flags);
}

template <int NT, int S, bool POT>
__global__ void __launch_bounds__(NT, 384 / NT)
eval_df_batched_kernel(const EvalArgs a, const BatchView b)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    auto &sm = *reinterpret_cast<DfSmem<NT, S, POT> *>(smem_raw);
    __shared__ EvalArgs sa;   // the launch's arguments with the item's system's softening
    if (threadIdx.x == 0) sa = a;
    init_mixed_ring(sm);
    Ring ring{0u, 0u};
    const int64_t total = b.hdr->total_items;
    for (;;) {
        if (threadIdx.x < 32) {
            const int64_t tk = take_item(b, total);
            if (threadIdx.x == 0) {
                sm.ticket = tk;
                if (tk >= 0) {
                    const double hs = b.sys[b.order[item_rank(b, tk)]].h;
                    set_softening(sa, hs > 0.0 ? hs : a.h);
                }
            }
        }
        __syncthreads();
        const int64_t ticket = sm.ticket;
        __syncthreads();
        if (ticket < 0) break;
        const int r = item_rank(b, ticket);
        const int s = b.order[r];
        ItemSpec it;
        it.idx = a.idx;
        it.slot0 = (int64_t)b.idx_lo[s] + (ticket - b.item_off[r]) * NT;
        it.slot_end = b.idx_hi[s];
        it.elem_lo = b.sys[s].offset;
        it.elem_hi = b.sys[s].offset + b.sys[s].n;
        it.t_begin = b.tile_off[s];
        it.t_end = b.tile_off[s + 1];
        it.sp = 0;
        it.split = 1;
        it.rows = 0;
        it.tile0 = b.tile_off[s];
        it.pad = 0;
        if (!df_item<NT, S, POT>(sa, sm, ring, it)) break;
        __syncthreads();
    }
    drain_mixed_ring(sm, ring, a.flags);
}

}  // namespace grav
