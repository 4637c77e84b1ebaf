// K7: adjoint of the force evaluation (reverse mode), all n elements targets.
//
// For a loss L(a, W) with a_bar = dL/da and w_bar = dL/dW (W = 1/2 sum m Phi):
//   pos_bar_k  = T_k a_bar_k + G m_k sum_{i!=k} [ f a_bar_i + g d (d . a_bar_i) ]
//                - w_bar m_k a_k
//   mass_bar_k = -G sum_{i!=k} f (d . a_bar_i) + w_bar Phi_k,      d = x_i - x_k,
// obtained by differentiating a_i = G sum_j m_j f(r) d (Eq. 4's acceleration)
// with respect to x_k and m_k; T_k = d a_k / d x_k is the forward tidal tensor.
// The paper has no adjoint.  The kernels are the forward direct sum with the
// source attribute a_bar_i in place of (v_i, m_i) (FP64: backward_kernel, pair
// terms in two-part FP32 as in grav_df.cuh;
// mixed: backward_pair_kernel on the forward's paired FP32x2 tile layout and
// per-warp TMA ring): per pair they accumulate
//   X1 += f a_bar_i,   X2 += g' (d . a_bar_i) d,   MB += f (d . a_bar_i)
// with g' = -g/3, recomputing every pair term instead of storing any, and the
// epilogue forms pos_bar = T a_bar + G m (X1 - 3 X2) - w_bar m a.
#include <cmath>
#include <mutex>

#include "grav_eval.cuh"

namespace grav {
namespace {

constexpr int kNB = 7;
enum { X10 = 0, X20 = 3, MBS = 6 };

struct BwdArgs {
    int64_t n;
    const TileGeom *geo;
    const void *src;
    int32_t n_tiles;
    int32_t max_split;
    int32_t grid;
    int32_t pad0;
    double *part;
    int64_t part_cap_rows;
    const double *pos, *mass, *a_bar;
    double w_bar;
    const double *acc, *tidal, *pot;
    double G, h;
    float h2f_up, hinvf;
    double *pos_bar, *mass_bar;
    int32_t *flags;
    const float *src_lo;   // mixed: per tile, kLoPlanes planes (x, y, z) of the offsets' low parts
};

__device__ __forceinline__ void bwd_write(const BwdArgs &a, int64_t k, const double s[kNB])
{
    const double m = a.mass[k];
    double px[3] = {0.0, 0.0, 0.0};
    double pm = 0.0;
    if (a.a_bar) {
        const double *t6 = a.tidal + 6 * k;
        const double *ak = a.a_bar + 3 * k;
        // (explicit fused multiply-adds: the same roundings in every kernel)
        px[0] = fma(t6[0], ak[0], fma(t6[3], ak[1], t6[4] * ak[2]));
        px[1] = fma(t6[3], ak[0], fma(t6[1], ak[1], t6[5] * ak[2]));
        px[2] = fma(t6[4], ak[0], fma(t6[5], ak[1], t6[2] * ak[2]));
        const double gm = a.G * m;
#pragma unroll
        for (int c = 0; c < 3; ++c) px[c] = fma(gm, fma(-3.0, s[X20 + c], s[X10 + c]), px[c]);
        pm = -a.G * s[MBS];
    }
    if (a.w_bar != 0.0) {
        const double wm = a.w_bar * m;
#pragma unroll
        for (int c = 0; c < 3; ++c) px[c] = fma(-wm, a.acc[3 * k + c], px[c]);
        pm = fma(a.w_bar, a.pot[k], pm);
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) a.pos_bar[3 * k + c] = px[c];
    a.mass_bar[k] = pm;
}

// One work item of the adjoint: the targets k0 + slot (slot < BT, below
// k_end) against the source tiles [t_begin, t_end).  With split > 1 the sums
// go to partial row slot0 + slot of chunk sp (rows per chunk), else straight
// to the outputs.
struct BwdItem {
    int64_t k0, k_end, slot0, rows;
    int32_t t_begin, t_end, sp, split;
};

// Shared memory of the FP64 adjoint: a two-stage ring of two-part (x, a_bar)
// tiles, and the targets' running FP64 sums (hi, lo).
template <int NT, int S>
struct BwdDfSmem {
    static constexpr int kStages = 2;
    float stage[kStages][df_words<S>()];
    double sum[kNB][2][NT];
    uint64_t bar[kStages];
    int done[kStages];           // warps finished with the tile in each stage
    unsigned issued[kStages];    // copies issued into each stage
    int abort_flag;
    long long ticket;
};

// One sub-block of 32 sources of the FP64 adjoint in two-part arithmetic (the
// forward's df_sub_loop with a_bar in the velocity's place and no mass).
template <bool LIST, typename Add>
__device__ __forceinline__ void bwd_df_loop(const float4 *__restrict__ P, const DfTarget &tg, float w3,
                                            float w2, float thr2, DfSum (&sums)[kNB], Add &&list)
{
    const float2 C3 = dup2(w3), C32 = dup2(df_second(w3)), C2 = dup2(w2), C22 = dup2(df_second(w2));
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
            const float4 q3 = r[3], q4 = r[4], q5 = r[5];
            float2 ah[3] = {make_float2(q3.x, q3.y), make_float2(q3.z, q3.w), make_float2(q4.x, q4.y)};
            float2 al[3] = {make_float2(q4.z, q4.w), make_float2(q5.x, q5.y), make_float2(q5.z, q5.w)};
            if (LIST && !(fminf(r2h.x, r2h.y) >= thr2)) {
                // (listed, or padding: no a_bar at distance 1 instead)
                if (!(r2h.x >= thr2)) {
                    list(2 * k);
#pragma unroll
                    for (int c = 0; c < 3; ++c) ah[c].x = al[c].x = 0.0f;
                    r2l.x = sq.x = 0.0f;
                    r2h.x = 1.0f;
                }
                if (!(r2h.y >= thr2)) {
                    list(2 * k + 1);
#pragma unroll
                    for (int c = 0; c < 3; ++c) ah[c].y = al[c].y = 0.0f;
                    r2l.y = sq.y = 0.0f;
                    r2h.y = 1.0f;
                }
            }
            const DfInv inv = df_inverse(r2h, r2l, sq);
            float2 fh, fl, gh, gl, dah, dal, xh, xl;
            df_inv3(inv, fh, fl);
            df_times_inv2(inv, fh, fl, gh, gl);
            df_dot3(d, e, ah, al, dah, dal);
            df_mul(gh, gl, dah, dal, xh, xl);
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                df_add_product(sums[X10 + c], C3, C32, fh, fl, ah[c], al[c]);
                df_add_product(sums[X20 + c], C3, C32, xh, xl, d[c], e[c]);
            }
            df_add_product(sums[MBS], C2, C22, fh, fl, dah, dal);
        }
#pragma unroll
        for (int c = 0; c < kNB; ++c) df_carry(sums[c], c == MBS ? C22 : C32);
    }
}

// One pair of the adjoint in FP64 (d, a_bar given): added to s[kNB].
__device__ __forceinline__ void bwd_pair_fp64(const double d[3], const double ab[3], double h2, double hinv,
                                              double hinv3, double hinv5, bool self, double s[kNB])
{
    const double r2 = fma(d[0], d[0], fma(d[1], d[1], d[2] * d[2]));
    const double ri = rsqrt(r2);
    const double ri2 = ri * ri;
    double f = ri * ri2;
    double gp = f * ri2;
    if (less_bits(r2, h2)) {
        double F, Gp, P;
        spline_kernel<double>(sqrt(r2) * hinv, F, Gp, P);
        f = F * hinv3;
        gp = Gp * hinv5;
        if (self) {
            f = 0.0;
            gp = 0.0;
        }
    }
    const double da = fma(d[0], ab[0], fma(d[1], ab[1], d[2] * ab[2]));
    const double gd = gp * da;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        s[X10 + c] = fma(f, ab[c], s[X10 + c]);
        s[X20 + c] = fma(gd, d[c], s[X20 + c]);
    }
    s[MBS] = fma(f, da, s[MBS]);
}

__device__ __forceinline__ void bwd_add_sums(double *sum, int stride, const double acc[kNB])
{
#pragma unroll
    for (int c = 0; c < kNB; ++c) {
        double hi = sum[2 * c * stride], lo = sum[(2 * c + 1) * stride];
        two_sum_ordered(hi, lo, acc[c]);
        sum[2 * c * stride] = hi;
        sum[(2 * c + 1) * stride] = lo;
    }
}

// The listed pairs of target k, added to its running sums.
__device__ __noinline__ void bwd_df_flush(const double *__restrict__ pos, const double *__restrict__ a_bar,
                                          double h, int64_t k, const int32_t *list, int cnt, double *sum,
                                          int stride)
{
    double acc[kNB];
#pragma unroll
    for (int c = 0; c < kNB; ++c) acc[c] = 0.0;
    const double xk[3] = {pos[3 * k], pos[3 * k + 1], pos[3 * k + 2]};
    const double h2 = h * h, hinv = 1.0 / h;
    const double hinv3 = hinv * hinv * hinv, hinv5 = hinv3 * hinv * hinv;
    for (int q = 0; q < cnt; ++q) {
        const int64_t j = list[q];
        const double d[3] = {pos[3 * j] - xk[0], pos[3 * j + 1] - xk[1], pos[3 * j + 2] - xk[2]};
        const double ab[3] = {a_bar[3 * j], a_bar[3 * j + 1], a_bar[3 * j + 2]};
        bwd_pair_fp64(d, ab, h2, hinv, hinv3, hinv5, false, acc);
    }
    bwd_add_sums(sum, stride, acc);
}

// A tile's sources that go to FP64 (reasons: df_fp64_loop of the forward).  Not
// inlined: its registers are not the two-part loop's (12289 elements of like a_bar
// 1.74 ms inlined, 1.69 ms; all in FP64 7.24 ms, 7.19 ms; FP64 tiles throughout 7.47 ms).
template <int S>
__device__ __noinline__ void bwd_fp64_tile(const double *__restrict__ pos, const double *__restrict__ a_bar,
                                           double h, const float *tile, uint32_t direct, int64_t first_of_tile,
                                           int count, double xk, double yk, double zk, int64_t ti,
                                           double sums[kNB])
{
    const DfSoftening hk(h);
    const double at[3] = {xk, yk, zk};
    double acc[kNB];
#pragma unroll
    for (int c = 0; c < kNB; ++c) acc[c] = sums[c];
    for (int q = 0; q < (count + kDfSub - 1) / kDfSub; ++q) {
        const uint32_t marks = df_fp64_sources<S>(tile, direct, q, min(kDfSub, count - kDfSub * q));
        if (!marks) continue;
        const int64_t first = first_of_tile + kDfSub * q;
        const DfMarked s(marks, ti - first);
        double x[3], b[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            x[c] = pos[3 * (first + s.own) + c];
            b[c] = a_bar[3 * (first + s.own) + c];
        }
#pragma unroll 2
        for (int p = 0; p < s.count; ++p) {
            double d[3], ab[3];
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                d[c] = __shfl_sync(0xffffffffu, x[c], p) - at[c];
                ab[c] = __shfl_sync(0xffffffffu, b[c], p);
            }
            bwd_pair_fp64(d, ab, hk.h2, hk.hinv, hk.hinv3, hk.hinv5, p == s.self, acc);
        }
    }
#pragma unroll
    for (int c = 0; c < kNB; ++c) sums[c] = acc[c];
}

// One item of the FP64 adjoint (structure and reasons: df_item of the forward,
// grav_eval_df.cuh); false once a bounded wait gave up.
template <int NT, int S>
__device__ __forceinline__ bool bwd_df_item(const BwdArgs &a, BwdDfSmem<NT, S> &sm, Ring &ring,
                                            const BwdItem &it, double h)
{
    constexpr int NSTAGE = BwdDfSmem<NT, S>::kStages;
    const char *src = static_cast<const char *>(a.src);
    const int t_begin = it.t_begin, t_end = it.t_end;
    const int64_t i = it.k0 + threadIdx.x;
    const bool live = i < it.k_end;
    double xk[3] = {0.0, 0.0, 0.0};
    if (live) {
#pragma unroll
        for (int c = 0; c < 3; ++c) xk[c] = a.pos[3 * i + c];
    }
    double *sum = &sm.sum[0][0][threadIdx.x];
#pragma unroll
    for (int c = 0; c < 2 * kNB; ++c) sum[c * NT] = 0.0;
    if (threadIdx.x == 0) {
        for (int s = 0; s < NSTAGE; ++s) {
            const int t = t_begin + s;
            if (t < t_end) {
                tma_load_1d(sm.stage[s], src + t * df_stride<S>(), df_bytes<S>(), &sm.bar[s]);
                sm.issued[s] += 1u;
            }
        }
    }
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
                const double il = df_offset(head, g.c, xk, tg);
                k = df_classify<S, false>(tile, head, tg, live, h, il);
            } else {
                k.direct = (1u << n_sub) - 1u;
            }
            double acc[kNB];
#pragma unroll
            for (int c = 0; c < kNB; ++c) acc[c] = 0.0;
            const int n_df = n_sub - __popc(k.direct);
            if (n_df > 0) {
                DfSum sums[kNB];
#pragma unroll
                for (int c = 0; c < kNB; ++c) sums[c] = DfSum{0u, 0u, make_float2(0.0f, 0.0f)};
                const float i1 = rsqrt_sfu(k.rmin2) * (1.0f + 0x1p-18f);
                // f a_bar, g (d.a_bar) d <= sqrt(3) r^-3; f (d.a_bar) <= sqrt(3) r^-2
                const float w3 = df_window(1.8f * (i1 * i1 * i1)), w2 = df_window(1.8f * (i1 * i1));
                const float4 *P = reinterpret_cast<const float4 *>(tile + df_records<S>());
                for (int q = 0; q < n_sub; ++q) {
                    if ((k.direct >> q) & 1u) continue;
                    const float4 *Pq = P + 7 * (kDfSub / 2) * q;
                    if ((k.close >> q) & 1u) {
                        if (__any_sync(0xffffffffu, cnt > kDfList - kDfSub)) {
                            if (cnt > 0) bwd_df_flush(a.pos, a.a_bar, h, i, list, cnt, sum, NT);
                            cnt = 0;
                            __syncwarp();
                        }
                        const int64_t j0 = g.first + kDfSub * q;
                        // (not padding, not the heavy ones)
                        const uint32_t light = (0xffffffffu >> (kDfSub - min(kDfSub, head.count - kDfSub * q))) &
                                               ~df_heavy<S>(tile, q);
                        auto add = [&](int j) {
                            if (live && (light >> j & 1u) && j0 + j != i) list[cnt++] = (int32_t)(j0 + j);
                        };
                        bwd_df_loop<true>(Pq, tg, w3, w2,
                                          df_radius2(k, df_diagonal2(tile + kDfHeader + 6 * q)), sums, add);
                    } else {
                        bwd_df_loop<false>(Pq, tg, w3, w2, 0.0f, sums, [](int) {});
                    }
                }
                const uint32_t n1 = kDfSub * n_df, n2 = n1 + n1 / kDfCarry;
                const double u3 = pow2d(head.ev - 3 * el), u2 = pow2d(head.ev - 2 * el);
#pragma unroll
                for (int c = 0; c < kNB; ++c)
                    acc[c] = df_value(sums[c], c == MBS ? w2 : w3, n1, n2, c == MBS ? u2 : u3);
            }
            if (df_any_fp64<S>(tile, k.direct, n_sub))
                bwd_fp64_tile<S>(a.pos, a.a_bar, h, tile, k.direct, g.first, head.count, xk[0], xk[1], xk[2], i,
                                 acc);
            bwd_add_sums(sum, NT, acc);
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
    __syncthreads();   // every warp is out of the tile loop: a uniform status
    if (cnt > 0) bwd_df_flush(a.pos, a.a_bar, h, i, list, cnt, sum, NT);
    if (live) {
        double total[kNB];
#pragma unroll
        for (int c = 0; c < kNB; ++c) total[c] = __dadd_rn(sum[2 * c * NT], sum[(2 * c + 1) * NT]);
        if (it.split == 1) {
            bwd_write(a, i, total);
        } else {
            const int64_t slot = it.slot0 + threadIdx.x;
#pragma unroll
            for (int c = 0; c < kNB; ++c) a.part[((int64_t)it.sp * kNB + c) * it.rows + slot] = total[c];
        }
    }
    return !sm.abort_flag;
}

// The FP64 adjoint over all n elements: work items of target blocks x source
// chunks.
template <int NT, int S, int MINB>
__global__ void __launch_bounds__(NT, MINB)
backward_kernel(const BwdArgs a)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    auto &sm = *reinterpret_cast<BwdDfSmem<NT, S> *>(smem_raw);
    init_mixed_ring(sm);
    Ring ring{0u, 0u};
    const int64_t n_tb = (a.n + NT - 1) / NT;
    const int split = choose_split(n_tb, a.n_tiles, a.grid, a.max_split, a.part_cap_rows, NT);
    const int64_t items = n_tb * split;
    for (int64_t item = blockIdx.x; item < items; item += gridDim.x) {
        const uint32_t tb = (uint32_t)item / (uint32_t)split;      // (32 bits, as the forward's)
        const int sp = (int)((uint32_t)item - tb * (uint32_t)split);
        BwdItem it;
        it.k0 = (int64_t)tb * NT;
        it.k_end = a.n;
        it.slot0 = (int64_t)tb * NT;
        it.rows = n_tb * NT;
        it.t_begin = chunk_begin(sp, a.n_tiles, split);
        it.t_end = chunk_begin(sp + 1, a.n_tiles, split);
        it.sp = sp;
        it.split = split;
        if (!bwd_df_item<NT, S>(a, sm, ring, it, a.h)) break;
        __syncthreads();
    }
    drain_mixed_ring(sm, ring, a.flags);
}

// Batched FP64 adjoint: the items of all systems from the plan, taken from
// the per-SM queues; each system's targets against its own tiles with its own
// support h (grav_system.h, or the call's h where it is 0).
template <int NT, int S, int MINB>
__global__ void __launch_bounds__(NT, MINB)
backward_batched_kernel(const BwdArgs a, const BatchView b)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    auto &sm = *reinterpret_cast<BwdDfSmem<NT, S> *>(smem_raw);
    init_mixed_ring(sm);
    Ring ring{0u, 0u};
    const int64_t total = b.hdr->total_items;
    for (;;) {
        if (threadIdx.x < 32) {
            const int64_t tk = take_item(b, total);
            if (threadIdx.x == 0) sm.ticket = tk;
        }
        __syncthreads();
        const int64_t ticket = sm.ticket;
        __syncthreads();
        if (ticket < 0) break;
        const int r = item_rank(b, ticket);
        const int s = b.order[r];
        const double h = b.sys[s].h > 0.0 ? b.sys[s].h : a.h;
        BwdItem it;
        it.k0 = (int64_t)b.idx_lo[s] + (ticket - b.item_off[r]) * NT;
        it.k_end = b.idx_hi[s];
        it.slot0 = 0;
        it.rows = 0;
        it.t_begin = b.tile_off[s];
        it.t_end = b.tile_off[s + 1];
        it.sp = 0;
        it.split = 1;
        if (!bwd_df_item<NT, S>(a, sm, ring, it, h)) break;
        __syncthreads();
    }
    drain_mixed_ring(sm, ring, a.flags);
}

// Mixed adjoint on the paired source layout of the forward kernel (the
// packer's velocity slots carry a_bar_i, its mass slots are unused): two
// sources per packed FP32x2 instruction in the Newtonian loop, 20 such
// instructions per source pair (the scalar loop's 20 per source).
template <int KT, int S, int U>
__device__ __forceinline__ void bwd_far_pair(const float *__restrict__ tile, const float tx[KT][3],
                                             float2 acc[KT][kNB])
{
    const float4 *P0 = reinterpret_cast<const float4 *>(tile);
    const float4 *P1 = P0 + S / 2;
    const float4 *V0 = P1 + S / 2;
    const float2 *V1 = reinterpret_cast<const float2 *>(V0 + S / 2);
    float2 ntx[KT], nty[KT], ntz[KT];
#pragma unroll
    for (int q = 0; q < KT; ++q) {
        ntx[q] = make_float2(-tx[q][0], -tx[q][0]);
        nty[q] = make_float2(-tx[q][1], -tx[q][1]);
        ntz[q] = make_float2(-tx[q][2], -tx[q][2]);
    }
#pragma unroll U
    for (int k = 0; k < S / 2; ++k) {
        const float4 p0 = P0[k], p1 = P1[k], v0 = V0[k];
        const float2 bz = V1[k];
        const float2 bx = make_float2(v0.x, v0.y), by = make_float2(v0.z, v0.w);
#pragma unroll
        for (int q = 0; q < KT; ++q) {
            const float2 dx = __fadd2_rn(make_float2(p0.x, p0.y), ntx[q]);
            const float2 dy = __fadd2_rn(make_float2(p0.z, p0.w), nty[q]);
            const float2 dz = __fadd2_rn(make_float2(p1.x, p1.y), ntz[q]);
            float2 r2 = __fmul2_rn(dz, dz);
            r2 = __ffma2_rn(dy, dy, r2);
            r2 = __ffma2_rn(dx, dx, r2);
            const float2 ri = make_float2(rsqrt_sfu(r2.x), rsqrt_sfu(r2.y));
            const float2 ri2 = __fmul2_rn(ri, ri);
            const float2 f = __fmul2_rn(ri, ri2);
            const float2 gp = __fmul2_rn(f, ri2);
            float2 da = __fmul2_rn(dz, bz);
            da = __ffma2_rn(dy, by, da);
            da = __ffma2_rn(dx, bx, da);
            acc[q][X10 + 0] = __ffma2_rn(f, bx, acc[q][X10 + 0]);
            acc[q][X10 + 1] = __ffma2_rn(f, by, acc[q][X10 + 1]);
            acc[q][X10 + 2] = __ffma2_rn(f, bz, acc[q][X10 + 2]);
            const float2 gd = __fmul2_rn(gp, da);
            acc[q][X20 + 0] = __ffma2_rn(gd, dx, acc[q][X20 + 0]);
            acc[q][X20 + 1] = __ffma2_rn(gd, dy, acc[q][X20 + 1]);
            acc[q][X20 + 2] = __ffma2_rn(gd, dz, acc[q][X20 + 2]);
            acc[q][MBS] = __ffma2_rn(f, da, acc[q][MBS]);
        }
    }
}

// Pairs of one target summed in FP64 after its tiles (at most this many per
// target; past that a pair stays in the FP32 sums).
constexpr int kBwdCloseList = 64;

// Near and loose tiles on the paired layout: the pair terms of two sources at
// a time in FP32x2, the sums source by source in order (lane x of the
// accumulators), the self pair excluded by index.  Separations are formed
// from both offsets' high and low parts, d = (s - t) + (s_lo - t_lo) (lo: the
// tile's planes of low parts; tl: the targets'), so they are good to a few
// units in the last place of d however far the tile centre lies.  A pair
// within 2h of its target is offered to record(q, j) and, when taken, left
// out of the FP32 sums: it is summed in FP64 after the item's tiles, where
// one such pair can outweigh the rest of the target's sum.
template <int KT, int S, typename Record>
__device__ __forceinline__ void bwd_near_pair(const float *__restrict__ tile,
                                              const float *__restrict__ lo, const float tx[KT][3],
                                              const float tl[KT][3], const int64_t tk[KT],
                                              int64_t jbase, float h2, float hinv,
                                              float2 acc[KT][kNB], Record &record)
{
    const float hinv3 = hinv * hinv * hinv;
    const float hinv5 = hinv3 * hinv * hinv;
    const float4 *P0 = reinterpret_cast<const float4 *>(tile);
    const float4 *P1 = P0 + S / 2;
    const float4 *V0 = P1 + S / 2;
    const float2 *V1 = reinterpret_cast<const float2 *>(V0 + S / 2);
    const float2 *L2 = reinterpret_cast<const float2 *>(lo);      // 3 planes of S/2 pairs
#pragma unroll 2
    for (int k = 0; k < S / 2; ++k) {
        const float4 p0 = P0[k], p1 = P1[k], v0 = V0[k];
        const float2 bz = V1[k];
        const float2 bx = make_float2(v0.x, v0.y), by = make_float2(v0.z, v0.w);
        const float2 lx = L2[k], ly = L2[S / 2 + k], lz = L2[S + k];
#pragma unroll
        for (int q = 0; q < KT; ++q) {
            const float2 dx = __fadd2_rn(__fadd2_rn(make_float2(p0.x, p0.y), make_float2(-tx[q][0], -tx[q][0])),
                                         __fadd2_rn(lx, make_float2(-tl[q][0], -tl[q][0])));
            const float2 dy = __fadd2_rn(__fadd2_rn(make_float2(p0.z, p0.w), make_float2(-tx[q][1], -tx[q][1])),
                                         __fadd2_rn(ly, make_float2(-tl[q][1], -tl[q][1])));
            const float2 dz = __fadd2_rn(__fadd2_rn(make_float2(p1.x, p1.y), make_float2(-tx[q][2], -tx[q][2])),
                                         __fadd2_rn(lz, make_float2(-tl[q][2], -tl[q][2])));
            const float2 r2 = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, __fmul2_rn(dz, dz)));
            const float2 ri = make_float2(rsqrt_sfu(r2.x), rsqrt_sfu(r2.y));
            const float2 ri2 = __fmul2_rn(ri, ri);
            float2 f = __fmul2_rn(ri, ri2);
            float2 gp = __fmul2_rn(f, ri2);
            if (fminf(r2.x, r2.y) < 4.0f * h2) {
                // a recorded pair leaves the FP32 sums: its terms become 0
                auto special = [&](float r2s, int64_t jg, float &fs, float &gs) {
                    if (!(r2s < 4.0f * h2)) return;
                    if (tk[q] >= 0 && jg != tk[q] && record(q, jg)) {
                        fs = gs = 0.0f;
                    } else if (r2s < h2) {
                        float F, Gp, P;
                        spline_kernel<float>(sqrtf(r2s) * hinv, F, Gp, P);
                        fs = F * hinv3;
                        gs = Gp * hinv5;
                        if (jg == tk[q]) fs = gs = 0.0f;
                    }
                };
                special(r2.x, jbase + 2 * k, f.x, gp.x);
                special(r2.y, jbase + 2 * k + 1, f.y, gp.y);
            }
            const float2 da = __ffma2_rn(dx, bx, __ffma2_rn(dy, by, __fmul2_rn(dz, bz)));
            const float2 gd = __fmul2_rn(gp, da);
            auto add = [&](float fs, float px, float py, float pz, float ux, float uy, float uz, float ds,
                           float gs) {
                acc[q][X10 + 0].x = fmaf(fs, ux, acc[q][X10 + 0].x);
                acc[q][X10 + 1].x = fmaf(fs, uy, acc[q][X10 + 1].x);
                acc[q][X10 + 2].x = fmaf(fs, uz, acc[q][X10 + 2].x);
                acc[q][X20 + 0].x = fmaf(gs, px, acc[q][X20 + 0].x);
                acc[q][X20 + 1].x = fmaf(gs, py, acc[q][X20 + 1].x);
                acc[q][X20 + 2].x = fmaf(gs, pz, acc[q][X20 + 2].x);
                acc[q][MBS].x = fmaf(fs, ds, acc[q][MBS].x);
            };
            add(f.x, dx.x, dy.x, dz.x, bx.x, by.x, bz.x, da.x, gd.x);
            add(f.y, dx.y, dy.y, dz.y, bx.y, by.y, bz.y, da.y, gd.y);
        }
    }
}

// One listed pair of the mixed adjoint in FP64 (target k at FP64 position
// xk, source i != k), from the FP64 positions and a_bar: added to s[kNB].
__device__ __forceinline__ void bwd_pair_d(const BwdArgs &a, double h, const double xk[3], int64_t i,
                                           double s[kNB])
{
    double d[3], ab[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        d[c] = __dsub_rn(a.pos[3 * i + c], xk[c]);
        ab[c] = a.a_bar[3 * i + c];
    }
    const double r2 = fma(d[0], d[0], fma(d[1], d[1], d[2] * d[2]));
    double f, gp;
    if (r2 < h * h) {
        const double hinv = 1.0 / h;
        double F, Gp, P;
        spline_kernel<double>(sqrt(r2) * hinv, F, Gp, P);
        const double hinv3 = hinv * hinv * hinv;
        f = F * hinv3;
        gp = Gp * hinv3 * hinv * hinv;
    } else {
        const double ri = 1.0 / sqrt(r2);
        f = ri * ri * ri;
        gp = f * ri * ri;
    }
    const double da = fma(d[0], ab[0], fma(d[1], ab[1], d[2] * ab[2]));
    const double gd = gp * da;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        s[X10 + c] = fma(f, ab[c], s[X10 + c]);
        s[X20 + c] = fma(gd, d[c], s[X20 + c]);
    }
    s[MBS] = fma(f, da, s[MBS]);
}

// Shared memory of the mixed adjoint: a three-stage ring of paired tiles.
template <int S>
struct BwdPairSmem {
    static constexpr int kStages = 3;
    // a stage: the paired tile (28 bytes per source), then the low parts of
    // its position offsets (12 bytes per source)
    static constexpr int kTileF4 = 7 * S / 4;
    float4 stage[kStages][kTileF4 + kLoPlanes * S / 4];
    uint64_t bar[kStages];
    int done[kStages];           // warps finished with the tile in each stage
    unsigned issued[kStages];    // copies issued into each stage
    float blo[3], bhi[3];
    int abort_flag;
    long long ticket;
};

template <int S>
__device__ __forceinline__ void bwd_pair_init(BwdPairSmem<S> &sm)
{
    if (threadIdx.x == 0) {
        for (int s = 0; s < BwdPairSmem<S>::kStages; ++s) {
            mbar_init(&sm.bar[s], 1);
            sm.done[s] = 0;
            sm.issued[s] = 0;
        }
        sm.abort_flag = 0;
        fence_barrier_init();
    }
    __syncthreads();
}

// Copies still in flight (only after a timed-out wait): a stage holds one
// exactly when thread 0 has seen fewer completions there than were issued.
template <int S>
__device__ __forceinline__ void bwd_pair_drain(BwdPairSmem<S> &sm, uint32_t parity, int32_t *flags)
{
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int s = 0; s < BwdPairSmem<S>::kStages; ++s)
            if ((sm.issued[s] & 1u) != ((parity >> s) & 1u))
                mbar_wait_bounded(&sm.bar[s], (parity >> s) & 1u, flags);
    }
}

// One item of the mixed adjoint: the structure of the forward mixed kernel
// (a three-stage TMA ring in which each warp releases a stage on its own and
// the last warp to release it issues the refill, each warp's near/far test
// against its own targets' box), with the adjoint's pair terms.  Per-tile
// FP32 sums are carried across tiles as compensated FP32 pairs (TwoSum); the
// result is FP64.  False once a bounded wait gave up.
template <int NT, int KT, int S, int U>
__device__ __forceinline__ bool bwd_pair_item(const BwdArgs &a, BwdPairSmem<S> &sm, uint32_t &parity,
                                              const BwdItem &it, double h, float h2, float hinv)
{
    using Sm = BwdPairSmem<S>;
    constexpr int NSTAGE = Sm::kStages;
    constexpr uint32_t kTileBytes = S * 28;
    const float4 *src = static_cast<const float4 *>(a.src);
    const int t_begin = it.t_begin, t_end = it.t_end;
    // a tile and the low parts of its offsets into stage s
    auto load_stage = [&](int s, int t) {
        tma_load_1d_two(sm.stage[s], src + (int64_t)t * 2 * S, kTileBytes, sm.stage[s] + Sm::kTileF4,
                        a.src_lo + (int64_t)t * kLoPlanes * S, 4u * kLoPlanes * S, &sm.bar[s]);
    };

    double xk[KT][3];
    int64_t tk[KT];
    float lo[3], hi[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        lo[c] = __int_as_float(0x7f800000);
        hi[c] = -__int_as_float(0x7f800000);
    }
#pragma unroll
    for (int q = 0; q < KT; ++q) {
        const int64_t k = it.k0 + (int64_t)q * NT + threadIdx.x;
        tk[q] = k < it.k_end ? k : -1;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            xk[q][c] = tk[q] >= 0 ? a.pos[3 * k + c] : 0.0;
            if (tk[q] >= 0) {
                lo[c] = fminf(lo[c], __double2float_rd(xk[q][c]));
                hi[c] = fmaxf(hi[c], __double2float_ru(xk[q][c]));
            }
        }
    }
    // lo/hi become the warp's box; tiles are tested against it
    block_bbox<NT>(lo, hi, sm.blo, sm.bhi);
    // pairs within 2h, listed per target for FP64
    int32_t nlist[KT][kBwdCloseList];
    int ncnt[KT];
#pragma unroll
    for (int q = 0; q < KT; ++q) ncnt[q] = 0;
    auto record = [&](int q, int64_t j) -> bool {
        if (ncnt[q] >= kBwdCloseList) return false;
        nlist[q][ncnt[q]++] = (int32_t)j;
        return true;
    };

    float shi[KT][kNB], slo[KT][kNB];
#pragma unroll
    for (int q = 0; q < KT; ++q)
#pragma unroll
        for (int c = 0; c < kNB; ++c) {
            shi[q][c] = 0.0f;
            slo[q][c] = 0.0f;
        }
    if (threadIdx.x == 0) {
        for (int s = 0; s < NSTAGE; ++s) {
            const int t = t_begin + s;
            if (t < t_end) {
                load_stage(s, t);
                sm.issued[s] += 1u;
            }
        }
    }
    for (int t = t_begin; t < t_end; ++t) {
        const int s = (t - t_begin) % NSTAGE;
        const TileGeom g = a.geo[t];
        // near: inside h of the warp's box; loose: within reach of the FP32
        // offsets' rounding (as in the forward kernel); both take the near
        // loop with two-part separations
        const float g2 = box_gap2(lo, hi, g);
        constexpr float kL = kLooseC / (1.0f - kLooseC);
        const bool close = !(g2 >= h2) || g2 < (kL * kL) * box_diag2(g.lo, g.hi);
        float tx[KT][3];
#pragma unroll
        for (int q = 0; q < KT; ++q)
#pragma unroll
            for (int c = 0; c < 3; ++c) tx[q][c] = __double2float_rn(__dsub_rn(xk[q][c], g.c[c]));
        const bool got = mbar_wait_bounded(&sm.bar[s], (parity >> s) & 1u, a.flags);
        if (got)
            parity ^= 1u << s;
        else
            atomicExch(&sm.abort_flag, 1);
        float2 acc[KT][kNB];
#pragma unroll
        for (int q = 0; q < KT; ++q)
#pragma unroll
            for (int c = 0; c < kNB; ++c) acc[q][c] = make_float2(0.0f, 0.0f);
        const float *tf = reinterpret_cast<const float *>(sm.stage[s]);
        if (!close) {
            bwd_far_pair<KT, S, U>(tf, tx, acc);
        } else {
            float tl[KT][3];
#pragma unroll
            for (int q = 0; q < KT; ++q)
#pragma unroll
                for (int c = 0; c < 3; ++c)
                    tl[q][c] = __double2float_rn(__dsub_rn(__dsub_rn(xk[q][c], g.c[c]), (double)tx[q][c]));
            bwd_near_pair<KT, S>(tf, reinterpret_cast<const float *>(sm.stage[s] + Sm::kTileF4), tx, tl,
                                 tk, g.first, h2, hinv, acc, record);
        }
#pragma unroll
        for (int q = 0; q < KT; ++q)
#pragma unroll
            for (int c = 0; c < kNB; ++c) two_sum_acc(shi[q][c], slo[q][c], acc[q][c].x + acc[q][c].y);
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
                    load_stage(s, t + NSTAGE);
                    sm.issued[s] += 1u;
                }
            }
        }
        __syncwarp();
        if (*(volatile int *)&sm.abort_flag) break;
    }
    __syncthreads();   // every warp is out of the tile loop: a uniform status
#pragma unroll
    for (int q = 0; q < KT; ++q) {
        double sum[kNB];
#pragma unroll
        for (int c = 0; c < kNB; ++c) sum[c] = 0.0;
        if (tk[q] >= 0)
            for (int k = 0; k < ncnt[q]; ++k) bwd_pair_d(a, h, xk[q], nlist[q][k], sum);
#pragma unroll
        for (int c = 0; c < kNB; ++c) sum[c] += (double)shi[q][c] + (double)slo[q][c];
        const int64_t slot = it.slot0 + (int64_t)q * NT + threadIdx.x;
        if (it.split == 1) {
            if (tk[q] >= 0) bwd_write(a, tk[q], sum);
        } else {
#pragma unroll
            for (int c = 0; c < kNB; ++c) a.part[((int64_t)it.sp * kNB + c) * it.rows + slot] = sum[c];
        }
    }
    return !sm.abort_flag;
}

// The mixed adjoint over all n elements: work items of target blocks x
// source chunks.
template <int NT, int KT, int S, int MINB, int U>
__global__ void __launch_bounds__(NT, MINB) backward_pair_kernel(const BwdArgs a)
{
    constexpr int BT = NT * KT;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    BwdPairSmem<S> &sm = *reinterpret_cast<BwdPairSmem<S> *>(smem_raw);
    bwd_pair_init(sm);
    uint32_t parity = 0;

    const int64_t n_tb = (a.n + BT - 1) / BT;
    const int split = choose_split(n_tb, a.n_tiles, a.grid, a.max_split, a.part_cap_rows, BT);
    const int64_t items = n_tb * split;
    const int64_t rows = n_tb * BT;

    for (int64_t item = blockIdx.x; item < items; item += gridDim.x) {
        const uint32_t tb = (uint32_t)item / (uint32_t)split;      // (32 bits, as the forward's)
        const int sp = (int)((uint32_t)item - tb * (uint32_t)split);
        BwdItem it;
        it.k0 = (int64_t)tb * BT;
        it.k_end = a.n;
        it.slot0 = (int64_t)tb * BT;
        it.rows = rows;
        it.t_begin = chunk_begin(sp, a.n_tiles, split);
        it.t_end = chunk_begin(sp + 1, a.n_tiles, split);
        it.sp = sp;
        it.split = split;
        if (!bwd_pair_item<NT, KT, S, U>(a, sm, parity, it, a.h, a.h2f_up, a.hinvf)) break;
        __syncthreads();
    }
    bwd_pair_drain(sm, parity, a.flags);
}

// Batched mixed adjoint: the items of all systems from the plan, taken
// from the per-SM queues; each system's targets against its own tiles with
// its own support h (grav_system.h, or the call's h where it is 0).
template <int NT, int KT, int S, int MINB, int U>
__global__ void __launch_bounds__(NT, MINB) backward_pair_batched_kernel(const BwdArgs a,
                                                                         const BatchView b)
{
    constexpr int BT = NT * KT;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    BwdPairSmem<S> &sm = *reinterpret_cast<BwdPairSmem<S> *>(smem_raw);
    bwd_pair_init(sm);
    uint32_t parity = 0;
    const int64_t total = b.hdr->total_items;
    for (;;) {
        if (threadIdx.x < 32) {
            const int64_t tk = take_item(b, total);
            if (threadIdx.x == 0) sm.ticket = tk;
        }
        __syncthreads();
        const int64_t ticket = sm.ticket;
        __syncthreads();
        if (ticket < 0) break;
        const int r = item_rank(b, ticket);
        const int s = b.order[r];
        const double h = b.sys[s].h > 0.0 ? b.sys[s].h : a.h;
        float h2f, hinvf;
        softening_f(h, h2f, hinvf);
        BwdItem it;
        it.k0 = (int64_t)b.idx_lo[s] + (ticket - b.item_off[r]) * BT;
        it.k_end = b.idx_hi[s];
        it.slot0 = 0;
        it.rows = 0;
        it.t_begin = b.tile_off[s];
        it.t_end = b.tile_off[s + 1];
        it.sp = 0;
        it.split = 1;
        if (!bwd_pair_item<NT, KT, S, U>(a, sm, parity, it, h, h2f, hinvf)) break;
        __syncthreads();
    }
    bwd_pair_drain(sm, parity, a.flags);
}

// One thread per (target, component) adds the chunk partials (FP64 bound, as
// the forward's reduction), then one per target forms the outputs.
constexpr int kBwdReduceThreads = 128;
constexpr int kBwdReduceTargets = kBwdReduceThreads / 8;

__global__ void __launch_bounds__(kBwdReduceThreads) backward_reduce_kernel(const BwdArgs a, int32_t BT)
{
    __shared__ double red[kBwdReduceTargets][kNB];
    const int64_t n_tb = (a.n + BT - 1) / BT;
    const int split = choose_split(n_tb, a.n_tiles, a.grid, a.max_split, a.part_cap_rows, BT);
    if (split <= 1) return;
    const int64_t rows = n_tb * BT;
    const int t = threadIdx.x % kBwdReduceTargets, c = threadIdx.x / kBwdReduceTargets;
    const int64_t k = (int64_t)blockIdx.x * kBwdReduceTargets + t;
    if (c < kNB && k < a.n) {
        const double *part = a.part + (int64_t)c * rows + k;
        const int64_t step = (int64_t)kNB * rows;
        double hi = part[0], lo = 0.0;
#pragma unroll 4
        for (int sp = 1; sp < split; ++sp) two_sum_ordered(hi, lo, part[sp * step]);
        red[t][c] = hi + lo;
    }
    __syncthreads();
    if (threadIdx.x < kBwdReduceTargets && k < a.n) {
        double sum[kNB];
#pragma unroll
        for (int q = 0; q < kNB; ++q) sum[q] = red[t][q];
        bwd_write(a, k, sum);
    }
}

// a_bar == NULL: only the potential-energy terms, elementwise.
__global__ void __launch_bounds__(256) backward_pot_only_kernel(const BwdArgs a)
{
    const int64_t k = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (k >= a.n) return;
    double zero[kNB] = {0, 0, 0, 0, 0, 0, 0};
    bwd_write(a, k, zero);
}

// Fixed tile shapes of the adjoint.
constexpr int kBwdNTf = 768, kBwdKTf = 1, kBwdSf = 256, kBwdMinBf = 1, kBwdUf = 4;
constexpr size_t kBwdSmemf = sizeof(BwdPairSmem<kBwdSf>);
// FP64: 256-source tiles, 128 below 2^25 pairs (the forward's line, kFinePairs, is 2^26)
constexpr int kBwdNTd = 128, kBwdSd = 256, kBwdSfine = 128, kBwdMinBd = 4;
constexpr int64_t kBwdFinePairs = 1LL << 25;
constexpr size_t kBwdSmemd = sizeof(BwdDfSmem<kBwdNTd, kBwdSd>);
constexpr size_t kBwdSmemfine = sizeof(BwdDfSmem<kBwdNTd, kBwdSfine>);

struct BwdLayout {
    int64_t n_tiles, geo_off, src_off, lo_off, part_off, total, part_cap_rows;
    int32_t max_split, S, BT;
};

bool bwd_fine(const grav_params *p, int64_t n)
{
    return p->precision == GRAV_F64 && p->max_split != 1 && n * n < kBwdFinePairs;
}

// The smallest (up to half an item, target block x tile, an SM: 1024 elements)
// keep FP64 pair terms: each SM runs one CTA or none, so a call takes as long as
// its slowest item, and a tile that takes both routes, two parts and FP64 sources,
// takes the sum of both (a_bar = -x, FP64 pairs / both / FP64 throughout: 500 elements 207 /
// 251 / 191 us, 1000 223 / 242 / 193; like a_bar 1536 344 / 212 / 298).
bool bwd_few(const grav_params *p, int64_t n)
{
    int sms = 0;
    if (device_sm_count(&sms) != GRAV_OK) return false;
    const int64_t items = ((n + kBwdNTd - 1) / kBwdNTd) * ((n + kBwdSfine - 1) / kBwdSfine);
    return bwd_fine(p, n) && 2 * items <= sms;
}

int bwd_layout(const grav_params *p, int64_t n, BwdLayout *L)
{
    int sms = 0;
    int rc = device_sm_count(&sms);
    if (rc) return rc;
    const bool mixed = p->precision == GRAV_MIXED;
    L->S = mixed ? kBwdSf : bwd_fine(p, n) ? kBwdSfine : kBwdSd;
    L->BT = mixed ? kBwdNTf * kBwdKTf : kBwdNTd;
    const int64_t bytes = mixed ? 32 : kDfBytesPerSource;
    L->max_split = p->max_split > 0 ? p->max_split : kDefaultMaxSplit;
    L->n_tiles = (n + L->S - 1) / L->S;
    L->geo_off = 0;
    L->src_off = round_up(L->n_tiles * (int64_t)sizeof(TileGeom), 256);
    L->lo_off = L->src_off + round_up(L->n_tiles * L->S * bytes, 256);
    L->part_off = L->lo_off + round_up(mixed ? L->n_tiles * kLoPlanes * L->S * 4 : 0, 256);
    const int64_t n_tb = (n + L->BT - 1) / L->BT;
    int64_t blocks = 0;
    if (L->max_split > 1 && L->n_tiles > 1) blocks = std::min<int64_t>(n_tb * L->max_split, 16LL * sms);
    L->part_cap_rows = blocks * L->BT;
    L->total = std::max<int64_t>(256, L->part_off + round_up(L->part_cap_rows * kNB * 8, 256));
    return GRAV_OK;
}

int bwd_grid(bool mixed, bool batched, bool fine, int *grid)
{
    static std::mutex mu;
    static int cache[64][2][3];
    int dev = 0, sms = 0;
    int rc = check_cuda(cudaGetDevice(&dev), "cudaGetDevice");
    if (rc) return rc;
    rc = device_sm_count(&sms);
    if (rc) return rc;
    if (dev >= 64) return fail(GRAV_ECUDA, "device ordinal out of range");
    std::lock_guard<std::mutex> lk(mu);
    int &slot = cache[dev][mixed ? 1 : 0][batched ? 1 : fine ? 2 : 0];
    if (slot == 0) {
        int b = 0;
        cudaError_t e = cudaSuccess;
        if (mixed && !batched) {
            auto k = backward_pair_kernel<kBwdNTf, kBwdKTf, kBwdSf, kBwdMinBf, kBwdUf>;
            e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kBwdSmemf);
            if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k, kBwdNTf, kBwdSmemf);
        } else if (mixed) {
            auto k = backward_pair_batched_kernel<kBwdNTf, kBwdKTf, kBwdSf, kBwdMinBf, kBwdUf>;
            e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kBwdSmemf);
            if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k, kBwdNTf, kBwdSmemf);
        } else {
            auto set = [&](auto k, size_t bytes) {
                e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
                if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k, kBwdNTd, bytes);
            };
            if (batched)
                set(backward_batched_kernel<kBwdNTd, kBwdSd, kBwdMinBd>, kBwdSmemd);
            else if (fine)
                set(backward_kernel<kBwdNTd, kBwdSfine, kBwdMinBd>, kBwdSmemfine);
            else
                set(backward_kernel<kBwdNTd, kBwdSd, kBwdMinBd>, kBwdSmemd);
        }
        rc = check_cuda(e, "cudaOccupancyMaxActiveBlocksPerMultiprocessor");
        if (rc) return rc;
        if (b < 1) return fail(GRAV_ECUDA, "adjoint kernel cannot be resident on an SM");
        slot = b * sms;
    }
    *grid = slot;
    return GRAV_OK;
}

// Workspace of a batched adjoint: the plan's arrays, then the tiles.
struct BwdBatchLayout {
    int64_t hdr, tile_off, idx_lo, idx_hi, ntb, order, item_off, geo, src, lo, total, max_tiles;
};

BwdBatchLayout bwd_batch_layout(bool mixed, int32_t n_sys, int64_t n_total)
{
    BwdBatchLayout L;
    const int64_t S = mixed ? kBwdSf : kBwdSd;
    const int64_t bytes = mixed ? 32 : kDfBytesPerSource;
    L.max_tiles = (n_total + S - 1) / S + n_sys;
    int64_t o = 0;
    L.hdr = o;
    o += kBatchHeaderBytes;
    L.tile_off = o;
    o += round_up(4 * ((int64_t)n_sys + 1), 256);
    L.idx_lo = o;
    o += round_up(4 * (int64_t)n_sys, 256);
    L.idx_hi = o;
    o += round_up(4 * (int64_t)n_sys, 256);
    L.ntb = o;
    o += round_up(4 * (int64_t)n_sys, 256);
    L.order = o;
    o += round_up(4 * (int64_t)n_sys, 256);
    L.item_off = o;
    o += round_up(8 * ((int64_t)n_sys + 1), 256);
    L.geo = o;
    o += round_up(L.max_tiles * (int64_t)sizeof(TileGeom), 256);
    L.src = o;
    o += round_up(L.max_tiles * S * bytes, 256);
    L.lo = o;
    o += round_up(mixed ? L.max_tiles * kLoPlanes * S * 4 : 0, 256);
    L.total = o;
    return L;
}

int check_bwd_params(const grav_params *p, const char *who)
{
    if (!p) return fail(GRAV_EINVAL, "%s: null params", who);
    if (!(p->G > 0.0) || !std::isfinite(p->G)) return fail(GRAV_EINVAL, "%s: G must be finite and > 0", who);
    if (!(p->h > 0.0) || !std::isfinite(p->h)) return fail(GRAV_EINVAL, "%s: h must be finite and > 0", who);
    if (p->precision != GRAV_F64 && p->precision != GRAV_MIXED)
        return fail(GRAV_EINVAL, "%s: precision must be GRAV_F64 or GRAV_MIXED", who);
    if (p->max_split < 0) return fail(GRAV_EINVAL, "%s: max_split < 0", who);
    if (p->box != 0.0) return fail(GRAV_EINVAL, "%s: the adjoint supports open boundaries only", who);
    return GRAV_OK;
}

}  // namespace
}  // namespace grav

using namespace grav;

extern "C" int64_t grav_backward_workspace_bytes(const grav_params *p, int64_t n)
{
    int rc = check_bwd_params(p, "grav_backward_workspace_bytes");
    if (rc) return rc;
    if (n < 0 || n > INT32_MAX) return fail(GRAV_EINVAL, "grav_backward_workspace_bytes: n outside [0, 2^31)");
    BwdLayout L;
    rc = bwd_layout(p, n, &L);
    if (rc) return rc;
    return L.total;
}

extern "C" int grav_eval_backward(const grav_params *p, int64_t n, const double *pos,
                                  const double *mass, const double *a_bar, double w_bar,
                                  const double *acc, const double *tidal, const double *pot,
                                  double *pos_bar, double *mass_bar, int32_t *flags_dev,
                                  void *workspace, int64_t workspace_bytes, void *stream)
{
    static const char *who = "grav_eval_backward";
    int rc = check_bwd_params(p, who);
    if (rc) return rc;
    if (n < 0 || n > INT32_MAX) return fail(GRAV_EINVAL, "%s: n outside [0, 2^31)", who);
    if (!std::isfinite(w_bar)) return fail(GRAV_EINVAL, "%s: w_bar not finite", who);
    if (n == 0) return GRAV_OK;
    if (!pos || !mass || !pos_bar || !mass_bar) return fail(GRAV_EINVAL, "%s: null array", who);
    if (a_bar && !tidal) return fail(GRAV_EINVAL, "%s: a_bar given but tidal is NULL", who);
    if (w_bar != 0.0 && (!acc || !pot)) return fail(GRAV_EINVAL, "%s: w_bar != 0 needs acc and pot", who);
    const bool mixed = p->precision == GRAV_MIXED;
    BwdLayout L;
    rc = bwd_layout(p, n, &L);
    if (rc) return rc;
    if (a_bar) {
        if (!workspace) return fail(GRAV_EINVAL, "%s: null workspace", who);
        if (!aligned(workspace, 256)) return fail(GRAV_EINVAL, "%s: workspace not 256-byte aligned", who);
        if (workspace_bytes < L.total)
            return fail(GRAV_ENOMEM, "%s: workspace of %lld bytes < %lld", who, (long long)workspace_bytes,
                        (long long)L.total);
    }
    int grid = 0;
    const bool fine = bwd_fine(p, n);
    rc = bwd_grid(mixed, false, fine, &grid);
    if (rc) return rc;
    char *ws = static_cast<char *>(workspace);
    BwdArgs a;
    a.n = n;
    a.geo = reinterpret_cast<const TileGeom *>(ws + L.geo_off);
    a.src = ws + L.src_off;
    a.n_tiles = (int32_t)L.n_tiles;
    a.max_split = L.max_split;
    a.grid = grid;
    a.pad0 = 0;
    a.part = reinterpret_cast<double *>(ws + L.part_off);
    a.part_cap_rows = L.part_cap_rows;
    a.pos = pos;
    a.mass = mass;
    a.a_bar = a_bar;
    a.w_bar = w_bar;
    a.acc = acc;
    a.tidal = tidal;
    a.pot = pot;
    a.G = p->G;
    a.h = p->h;
    double h2 = p->h * p->h;
    float h2f = (float)h2;
    if ((double)h2f < h2) h2f = std::nextafter(h2f, INFINITY);
    a.h2f_up = h2f;
    a.hinvf = (float)(1.0 / p->h);
    a.pos_bar = pos_bar;
    a.mass_bar = mass_bar;
    a.flags = flags_dev;
    a.src_lo = mixed ? reinterpret_cast<const float *>(ws + L.lo_off) : nullptr;
    cudaStream_t st = as_stream(stream);
    const unsigned eblocks = (unsigned)((n + 255) / 256);
    if (!a_bar) {
        backward_pot_only_kernel<<<eblocks, 256, 0, st>>>(a);
        return check_launch("grav_eval_backward/pot");
    }
    // Pack (x, a_bar) tiles: the forward packer with a_bar in the velocity
    // slot and no mass.
    if (mixed)
        pack_tiles_kernel<kBwdSf, true, false, true><<<(unsigned)L.n_tiles, kBwdSf, 0, st>>>(
            n, pos, a_bar, nullptr, const_cast<TileGeom *>(a.geo), const_cast<void *>(a.src), flags_dev,
            const_cast<float *>(a.src_lo));
    else if (fine)
        pack_tiles_kernel<kBwdSfine, false, false, false, true><<<(unsigned)L.n_tiles, kBwdSfine, 0, st>>>(
            n, pos, a_bar, nullptr, const_cast<TileGeom *>(a.geo), const_cast<void *>(a.src), flags_dev, nullptr,
            bwd_few(p, n));
    else
        pack_tiles_kernel<kBwdSd, false, false, false, true><<<(unsigned)L.n_tiles, kBwdSd, 0, st>>>(
            n, pos, a_bar, nullptr, const_cast<TileGeom *>(a.geo), const_cast<void *>(a.src), flags_dev);
    rc = check_launch("grav_eval_backward/pack");
    if (rc) return rc;
    if (mixed)
        backward_pair_kernel<kBwdNTf, kBwdKTf, kBwdSf, kBwdMinBf, kBwdUf><<<grid, kBwdNTf, kBwdSmemf, st>>>(a);
    else if (fine)
        backward_kernel<kBwdNTd, kBwdSfine, kBwdMinBd><<<grid, kBwdNTd, kBwdSmemfine, st>>>(a);
    else
        backward_kernel<kBwdNTd, kBwdSd, kBwdMinBd><<<grid, kBwdNTd, kBwdSmemd, st>>>(a);
    rc = check_launch("grav_eval_backward/sum");
    if (rc) return rc;
    const int64_t n_tb = (n + L.BT - 1) / L.BT;
    if (L.part_cap_rows > 0 &&
        choose_split(n_tb, a.n_tiles, grid, a.max_split, a.part_cap_rows, L.BT) > 1) {
        backward_reduce_kernel<<<(unsigned)((n + kBwdReduceTargets - 1) / kBwdReduceTargets),
                                 kBwdReduceThreads, 0, st>>>(a, L.BT);
        rc = check_launch("grav_eval_backward/reduce");
    }
    return rc;
}

extern "C" int64_t grav_backward_batched_workspace_bytes(const grav_params *p, int32_t n_sys,
                                                        int64_t n_total)
{
    static const char *who = "grav_backward_batched_workspace_bytes";
    int rc = check_bwd_params(p, who);
    if (rc) return rc;
    if (n_sys < 0 || n_sys > GRAV_BATCH_MAX_SYSTEMS)
        return fail(GRAV_EINVAL, "%s: n_sys outside [0, %d]", who, GRAV_BATCH_MAX_SYSTEMS);
    if (n_total < 0 || n_total > INT32_MAX) return fail(GRAV_EINVAL, "%s: n_total outside [0, 2^31)", who);
    return bwd_batch_layout(p->precision == GRAV_MIXED, n_sys, n_total).total;
}

extern "C" int grav_eval_backward_batched(const grav_params *p, int32_t n_sys,
                                          const grav_system *systems, int64_t n_total,
                                          const double *pos, const double *mass, const double *a_bar,
                                          double w_bar, const double *acc, const double *tidal,
                                          const double *pot, double *pos_bar, double *mass_bar,
                                          int32_t *flags_dev, void *workspace,
                                          int64_t workspace_bytes, void *stream)
{
    static const char *who = "grav_eval_backward_batched";
    int rc = check_bwd_params(p, who);
    if (rc) return rc;
    if (n_sys < 0 || n_sys > GRAV_BATCH_MAX_SYSTEMS)
        return fail(GRAV_EINVAL, "%s: n_sys outside [0, %d]", who, GRAV_BATCH_MAX_SYSTEMS);
    if (n_total < 0 || n_total > INT32_MAX) return fail(GRAV_EINVAL, "%s: n_total outside [0, 2^31)", who);
    if (!std::isfinite(w_bar)) return fail(GRAV_EINVAL, "%s: w_bar not finite", who);
    if (n_sys == 0 || n_total == 0) return GRAV_OK;
    if (!systems || !pos || !mass || !pos_bar || !mass_bar) return fail(GRAV_EINVAL, "%s: null array", who);
    if (a_bar && !tidal) return fail(GRAV_EINVAL, "%s: a_bar given but tidal is NULL", who);
    if (w_bar != 0.0 && (!acc || !pot)) return fail(GRAV_EINVAL, "%s: w_bar != 0 needs acc and pot", who);
    if (!workspace || !aligned(workspace, 256))
        return fail(GRAV_EINVAL, "%s: workspace missing or not 256-byte aligned", who);
    const bool mixed = p->precision == GRAV_MIXED;
    const BwdBatchLayout L = bwd_batch_layout(mixed, n_sys, n_total);
    if (workspace_bytes < L.total)
        return fail(GRAV_ENOMEM, "%s: workspace of %lld bytes < %lld", who, (long long)workspace_bytes,
                    (long long)L.total);
    int grid = 0;
    rc = bwd_grid(mixed, true, false, &grid);
    if (rc) return rc;
    char *ws = static_cast<char *>(workspace);
    BatchView b;
    b.hdr = reinterpret_cast<BatchHeader *>(ws + L.hdr);
    b.sys = systems;
    b.tile_off = reinterpret_cast<int32_t *>(ws + L.tile_off);
    b.idx_lo = reinterpret_cast<int32_t *>(ws + L.idx_lo);
    b.idx_hi = reinterpret_cast<int32_t *>(ws + L.idx_hi);
    b.ntb = reinterpret_cast<int32_t *>(ws + L.ntb);
    b.order = reinterpret_cast<int32_t *>(ws + L.order);
    b.item_off = reinterpret_cast<int64_t *>(ws + L.item_off);
    b.n_sys = n_sys;
    rc = batch_queues(&b.n_queues);
    if (rc) return rc;

    BwdArgs a;
    a.n = n_total;
    a.geo = reinterpret_cast<const TileGeom *>(ws + L.geo);
    a.src = ws + L.src;
    a.n_tiles = 0;
    a.max_split = 1;
    a.grid = grid;
    a.pad0 = 0;
    a.part = nullptr;
    a.part_cap_rows = 0;
    a.pos = pos;
    a.mass = mass;
    a.a_bar = a_bar;
    a.w_bar = w_bar;
    a.acc = acc;
    a.tidal = tidal;
    a.pot = pot;
    a.G = p->G;
    a.h = p->h;
    double h2 = p->h * p->h;
    float h2f = (float)h2;
    if ((double)h2f < h2) h2f = std::nextafter(h2f, INFINITY);
    a.h2f_up = h2f;
    a.hinvf = (float)(1.0 / p->h);
    a.pos_bar = pos_bar;
    a.mass_bar = mass_bar;
    a.flags = flags_dev;
    a.src_lo = mixed ? reinterpret_cast<const float *>(ws + L.lo) : nullptr;
    cudaStream_t st = as_stream(stream);
    if (!a_bar) {
        // only the potential-energy terms, elementwise (no system structure)
        backward_pot_only_kernel<<<(unsigned)((n_total + 255) / 256), 256, 0, st>>>(a);
        return check_launch("grav_eval_backward_batched/pot");
    }
    const int32_t S = mixed ? kBwdSf : kBwdSd;
    const int32_t BT = mixed ? kBwdNTf * kBwdKTf : kBwdNTd;
    // every element a target: the plan takes each system's element range
    rc = launch_batch_plan(b, nullptr, nullptr, n_total, n_total, S, BT, 0.0, flags_dev, st);
    if (rc) return rc;
    // (x, a_bar) tiles: the forward's batched packer with a_bar in the
    // velocity slot and no mass
    if (mixed)
        pack_tiles_batched_kernel<kBwdSf, true, false, true><<<(unsigned)L.max_tiles, kBwdSf, 0, st>>>(
            b, pos, a_bar, nullptr, const_cast<TileGeom *>(a.geo), const_cast<void *>(a.src), flags_dev,
            const_cast<float *>(a.src_lo));
    else
        pack_tiles_batched_kernel<kBwdSd, false, false, false, true><<<(unsigned)L.max_tiles, kBwdSd, 0, st>>>(
            b, pos, a_bar, nullptr, const_cast<TileGeom *>(a.geo), const_cast<void *>(a.src), flags_dev,
            nullptr);
    rc = check_launch("grav_eval_backward_batched/pack");
    if (rc) return rc;
    if (mixed)
        backward_pair_batched_kernel<kBwdNTf, kBwdKTf, kBwdSf, kBwdMinBf, kBwdUf>
            <<<grid, kBwdNTf, kBwdSmemf, st>>>(a, b);
    else
        backward_batched_kernel<kBwdNTd, kBwdSd, kBwdMinBd><<<grid, kBwdNTd, kBwdSmemd, st>>>(a, b);
    return check_launch("grav_eval_backward_batched/sum");
}
