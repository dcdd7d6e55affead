// teuk_pair_tile.cuh -- the FP32 step kernels for 128 < Ntheta <= 256 (a
// multiple of 4): one to three full time steps per launch on packed pairs.
//
// split_tile's form for these rows held eight elements a lane in scalar
// registers: 207 to 222 registers, one CTA of eight warps per SM, 31 % issue,
// bound by instruction latency.  Here the tile's state lies in shared memory
// as pairs (theta j, theta 128 + j), so that the implicit stage (pair_core)
// and the Lax-Wendroff stages both run on packed FP32 registers, two points
// per instruction, without packing or unpacking in between.  An element of a
// tile row is (x lo, x hi, y lo, y hi), 16 bytes; theta 4 g + k of lane g lies
// at position 32 k + g, so a warp's accesses are contiguous in both stages.
// The rows arrive in their own layout by bulk copies, are turned into pairs in
// place by the first implicit stage (a warp reads its whole row before it
// writes), and the last Lax-Wendroff stage writes the output rows straight to
// global memory.  With eight warps per SM the latency of a row solve's chain
// and of its pivot loads still bounds the stage (3.3k of the 13k cycles a
// 36-row step takes it are issue).  The same layout with two r* rows as the
// pair was slower than split_tile's scalar form for Ntheta <= 128 (27.5
// against 25.3 us a step on 16384 x 128): there the scalar form needs half
// the registers and has twice the warps.
#pragma once

#include "teuk_dev.cuh"

namespace teuk {

// Fields of the Lax-Wendroff table, pairs of (lo, hi) step-table values; per
// block those of its node rows, then those of the half nodes above them.
constexpr int kLwFields = 10, kSrcFields = 3;

struct PairSmem {
    unsigned phi, pi, tha, thb, thc, rowi, rowl, rows, total;
};
__host__ __device__ inline PairSmem pair_smem_plan(int R, int N)
{
    (void)N;
    const unsigned nb = (unsigned)R, np = 128u;
    PairSmem s;
    s.phi = 0;
    s.pi = s.phi + nb * np * 16u;
    s.tha = s.pi + nb * np * 16u;              // (AM, AP) pairs per position
    s.thb = s.tha + np * 16u;           // (A0, sin^2)
    s.thc = s.thb + np * 16u;           // cos
    s.rowi = smem_align16(s.thc + np * 8u);
    s.rowl = s.rowi + nb * 64u;                // implicit row constants
    s.rows = s.rowl + nb * 2u * kLwFields * 8u;
    s.total = smem_align16(s.rows + nb * 2u * kSrcFields * 8u);
    return s;
}

namespace {

__device__ __forceinline__ f2x p_sub(f2x a, f2x b)
{
    f2x d;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

// lw_coef on a pair: beta = c_p b, kap = c_p K and 1/Sigma^2 from the fields
// R2, AD, RB, E2, E3, RCTR, CSE, RCTC, RCTI, CSI.
struct LwPair {
    f2x beta, kx, ky, sg;
};
__device__ __forceinline__ LwPair lw_pair_coef(const ulonglong2 *f, f2x nS2, f2x C)
{
    const ulonglong2 f0 = f[0], f1 = f[1], f2 = f[2], f3 = f[3], f4 = f[4];
    const f2x sig = p_fma(f0.y, nS2, f0.x);
    const f2x rs = pk2(rsq_(p_lo(sig)), rsq_(p_hi(sig)));
    LwPair o;
    o.sg = p_mul(rs, rs);
    o.beta = p_mul(rs, f1.x);
    const f2x kx = p_fma(o.sg, p_fma(f2.x, nS2, f1.y), p_fma(rs, f2.y, f3.x));
    const f2x ky = p_fma(rs, p_fma(f3.y, C, f4.x), f4.y);
    o.kx = p_mul(o.sg, kx);
    o.ky = p_mul(o.sg, ky);
    return o;
}
__device__ __forceinline__ int lw_pair_field(int q)
{
    constexpr int f[kLwFields] = {SF_R2, SF_AD, SF_RB, SF_E2, SF_E3, SF_RCTR, SF_CSE, SF_RCTC, SF_RCTI, SF_CSI};
    int r = f[0];
#pragma unroll
    for (int k = 1; k < kLwFields; ++k)
        if (q == k) r = f[k];
    return r;
}

// The work of one CTA, as split_tile's for full steps of a context (no first
// step, no state output, no caller buffers).  OWN (one step): the tile samples
// its step.
template <int KS, bool OWN = false>
__device__ __forceinline__ void pair_tile(const StepParams<float> &p, int i0, int ntiles)
{
    constexpr int kMaxChunks = 8;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ double2 sph[2 * KS];
    __shared__ __align__(8) unsigned long long s_mbar[kMaxChunks];
    __shared__ int s_plan[kMaxTileRows + 8];
    const int Nr = p.Nr, N = p.Nth, TR = p.tile_rows, R = TR + 2 * KS;
    constexpr int NP = 128, NL = 32;                 // pairs of a row, lanes
    const int tid = threadIdx.x, NT = blockDim.x, lane = tid & 31;
    const int g0 = i0 - KS;
    const PairSmem L = pair_smem_plan(R, N);
    unsigned char *sPhi = smem_raw + L.phi, *sPi = smem_raw + L.pi;
    constexpr unsigned bb = NP * 16u;                // bytes of a row of pairs
    ulonglong2 *thA = (ulonglong2 *)(smem_raw + L.tha), *thB = (ulonglong2 *)(smem_raw + L.thb);
    f2x *thC = (f2x *)(smem_raw + L.thc);
    f2x *rowI = (f2x *)(smem_raw + L.rowi), *rowL = (f2x *)(smem_raw + L.rowl), *rowS = (f2x *)(smem_raw + L.rows);
    const ImpConst<float> &K = p.full;
    const bool src = p.patch_np > 0 && i0 + TR + KS - 1 >= p.patch_p0 && g0 <= p.patch_p0 + p.patch_np;
    const long long n_in = *((volatile long long *)&p.ctl->step);

    // ---- load: tile rows 0 .. R - 1 that lie on the grid, in chunks of whole
    // implicit passes, one mbarrier each (each warp issues its chunk's copies)
    const int warp = tid >> 5, nwarp = NT >> 5;
    int cr = nwarp;
    while (udiv(R + cr - 1, cr) > kMaxChunks) cr += nwarp;
    const int nch = udiv(R + cr - 1, cr);
    const unsigned rb8 = (unsigned)N * 8u;           // bytes of a row
    for (int c = warp; c < nch; c += nwarp) {
        if (lane != 0) break;
        int r0 = c * cr, r1 = r0 + cr < R ? r0 + cr : R;
        if (g0 + r0 < 0) r0 = -g0;
        if (g0 + r1 > Nr) r1 = Nr - g0;
        const unsigned rows = r1 > r0 ? (unsigned)(r1 - r0) : 0u;
        mbar_init(&s_mbar[c], 1);
        mbar_expect_tx(&s_mbar[c], 2u * rb8 * rows);
        if (!rows) continue;
        const float2 *f = p.uin + (size_t)(g0 + r0) * N, *g = f + (size_t)Nr * N;
        if (rb8 == bb) {
            bulk_g2s(sPhi + r0 * bb, f, rows * bb, &s_mbar[c]);
            bulk_g2s(sPi + r0 * bb, g, rows * bb, &s_mbar[c]);
        } else {
            for (unsigned r = 0; r < rows; ++r) {
                bulk_g2s(sPhi + (r0 + r) * bb, f + (size_t)r * N, rb8, &s_mbar[c]);
                bulk_g2s(sPi + (r0 + r) * bb, g + (size_t)r * N, rb8, &s_mbar[c]);
            }
        }
        // the chunk's pivot rows, which the row solves read from global memory
        prefetch_l2(K.piv + (size_t)(g0 + r0) * N, rows * rb8);
    }
    // ---- tables: theta, implicit rows (a valid interior row's constants for
    // the others), Lax-Wendroff and source rows
    auto th_pair = [&](int f, int pos) {
        const int j = 4 * (pos % NL) + pos / NL;
        const float lo = p.thtab[f * N + j];
        return pk2(lo, j + 128 < N ? p.thtab[f * N + j + 128] : 0.0f);
    };
    for (int pos = tid; pos < NP; pos += NT) {
        thA[pos] = make_ulonglong2(th_pair(TF_AM, pos), th_pair(TF_AP, pos));
        thB[pos] = make_ulonglong2(th_pair(TF_A0, pos), th_pair(TF_S2, pos));
        thC[pos] = th_pair(TF_C, pos);
    }
    auto clampi = [](int x, int lo, int hi) { return x < lo ? lo : (x > hi ? hi : x); };
    for (int idx = tid; idx < R * 8; idx += NT) {
        const int m = idx >> 3, q = idx & 7;
        rowI[idx] = p_dup(p.stab[(size_t)(2 * clampi(g0 + m, 1, Nr - 2)) * NSF + q]);
    }
    // a warp per tile row, a lane per field and position
    if (lane < 2 * kLwFields) {
        const int half = lane >= kLwFields ? 1 : 0, f = lw_pair_field(lane - half * kLwFields);
#pragma unroll 4
        for (int e = warp; e < R; e += nwarp) {
            const int ra = clampi(g0 + e, 0, Nr - 1 - half);
            rowL[e * 2 * kLwFields + lane] = p_dup(p.stab[(size_t)(2 * ra + half) * NSF + f]);
        }
    } else if (src && lane < 2 * kLwFields + 2 * kSrcFields) {
        const int r = lane - 2 * kLwFields, half = r >= kSrcFields ? 1 : 0, f = SF_SRE + r - half * kSrcFields;
        for (int e = warp; e < R; e += nwarp) {
            const int ra = clampi(g0 + e, 0, Nr - 1 - half);
            rowS[e * 2 * kSrcFields + r] = p_dup(p.stab[(size_t)(2 * ra + half) * NSF + f]);
        }
    }
    for (int lr = tid; lr < R; lr += NT) s_plan[lr] = g0 + lr >= 0 && g0 + lr < Nr ? K.plan[g0 + lr] : 0;
    __syncthreads();
    if (tid == 0) {
        // the last CTA to have read the step index advances it (as in split_tile)
        __threadfence();
        unsigned t = atomicAdd(&p.ctl->ticket, 1u);
        if (t == (unsigned)ntiles - 1u) {
            p.ctl->ticket = 0u;
            p.ctl->step = n_in + KS;
        }
    }
    const bool sampler = tid >= NT - 32;
    if (src && sampler && lane < 2 * KS) {
        const double t = (double)(n_in + (lane >> 1)) * p.dt64, len = (lane & 1) ? p.dt64 : 0.5 * p.dt64;
        const double2 e = phase_at(p.mOmega, (lane & 1) ? t + 0.5 * p.dt64 : t);
        sph[lane] = make_double2(len * e.x, len * e.y);
    }
    // ---- extraction row, left for the sampling launch (see split_tile)
    const bool ext = p.i_ext >= i0 && p.i_ext < i0 + TR && p.i_ext < Nr;
    const int lx = p.i_ext - g0;
    auto raw_row = [&](long long n) { return p.raw + (size_t)(n % kRawSlots) * 2 * N; };

    const int g = lane;
    const bool inB = 128 + 4 * g < N;                // the lane's high elements exist (whole segments)
    const int wait_lim = p.wait0 >= 0 ? p.wait0 : kWaitLimit;
    const float2 zero2 = make_float2(0.0f, 0.0f), one2 = make_float2(1.0f, 0.0f);
    int ok = 1;
    // rows off the grid and boundary rows exist only in the first and last tiles
    const bool interior = g0 >= 1 && g0 + R <= Nr - 1;
    auto inner = [&](int lr) { return g0 + lr >= 1 && g0 + lr <= Nr - 2; };

#pragma unroll 1
    for (int step = 0; step < KS; ++step) {
        // ---- implicit stage: a warp per row
#pragma unroll 1
        for (int m = warp + step; m < R - step; m += nwarp) {
            if (step == 0 && ok) ok &= (int)mbar_wait(&s_mbar[udiv(m, cr)], 0, wait_lim);
            const bool act = inner(m);
            const size_t gr = act ? (size_t)(g0 + m) : 1;
            const int jA = 4 * g, jB = jA + 128;
            PairCoef C;
            PC w[4], y[4];
            float2 ra[4], rb[4];
            auto ld4 = [](const float2 *s, bool in, float2 pad, float2(&r)[4]) {
                if (in) vload<4>(r, s);
                else
#pragma unroll
                    for (int k = 0; k < 4; ++k) r[k] = pad;
            };
            vload<4>(ra, K.piv + gr * N + jA);
            ld4(K.piv + gr * N + jB, inB, one2, rb);
            C.plan = act ? s_plan[m] : 0;
            C.Af.x = C.Af.y = C.Ab.x = C.Ab.y = 0ull;
            if (C.plan) {
                const float4 *sp = reinterpret_cast<const float4 *>(K.seg + (gr * 32 + g) * 4);
                const float4 sa = sp[0], sb = sp[1];
                C.Af = pc_pack(make_float2(sa.x, sa.y), make_float2(sb.x, sb.y));
                C.Ab = pc_pack(make_float2(sa.z, sa.w), make_float2(sb.z, sb.w));
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                C.ex[k] = pk2(ra[k].x, rb[k].x);
                C.ey[k] = pk2(ra[k].y, rb[k].y);
            }
            unsigned char *bf = sPhi + m * bb, *bg = sPi + m * bb;
            if (step == 0) {
                // the row as it was copied; boundary and off-grid rows are zero
                ld4((const float2 *)bf + jA, act, zero2, ra);
                ld4((const float2 *)bf + jB, inB && act, zero2, rb);
#pragma unroll
                for (int k = 0; k < 4; ++k) w[k] = pc_pack(ra[k], rb[k]);
                ld4((const float2 *)bg + jA, act, zero2, ra);
                ld4((const float2 *)bg + jB, inB && act, zero2, rb);
#pragma unroll
                for (int k = 0; k < 4; ++k) y[k] = pc_pack(ra[k], rb[k]);
            } else {
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const ulonglong2 a = ((const ulonglong2 *)bf)[k * NL + g], b = ((const ulonglong2 *)bg)[k * NL + g];
                    w[k].x = a.x;
                    w[k].y = a.y;
                    y[k].x = b.x;
                    y[k].y = b.y;
                }
            }
            const ulonglong2 *ri = (const ulonglong2 *)(rowI + m * 8);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const ulonglong2 v = ri[q];
                C.row[2 * q] = v.x;
                C.row[2 * q + 1] = v.y;
            }
            ulonglong2 ta[4], tb[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                ta[k] = thA[k * NL + g];
                tb[k] = thB[k * NL + g];
            }
            pair_core(
                K, C, w, y, g,
                [&](int k, int q) {
                    return q == 0 ? tb[k].y : (q == 1 ? thC[k * NL + g] : (q == 2 ? ta[k].x : (q == 3 ? tb[k].x : ta[k].y)));
                },
                [](const PC(&)[4], const PC(&)[4]) {});
            __syncwarp();
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                ((ulonglong2 *)bf)[k * NL + g] = make_ulonglong2(w[k].x, w[k].y);
                ((ulonglong2 *)bg)[k * NL + g] = make_ulonglong2(y[k].x, y[k].y);
            }
        }
        if (step == 0) {
            // all threads agree on the outcome of the bounded waits before acting on it
            // (every row of the tile has been waited for by its warp)
            if (!__syncthreads_and(ok)) {
                if (tid == 0) {
                    atomicOr(&p.ctl->flags, FLAG_TIMEOUT);
                    for (int c = 0; c < nch; ++c) mbar_wait(&s_mbar[c], 0, kWaitLimit);
                }
                return;
            }
        } else {
            __syncthreads();
        }
        // ---- Lax-Wendroff stages: thread (segment, position) marches over
        // blocks [ra, rb) of its position
        const int r0 = step + 1, cnt = R - 2 - 2 * step;
        const int nseg = udiv(NT, NP), sl = udiv(cnt + nseg - 1, nseg);
        const int sgm = udiv(tid, NP), pos = tid - sgm * NP;
        const int ra = r0 + sgm * sl, rb = ra + sl < r0 + cnt ? ra + sl : r0 + cnt;
        const bool work = sgm < nseg && ra < rb;
        auto el = [&](const unsigned char *s, int m) {
            const ulonglong2 v = *(const ulonglong2 *)(s + m * bb + pos * 16);
            PC r;
            r.x = v.x;
            r.y = v.y;
            return r;
        };
        // the values on either side of the segment, before its neighbours overwrite them
        PC pf, pg, nf, ng;
        pf.x = pf.y = pg.x = pg.y = nf.x = nf.y = ng.x = ng.y = 0ull;
        if (work) {
            pf = el(sPhi, ra - 1);
            pg = el(sPi, ra - 1);
            nf = el(sPhi, rb);
            ng = el(sPi, rb);
        }
        __syncthreads();
        const bool last = step == KS - 1;
        const int jt = 4 * (pos % NL) + pos / NL;
        const f2x nS2 = p_neg(thB[work ? pos : 0].y), Cc = thC[work ? pos : 0], half = p_dup(0.5f);
        f2x gth = 0ull, ga2 = 0ull;
        float2 ph1 = zero2, ph2 = zero2;
        if (src) {
            ph1 = from_d2<float>(sph[2 * step]);
            ph2 = from_d2<float>(sph[2 * step + 1]);
            const int jb = jt + 128 < N ? jt + 128 : jt;
            gth = pk2(p.thtab[TF_GTH * N + jt], p.thtab[TF_GTH * N + jb]);
            ga2 = pk2(p.thtab[TF_GA2 * N + jt], p.thtab[TF_GA2 * N + jb]);
        }
        auto march = [&](auto general) {
            constexpr bool GEN = decltype(general)::value;   // source terms and boundary rows
            auto table = [&](int m, int hf) { return (const ulonglong2 *)(rowL + (m * 2 + hf) * kLwFields); };
            auto add_source = [&](PC t, int m, int hf, f2x sg, float2 ph) {
                const f2x *f = rowS + (m * 2 + hf) * kSrcFields;
                const f2x s = p_mul(sg, p_fma(f[2], gth, ga2));
                const f2x Fx = p_mul(s, f[0]), Fy = p_mul(s, f[1]);
                const f2x px = p_dup(ph.x), py = p_dup(ph.y);
                t.x = p_add(t.x, p_fma(Fx, px, p_mul(Fy, p_neg(py))));
                t.y = p_add(t.y, p_fma(Fx, py, p_mul(Fy, px)));
                return t;
            };
            auto mid1 = [&](f2x a, f2x b) { return p_mul(half, p_add(a, b)); };
            auto midpoint = [&](int m, const LwPair &c, PC fa, PC ga, PC fb, PC gb, PC &mf, PC &mg) {
                const f2x nbeta = p_neg(c.beta), nky = p_neg(c.ky);
                const f2x dx = p_sub(fb.x, fa.x), dy = p_sub(fb.y, fa.y);
                mf.x = p_fma(nbeta, dx, mid1(fa.x, fb.x));
                mf.y = p_fma(nbeta, dy, mid1(fa.y, fb.y));
                PC t;
                t.x = p_fma(c.beta, p_sub(gb.x, ga.x), mid1(ga.x, gb.x));
                t.y = p_fma(c.beta, p_sub(gb.y, ga.y), mid1(ga.y, gb.y));
                if (GEN && src) t = add_source(t, m, 1, c.sg, ph1);
                mg.x = p_fma(c.kx, dx, p_fma(nky, dy, t.x));
                mg.y = p_fma(c.kx, dy, p_fma(c.ky, dx, t.y));
            };
            PC fb = el(sPhi, ra), gb = el(sPi, ra), fc = nf, gc = ng;
            if (ra + 1 < rb) {
                fc = el(sPhi, ra + 1);
                gc = el(sPi, ra + 1);
            }
            PC mfp, mgp;
            midpoint(ra - 1, lw_pair_coef(table(ra - 1, 1), nS2, Cc), pf, pg, fb, gb, mfp, mgp);
            LwPair cn = lw_pair_coef(table(ra, 0), nS2, Cc), ch = lw_pair_coef(table(ra, 1), nS2, Cc);
            float2 *oA = p.uout + (long long)(g0 + ra) * N + jt;
            const long long pl = (long long)Nr * N;
#pragma unroll 2
            for (int m = ra; m < rb; ++m) {
                // the next block's state and coefficients are on their way while
                // this one is updated (a store ends the reach of later loads)
                PC fd = nf, gd = ng;
                if (m + 2 < rb) {
                    fd = el(sPhi, m + 2);
                    gd = el(sPi, m + 2);
                }
                const LwPair cn2 = lw_pair_coef(table(m + 1, 0), nS2, Cc), ch2 = lw_pair_coef(table(m + 1, 1), nS2, Cc);
                PC mf, mg;
                midpoint(m, ch, fb, gb, fc, gc, mf, mg);
                const f2x dx = p_sub(mf.x, mfp.x), dy = p_sub(mf.y, mfp.y);
                const f2x nbeta = p_neg(cn.beta), nky = p_neg(cn.ky);
                PC a, b, t;
                a.x = p_fma(nbeta, dx, fb.x);
                a.y = p_fma(nbeta, dy, fb.y);
                t.x = p_fma(cn.beta, p_sub(mg.x, mgp.x), gb.x);
                t.y = p_fma(cn.beta, p_sub(mg.y, mgp.y), gb.y);
                if (GEN && src) t = add_source(t, m, 0, cn.sg, ph2);
                b.x = p_fma(cn.kx, dx, p_fma(nky, dy, t.x));
                b.y = p_fma(cn.kx, dy, p_fma(cn.ky, dx, t.y));
                if (GEN && !interior) {
                    const f2x keep = inner(m) ? ~0ull : 0ull;
                    a.x &= keep;
                    a.y &= keep;
                    b.x &= keep;
                    b.y &= keep;
                }
                if (last) {
                    if (m >= KS && m < KS + TR && g0 + m < Nr) {
                        oA[0] = make_float2(p_lo(a.x), p_lo(a.y));
                        oA[pl] = make_float2(p_lo(b.x), p_lo(b.y));
                        if (jt + 128 < N) {
                            oA[128] = make_float2(p_hi(a.x), p_hi(a.y));
                            oA[pl + 128] = make_float2(p_hi(b.x), p_hi(b.y));
                        }
                    }
                    oA += N;
                    if (ext && m == lx) {
                        float2 *dst = raw_row(n_in + KS);
                        dst[jt] = make_float2(p_lo(a.x), p_lo(a.y));
                        dst[N + jt] = make_float2(p_lo(b.x), p_lo(b.y));
                        if (jt + 128 < N) {
                            dst[jt + 128] = make_float2(p_hi(a.x), p_hi(a.y));
                            dst[N + jt + 128] = make_float2(p_hi(b.x), p_hi(b.y));
                        }
                    }
                } else {
                    *(ulonglong2 *)(sPhi + m * bb + pos * 16) = make_ulonglong2(a.x, a.y);
                    *(ulonglong2 *)(sPi + m * bb + pos * 16) = make_ulonglong2(b.x, b.y);
                }
                fb = fc;
                gb = gc;
                fc = fd;
                gc = gd;
                mfp = mf;
                mgp = mg;
                cn = cn2;
                ch = ch2;
            }
        };
        if (work) {
            if (interior && !src)
                march(std::false_type{});
            else
                march(std::true_type{});
        }
        if (!last) {
            __syncthreads();
            if (ext) {
                float2 *dst = raw_row(n_in + step + 1);
                for (int j = tid; j < N; j += NT) {
                    const int jj = j & 127, ps = (jj & 3) * NL + (jj >> 2);
                    const bool hi = j >= 128;
                    const float4 a = *(const float4 *)(sPhi + lx * bb + ps * 16), b = *(const float4 *)(sPi + lx * bb + ps * 16);
                    dst[j] = hi ? make_float2(a.y, a.w) : make_float2(a.x, a.z);
                    dst[N + j] = hi ? make_float2(b.y, b.w) : make_float2(b.x, b.z);
                }
                __syncthreads();   // the next implicit stage works in place
            }
        }
    }
    if constexpr (OWN) {
        static_assert(KS == 1, "the sample of the launch's last step");
        if (!ext) return;
        __syncthreads();   // the row is in p.raw, the tile's shared memory is free
        if (warp == 0) {
            float2 *rf = (float2 *)sPhi, *rg = (float2 *)sPi;
            const float2 *src_row = raw_row(n_in + 1);
            for (int j = lane; j < N; j += 32) {
                rf[j] = src_row[j];
                rg[j] = src_row[N + j];
            }
            __syncwarp();
            const bool active = p.i_ext >= 1 && p.i_ext <= Nr - 2;
            implicit_row_one<float, kSeg>(p.half, rf, rg, p.i_ext, p.stab + (size_t)(2 * p.i_ext) * NSF, nullptr, p.th2, N,
                                          active, true, lane, 32, p.vec != 0, p.half.plan[p.i_ext]);
            __syncwarp();
            extract_warp<float>(p, rf, n_in + 1);
            if (lane == 0) p.ctl->sampled = n_in + 1;
        }
    }
}

template <int KS, bool OWN = false>
__global__ void __launch_bounds__(256, 1) k_pair_step(const StepParams<float> p)
{
    launch_turn();
    pair_tile<KS, OWN>(p, (int)blockIdx.x * p.tile_rows, (int)gridDim.x);
}

// Batched form, as k_split_batch: entry blockIdx.x of the tile list.
template <int KS>
__global__ void __launch_bounds__(256, 1) k_pair_batch(const StepParams<float> *params, const int2 *tiles)
{
    __shared__ __align__(16) StepParams<float> sp;
    const int2 e = tiles[blockIdx.x];
    batch_params(sp, params, e);
    launch_turn();
    pair_tile<KS>(sp, e.y, sp.ntiles);
}

}  // namespace
}  // namespace teuk
