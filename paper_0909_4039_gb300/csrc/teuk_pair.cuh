// teuk_pair.cuh -- the FP32 implicit row solve for 128 < Ntheta <= 256.
//
// One warp solves one theta row.  A lane holds elements [4 g, 4 g + 4) of the
// row's two halves [0, 128) and [128, Ntheta) in the two halves of packed
// FP32 registers (add/mul/fma .f32x2 of the sm_100 family), so one
// instruction serves both, complex products included (real and imaginary
// parts are separate registers), and the two LU recurrences of a lane hide
// each other's latency; the halves join at lane 31 / lane 0 of the scans.
#pragma once

namespace teuk {
namespace {

typedef unsigned long long f2x;   // packed pair (lo, hi) of FP32 values

__device__ __forceinline__ f2x p_add(f2x a, f2x b)
{
    f2x d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f2x p_mul(f2x a, f2x b)
{
    f2x d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f2x p_fma(f2x a, f2x b, f2x c)
{
    f2x d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ f2x p_dup(float x) { return pk2(x, x); }
__device__ __forceinline__ float p_lo(f2x a) { return upk2(a).x; }
__device__ __forceinline__ float p_hi(f2x a) { return upk2(a).y; }
__device__ __forceinline__ f2x p_neg(f2x a) { return a ^ 0x8000000080000000ull; }

// A pair of complex values.
struct PC {
    f2x x, y;
};
__device__ __forceinline__ PC pc_pack(float2 a, float2 b)
{
    PC r;
    r.x = pk2(a.x, b.x);
    r.y = pk2(a.y, b.y);
    return r;
}
__device__ __forceinline__ PC pc_axpy(f2x s, PC a, PC b)   // b + s a, as caxpy
{
    PC r;
    r.x = p_fma(s, a.x, b.x);
    r.y = p_fma(s, a.y, b.y);
    return r;
}
// a b with (ax, ay, nay = -ay), as cmul(a, b)
__device__ __forceinline__ PC pc_mul(f2x ax, f2x ay, f2x nay, PC b)
{
    PC r;
    r.x = p_fma(ax, b.x, p_mul(nay, b.y));
    r.y = p_fma(ax, b.y, p_mul(ay, b.x));
    return r;
}
// c + a b, as cfma(a, b, c); with a = -f given as (-fx, -fy, fy) it is cfnma(f, b, c)
__device__ __forceinline__ PC pc_fma(f2x ax, f2x ay, f2x nay, PC b, PC c)
{
    PC r;
    r.x = p_fma(ax, b.x, p_fma(nay, b.y, c.x));
    r.y = p_fma(ax, b.y, p_fma(ay, b.x, c.y));
    return r;
}

// The value d segments below / above, over the 64 segments lo[0..31],
// hi[0..31] of the row.  Past the ends the result is some other value of the
// row, which meets a zero factor.
__device__ __forceinline__ f2x p_up(f2x v, int d)
{
    const int lane = threadIdx.x & 31;
    const float lo = __shfl_sync(0xffffffffu, p_lo(v), lane - d), hi = __shfl_sync(0xffffffffu, p_hi(v), lane - d);
    return pk2(lo, lane < d ? lo : hi);
}
__device__ __forceinline__ f2x p_down(f2x v, int d)
{
    const int lane = threadIdx.x & 31;
    const float lo = __shfl_sync(0xffffffffu, p_lo(v), lane + d), hi = __shfl_sync(0xffffffffu, p_hi(v), lane + d);
    return pk2(lane + d >= 32 ? hi : lo, hi);
}
__device__ __forceinline__ PC pc_up(PC v, int d)
{
    v.x = p_up(v.x, d);
    v.y = p_up(v.y, d);
    return v;
}
__device__ __forceinline__ PC pc_down(PC v, int d)
{
    v.x = p_down(v.x, d);
    v.y = p_down(v.y, d);
    return v;
}

// What a lane's part of the row needs besides the state: the pivots, the
// segments' multiplier products (ImpConst::seg; read where a level is used),
// the scan levels (forward | backward << 8) and the row
// constants (the implicit block of the step table).
struct PairCoef {
    f2x ex[4], ey[4];
    PC Af, Ab;
    int plan;
    f2x row[8];
};

// One implicit SDIRK2 step of length h (constants K) on a row: the map of
// implicit_row_fwd, lane g holding theta elements [4 g, 4 g + 4).  On entry
// (w, y) = (Phi, Pi), on exit the result.  th(k, q): the paired theta table at
// element k (q: 0 sin^2, 1 cos, 2 AM, 3 A0, 4 AP; zero past the row's end, so
// that padding elements, which hold zero data and unit pivots, have no
// coupling).  u1(w, y) receives the first stage value.  Every lane of the
// warp calls it.
template <typename Th, typename U1>
__device__ __forceinline__ void pair_core(const ImpConst<float> &K, const PairCoef &C, PC (&w)[4], PC (&y)[4], int g, Th th,
                                          U1 u1)
{
    const int nf = C.plan & 0xff, nb = (C.plan >> 8) & 0xff;

    // ---- coefficients (imp_row, imp_elem)
    f2x ney[4], sg[4], qam[4], qap[4], nsub[4], dx[4], dy[4], ndy[4], nfx[4], fy[4], nfy[4];
    {
        const f2x nAD = p_neg(C.row[SF_AD]), nc0r = p_neg(C.row[SF_C0R]), ngh2 = p_dup(-K.gh2);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const f2x s = p_fma(nAD, th(k, 0), C.row[SF_R2]);
            sg[k] = pk2(rcp_fast(p_lo(s)), rcp_fast(p_hi(s)));
            const f2x q = p_mul(C.row[SF_DELTA], sg[k]);
            qam[k] = p_mul(q, th(k, 2));
            qap[k] = p_mul(q, th(k, 4));
            dx[k] = p_fma(q, th(k, 3), p_mul(sg[k], nc0r));
            ndy[k] = p_mul(sg[k], C.row[SF_C0I]);
            dy[k] = p_neg(ndy[k]);
            nsub[k] = p_mul(ngh2, qam[k]);
            const f2x nsup = p_mul(ngh2, qap[k]);
            nfx[k] = p_mul(nsup, C.ex[k]);
            nfy[k] = p_mul(nsup, C.ey[k]);
            fy[k] = p_neg(nfy[k]);
            ney[k] = p_neg(C.ey[k]);
        }
    }
    // out = W x (apply_W)
    auto apply = [&](const PC(&x)[4], PC(&out)[4]) {
        const PC xl = pc_up(x[3], 1), xr = pc_down(x[0], 1);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const PC xm = k ? x[k ? k - 1 : 0] : xl, xp = k < 3 ? x[k < 3 ? k + 1 : 3] : xr;
            PC t;
            t.x = p_fma(qap[k], xp.x, p_mul(qam[k], xm.x));
            t.y = p_fma(qap[k], xp.y, p_mul(qam[k], xm.y));
            out[k] = pc_fma(dx[k], dy[k], ndy[k], x[k], t);
        }
    };
    // B += (multiplier) * (value d segments away)
    auto keep = [](f2x m, bool lo, bool hi) {
        return m & ((lo ? 0x00000000ffffffffull : 0ull) | (hi ? 0xffffffff00000000ull : 0ull));
    };
    auto scan_up = [&](PC Bv) {
        PC Am = C.Af;
#pragma unroll 1
        for (int l = 0; l < nf; ++l) {
            const int d = 1 << l;
            const PC Bo = pc_up(Bv, d);
            const bool lo = g >= d, hi = true;
            const f2x mx = keep(Am.x, lo, hi), my = keep(Am.y, lo, hi);
            Bv = pc_fma(mx, my, p_neg(my), Bo, Bv);
            if (l + 1 < nf) Am = pc_mul(Am.x, Am.y, p_neg(Am.y), pc_up(Am, d));
        }
        return Bv;
    };
    auto scan_down = [&](PC Bv) {
        PC Am = C.Ab;
#pragma unroll 1
        for (int l = 0; l < nb; ++l) {
            const int d = 1 << l;
            const PC Bo = pc_down(Bv, d);
            const bool lo = true, hi = g + d < 32;
            const f2x mx = keep(Am.x, lo, hi), my = keep(Am.y, lo, hi);
            Bv = pc_fma(mx, my, p_neg(my), Bo, Bv);
            if (l + 1 < nb) Am = pc_mul(Am.x, Am.y, p_neg(Am.y), pc_down(Am, d));
        }
        return Bv;
    };
    // r <- M^{-1} r (seg_solve_lu)
    auto solve = [&](PC(&r)[4]) {
        PC z = pc_mul(C.ex[0], C.ey[0], ney[0], r[0]);
#pragma unroll
        for (int k = 1; k < 4; ++k) z = pc_mul(C.ex[k], C.ey[k], ney[k], pc_axpy(nsub[k], z, r[k]));
        z = pc_up(scan_up(z), 1);   // the first segment's meets sub = 0
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            z = pc_mul(C.ex[k], C.ey[k], ney[k], pc_axpy(nsub[k], z, r[k]));
            r[k] = z;
        }
        PC x = r[3];
#pragma unroll
        for (int k = 2; k >= 0; --k) x = pc_fma(nfx[k], nfy[k], fy[k], x, r[k]);
        x = pc_down(scan_down(x), 1);   // the last segment's meets fk = 0
#pragma unroll
        for (int k = 3; k >= 0; --k) {
            x = pc_fma(nfx[k], nfy[k], fy[k], x, r[k]);
            r[k] = x;
        }
    };
    PC v[4];
    {
        PC Wu[4];
        apply(w, Wu);
        const f2x mh = p_dup(-K.h), mgh = p_dup(-K.gh);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            v[k] = pc_axpy(mh, Wu[k], y[k]);     // u_Pi - h Wu
            y[k] = pc_axpy(mgh, Wu[k], y[k]);    // stage 1 right side
        }
    }
    solve(y);                                    // U1_Pi
    u1(w, y);
    {
        PC Y[4];
        apply(y, Y);
        const f2x h1g = p_dup(K.h1g), mg2 = p_dup(-K.g2h1);
        const f2x ctr = p_mul(h1g, C.row[SF_CTR]), cti = p_mul(h1g, C.row[SF_CTI]), ctc = p_mul(h1g, C.row[SF_CTC]);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            w[k] = pc_axpy(h1g, y[k], w[k]);     // u_Phi + (1 - gamma) h U1_Pi
            const f2x nctx = p_neg(p_mul(sg[k], ctr)), cty = p_mul(sg[k], p_fma(ctc, th(k, 1), cti));
            v[k] = pc_fma(nctx, p_neg(cty), cty, y[k], pc_axpy(mg2, Y[k], v[k]));   // stage 2 right side
        }
    }
    solve(v);                                    // U2_Pi
    const f2x gh = p_dup(K.gh);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        w[k] = pc_axpy(gh, v[k], w[k]);
        y[k] = v[k];
    }
}

// One half of the row: its elements in shared memory, the pivots, the lane's
// segment products, the step-table entry (a valid interior row's even where
// the row itself is not active), the stored scan levels and, for the
// adjoint's tape, where U1 goes (or NULL).  An active row is solved; a row in
// the tile that is not active is set to zero; other rows are left alone.
struct PairRow {
    float2 *phi, *pi;
    const float2 *piv, *seg;
    const float *f;
    float2 *u1f, *u1g;
    int plan, n;             // theta elements of the part
    bool active, in_tile;
};

// Fills the paired theta table (StepParams::th2, and the tiles' copies): entry j holds the values at theta j and
// 128 + j; zero past the row's end, so that padding elements have no coupling.
__device__ __forceinline__ void pair_th_fill(f2x *th2, const float *thtab, int N, int tid, int NT)
{
    constexpr int NP = 128;
    const int src[kPairTh] = {TF_S2, TF_C, TF_AM, TF_A0, TF_AP};
    for (int idx = tid; idx < kPairTh * NP; idx += NT) {
        const int q = idx / NP, j = idx - q * NP, jh = j + 128;
        int f = src[0];
#pragma unroll
        for (int k = 1; k < kPairTh; ++k)
            if (q == k) f = src[k];
        th2[idx] = pk2(j < N ? thtab[f * N + j] : 0.0f, jh < N ? thtab[f * N + jh] : 0.0f);
    }
}

__device__ __forceinline__ void pair_load4(const float2 *src, int j0, int len, bool vec, float2 pad, float2 (&r)[4])
{
    if (vec && len == 4) {
        vload<4>(r, src + j0);
    } else {
#pragma unroll
        for (int k = 0; k < 4; ++k) r[k] = k < len ? src[j0 + k] : pad;
    }
}
__device__ __forceinline__ void pair_store4(float2 *dst, int j0, int len, bool vec, const float2 (&r)[4])
{
    if (vec && len == 4) {
        vstore<4>(dst + j0, r);
    } else {
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (k < len) dst[j0 + k] = r[k];
    }
}
__device__ __forceinline__ void pair_store(const PairRow &A, const PairRow &B, float2 *PairRow::*dst, int j0, int lenA,
                                           int lenB, bool vec, const PC (&v)[4])
{
    float2 a[4], b[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        a[k] = make_float2(p_lo(v[k].x), p_lo(v[k].y));
        b[k] = make_float2(p_hi(v[k].x), p_hi(v[k].y));
    }
    if (A.in_tile) pair_store4(A.*dst, j0, lenA, vec, a);
    if (B.in_tile) pair_store4(B.*dst, j0, lenB, vec, b);
}

// One implicit SDIRK2 step of length h (constants K) on the row of halves
// (A, B) in shared memory, one warp (lane g).  th2: the paired theta table.
__device__ __forceinline__ void implicit_pair(const ImpConst<float> &K0, const PairRow &A, const PairRow &B,
                                              const f2x *th2, int g, bool vec)
{
    const ImpConst<float> K = K0;
    const int j0 = 4 * g;
    auto clamp4 = [](int n) { return n < 0 ? 0 : (n > 4 ? 4 : n); };
    const int lenA = clamp4(A.n - j0), lenB = clamp4(B.n - j0);
    const float2 zero = make_float2(0.0f, 0.0f), one = make_float2(1.0f, 0.0f);
    PairCoef C;
    PC w[4], y[4];
    float2 ra[4], rb[4];
    pair_load4(A.piv, j0, lenA, vec, one, ra);
    pair_load4(B.piv, j0, lenB, vec, one, rb);
    C.plan = A.plan;
    C.Af.x = C.Af.y = C.Ab.x = C.Ab.y = 0ull;
    if (A.plan) {
        const float4 sa = *reinterpret_cast<const float4 *>(A.seg), sb = *reinterpret_cast<const float4 *>(B.seg);
        C.Af = pc_pack(make_float2(sa.x, sa.y), make_float2(sb.x, sb.y));
        C.Ab = pc_pack(make_float2(sa.z, sa.w), make_float2(sb.z, sb.w));
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        C.ex[k] = pk2(ra[k].x, rb[k].x);
        C.ey[k] = pk2(ra[k].y, rb[k].y);
    }
    pair_load4(A.phi, j0, A.active ? lenA : 0, vec, zero, ra);
    pair_load4(B.phi, j0, B.active ? lenB : 0, vec, zero, rb);
#pragma unroll
    for (int k = 0; k < 4; ++k) w[k] = pc_pack(ra[k], rb[k]);
    pair_load4(A.pi, j0, A.active ? lenA : 0, vec, zero, ra);
    pair_load4(B.pi, j0, B.active ? lenB : 0, vec, zero, rb);
#pragma unroll
    for (int k = 0; k < 4; ++k) y[k] = pc_pack(ra[k], rb[k]);
    float f[8];
    vload<8>(f, A.f);
#pragma unroll
    for (int q = 0; q < 8; ++q) C.row[q] = p_dup(f[q]);
    pair_core(
        K, C, w, y, g, [&](int k, int q) { return th2[q * 128 + j0 + k]; },
        [&](const PC(&w1)[4], const PC(&y1)[4]) {
            if (!A.u1f) return;
            // the first stage value U1 (U1_Phi = u_Phi + gh U1_Pi), for the adjoint's spin term
            const f2x gh = p_dup(K.gh);
            PC t[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) t[k] = pc_axpy(gh, y1[k], w1[k]);
            pair_store(A, B, &PairRow::u1f, j0, lenA, lenB, vec, t);
            pair_store(A, B, &PairRow::u1g, j0, lenA, lenB, vec, y1);
        });
    pair_store(A, B, &PairRow::phi, j0, lenA, lenB, vec, w);
    pair_store(A, B, &PairRow::pi, j0, lenA, lenB, vec, y);
}

}  // namespace
}  // namespace teuk
