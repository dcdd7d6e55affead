// teuk_adjoint_f64.cu -- the FP64 adjoint step on materialised planes.
//
// What k_adjoint_spin does for a full step, in the fewest FP64 instructions
// (the FP64 pipe starts one per scheduler and 64 cycles and bounds the step):
//   - the transposed Lax-Wendroff stages are the transposed three-point
//     stencil of the forward step's planes (16 multiply-adds and 8 additions
//     an element; the two transposed stages took 60), their spin term the
//     forward stencil with differentiated coefficients (20 and 8; 50), and no
//     midpoint is stored;
//   - C_h^H reads the forward step's planes too: with nu2 = A^{-H} mu and
//     nu1 = A^{-H}(c J^H nu2) (see teuk_adjoint.cu), the right side of the
//     second solve is c mu_Phi minus the second stage's operator, transposed,
//     on nu2_Pi, and C_h^H mu = (mu_Phi - gh W^H (nu1_Pi + nu2_Pi / gamma),
//     nu1_Pi + nu2_Pi): 57 an element and 48 a segment for the two products
//     with W^H, the solves and the rest, as the forward row solve (about 100
//     before, and the scan levels were voted for in every call);
//   - the sample's adjoint and spin term, which are linear in g_n, come from
//     two vectors formed once (launch_seed, launch_delta) instead of an FP64
//     row solve by one warp at the side of the first tile.
// 4096 x 64, per step: with the spin term from the tape 156 -> 108 us, recomputing
// the stage values 199 -> 140.
#include "teuk_adjoint.cuh"

namespace teuk {
namespace {

// C_h^H on one row in place (see above), and with SPIN this lane's part of
// <mu, dC_h u> from the forward stage values (u1, u2 as in
// implicit_row_adj_spin).
template <int S, bool SPIN>
__device__ __forceinline__ double row_adjoint(const ImpConst<double> &K, const StepPlanes<double> &M,
                                              const AdjPlanes &A, double2 *lf, double2 *lg, const double2 *u1f,
                                              const double2 *u1g, const double2 *u2f, const double2 *u2g, int gi, int N,
                                              bool active, bool in_tile, int g, int G, bool vec)
{
    typedef double2 c2;
    const c2 zero = cmk<c2>(0.0, 0.0), one = cmk<c2>(1.0, 0.0);
    const int j0 = g * S;
    int len = N - j0;
    len = len < 0 ? 0 : (len > S ? S : len);
    const int lenw = len;
    if (!active) {
        len = 0;
        gi = 1;
    }
    const size_t o = (size_t)gi * N + j0;
    const bool whole = vec && len == S;
    auto cseg = [&](const c2 *src, c2 pad, c2(&r)[S]) {
        if (whole) {
            vload<S>(r, src);
        } else {
#pragma unroll
            for (int k = 0; k < S; ++k) r[k] = k < len ? src[k] : pad;
        }
    };
    auto rseg = [&](const double *src, double(&r)[S]) {
        if (whole) {
            vload<S>(r, src);
        } else {
#pragma unroll
            for (int k = 0; k < S; ++k) r[k] = k < len ? src[k] : 0.0;
        }
    };
    // M^H = U^H L^H: t_j = r_j - conj(fk_{j-1}) t_{j-1},
    // x_j = conj(e_j) (t_j - sub_{j+1} x_{j+1})
    c2 e[S], fm[S], pb[S];
    double subn[S];
    {
        c2 fk[S];
        double sub[S];
        cseg(K.piv + o, one, e);
        cseg(M.fk + o, zero, fk);
        rseg(M.sub + o, sub);
        cseg(A.pb + o, zero, pb);
        const c2 fkp = shfl_up_c(fk[S - 1], 1, G);
        const double sn = __shfl_down_sync(0xffffffffu, sub[0], 1, G);
#pragma unroll
        for (int k = 0; k < S; ++k) {
            e[k] = conj_c(e[k]);
            fm[k] = k ? conj_c(fk[k ? k - 1 : 0]) : (g == 0 ? zero : conj_c(fkp));
            subn[k] = k + 1 < S ? sub[k + 1 < S ? k + 1 : 0] : (g == G - 1 ? 0.0 : sn);
        }
    }
    const int plan = active ? A.plan[gi] : 0, nf = plan & 0xff, nb = (plan >> 8) & 0xff;
    const int nfw = (int)__reduce_max_sync(0xffffffffu, (unsigned)nf), nbw = (int)__reduce_max_sync(0xffffffffu, (unsigned)nb);
    c2 Af = zero;
    if (nfw > 0) Af = A.af[(size_t)gi * G + g];
    auto solve = [&](c2(&r)[S]) {
        c2 B = r[0], Am = Af;
#pragma unroll
        for (int k = 1; k < S; ++k) B = cfnma(fm[k], B, r[k]);
#pragma unroll 1
        for (int l = 0; l < nfw; ++l) {
            const int d = 1 << l;
            const c2 Bo = shfl_up_c(B, d, G);
            c2 Ao = one;
            if (l + 1 < nfw) Ao = shfl_up_c(Am, d, G);
            if (l < nf && g >= d) {
                B = cfma(Am, Bo, B);
                if (l + 1 < nf) Am = cmul(Am, Ao);
            }
        }
        c2 t = shfl_up_c(B, 1, G);   // lane 0's meets fm = 0
#pragma unroll
        for (int k = 0; k < S; ++k) {
            t = cfnma(fm[k], t, r[k]);
            r[k] = t;
        }
        r[S - 1] = cmul(e[S - 1], r[S - 1]);
#pragma unroll
        for (int k = S - 2; k >= 0; --k) r[k] = cmul(e[k], caxpy(-subn[k], r[k + 1], r[k]));
        B = r[0];
        Am = pb[0];
#pragma unroll 1
        for (int l = 0; l < nbw; ++l) {
            const int d = 1 << l;
            const c2 Bo = shfl_down_c(B, d, G);
            c2 Ao = one;
            if (l + 1 < nbw) Ao = shfl_down_c(Am, d, G);
            if (l < nb && g + d < G) {
                B = cfma(Am, Bo, B);
                if (l + 1 < nb) Am = cmul(Am, Ao);
            }
        }
        const c2 x = shfl_down_c(B, 1, G);   // the last lane's meets pb = 0
#pragma unroll
        for (int k = 0; k < S; ++k) r[k] = cfma(pb[k], x, r[k]);
    };
    // acc - (wu_{j-1} x_{j-1} + conj(d_j) x_j + wl_{j+1} x_{j+1})
    auto minus_tri_h = [&](const double *wl_, const c2 *d_, const double *wu_, const c2(&x)[S], c2(&acc)[S]) {
        double wl[S], wu[S];
        c2 d[S];
        rseg(wl_ + o, wl);
        cseg(d_ + o, zero, d);
        rseg(wu_ + o, wu);
        double wup = __shfl_up_sync(0xffffffffu, wu[S - 1], 1, G), wln = __shfl_down_sync(0xffffffffu, wl[0], 1, G);
        if (g == 0) wup = 0.0;
        if (g == G - 1) wln = 0.0;
        const c2 xl = shfl_up_c(x[S - 1], 1, G), xr = shfl_down_c(x[0], 1, G);
#pragma unroll
        for (int k = 0; k < S; ++k) {
            const c2 xm = k ? x[k ? k - 1 : 0] : xl, xp = (k + 1 < S) ? x[(k + 1) < S ? k + 1 : S - 1] : xr;
            const double a = k ? wu[k ? k - 1 : 0] : wup, b = (k + 1 < S) ? wl[(k + 1) < S ? k + 1 : S - 1] : wln;
            acc[k] = cfnma(conj_c(d[k]), x[k], caxpy(-b, xp, caxpy(-a, xm, acc[k])));
        }
    };
    const double gh = K.gh, c = K.h1g;
    c2 w[S], n2[S], n1[S];   // mu_Phi, nu2_Pi, nu1_Pi
    cseg(lf + j0, zero, w);
    cseg(lg + j0, zero, n2);
#pragma unroll
    for (int k = 0; k < S; ++k) {
        n2[k] = caxpy(gh, w[k], n2[k]);
        n1[k] = cscale<c2>(c, w[k]);
    }
    solve(n2);
    minus_tri_h(M.w2l, M.d2, M.w2u, n2, n1);
    solve(n1);
    {
        c2 q[S];
#pragma unroll
        for (int k = 0; k < S; ++k) q[k] = caxpy(1.0 / kGamma, n2[k], n1[k]);
        minus_tri_h(M.w1l, M.d1, M.w1u, q, w);
#pragma unroll
        for (int k = 0; k < S; ++k) q[k] = cadd(n1[k], n2[k]);
        if (in_tile) row_store<double, S>(lf, lg, w, q, j0, lenw, vec);
    }
    if constexpr (!SPIN) return 0.0;
    // -Re sum conj(c nu2 + gh nu1) Q1 + conj(gh nu2) Q2, Q = dW x_Phi + dc_t x_Pi of the stage values
    double acc = 0.0;
#pragma unroll
    for (int k = 0; k < S; ++k) {
        n1[k] = caxpy(c, n2[k], cscale<c2>(gh, n1[k]));
        n2[k] = cscale<c2>(gh, n2[k]);
    }
    auto dots = [&](const c2 *uf, const c2 *ug, const c2(&nu)[S]) {
        c2 a[S];
        cseg(uf + j0, zero, a);
        c2 vl = shfl_up_c(a[S - 1], 1, G), vr = shfl_down_c(a[0], 1, G);
        if (g == 0) vl = zero;
        if (g == G - 1) vr = zero;
#pragma unroll
        for (int k = 0; k < S; ++k) {
            if (k < len) {
                const c2 b = ug[j0 + k];
                const size_t q = ((size_t)gi * 3) * N + j0 + k;
                const c2 ddg = A.dimp[q], dct = A.dimp[q + N], dq = A.dimp[q + 2 * (size_t)N];
                const c2 vm = k ? a[k ? k - 1 : 0] : vl, vp = (k + 1 < S) ? a[(k + 1) < S ? k + 1 : S - 1] : vr;
                const c2 Q = cfma(dct, b, cfma(ddg, a[k], caxpy(dq.y, vp, cscale<c2>(dq.x, vm))));
                acc = fma(-nu[k].x, Q.x, fma(-nu[k].y, Q.y, acc));
            }
        }
    };
    dots(u1f, u1g, n1);
    dots(u2f, u2g, n2);
    return acc;
}

// One full adjoint step; arguments and per-CTA sums as k_adjoint_spin.  Tile
// rows i0-1 .. i0+TR: lam_{n+1} (lF, lG), with SPIN the forward stage values
// U2 (vF, vG) and U1 (uF, uG).  seed: the sample's adjoint vector, delta: the
// sample's spin derivative as a vector on the extraction row ([2][N] each).
template <int S, bool SPIN>
__global__ void __launch_bounds__(256, 1)
    k_adjoint_f64(const StepParams<double> p, const double2 *sin, const double2 *tape, const double2 *gseed,
                  const AdjPlanes A, double *part)
{
    launch_turn();
    typedef double2 c2;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ double s_red[8][kNPart];
    __shared__ double2 s_ph[2];   // the source phases at t_n and t_n + dt/2
    const int Nr = p.Nr, N = p.Nth, TR = p.tile_rows, R = TR + 2;
    const int tid = threadIdx.x, NT = blockDim.x;
    const int tile = (int)blockIdx.x, i0 = tile * TR, g0 = i0 - 1;
    const int G = p.group, g = tid % G;
    const ImpConst<double> &K = p.full;
    const c2 zero = cmk<c2>(0.0, 0.0);
    const bool vec = p.vec != 0;
    const unsigned plane = (unsigned)R * (unsigned)N;
    c2 *lF = (c2 *)smem_raw, *lG = lF + plane;
    c2 *vF = lG + plane, *vG = vF + plane, *uF = vG + plane, *uG = uF + plane;   // SPIN only

    // ---- lam_{n+1}, and s_n or the recorded stage values
    const c2 *t1 = tape, *t2 = tape ? tape + tape_u2_off(Nr, N) : sin;
    for (int lr = tid / N, j = tid - lr * N; lr < R;) {
        const int gi = g0 + lr, idx = lr * N + j;
        const bool on = gi >= 0 && gi < Nr;
        const size_t qf = (size_t)gi * N + j, qg = ((size_t)Nr + gi) * N + j;
        lF[idx] = on ? p.uin[qf] : zero;
        lG[idx] = on ? p.uin[qg] : zero;
        if constexpr (SPIN) {
            vF[idx] = on ? t2[qf] : zero;
            vG[idx] = on ? t2[qg] : zero;
            if (tape) {
                uF[idx] = on ? t1[qf] : zero;
                uG[idx] = on ? t1[qg] : zero;
            }
        }
        for (j += NT; j >= N; j -= N) ++lr;
    }
    const bool src = SPIN && p.patch_np > 0 && i0 + TR >= p.patch_p0 && g0 <= p.patch_p0 + p.patch_np;
    const bool srcu = p.unit_np > 0 && i0 + TR >= p.unit_p0 && g0 <= p.unit_p0 + p.unit_np;
    const double t1s = (double)p.nfix * p.dt64, t2s = t1s + 0.5 * p.dt64;
    if ((src || srcu) && tid >= NT - 2) s_ph[tid - (NT - 2)] = phase_at(p.mOmega, tid == NT - 2 ? t1s : t2s);
    __syncthreads();
    const int rpp = NT / G, wq = (tid & ~31) / G, tq = tid / G;
    if constexpr (SPIN) {
        if (!tape) {
            // forward implicit stage: (vF, vG) <- U2 = C_h s_n, (uF, uG) <- U1, bit for bit the step's
            for (int base = 0; base < R; base += rpp) {
                if (base + wq >= R) continue;
                const int lr = base + tq, gi = g0 + lr;
                const bool in_tile = lr < R, active = in_tile && gi >= 1 && gi <= Nr - 2;
                const int lrc = in_tile ? lr : 0;
                implicit_row_mat<double, S>(K, p.mat, vF + lrc * N, vG + lrc * N, gi, N, active, in_tile, g, G, vec,
                                            active ? K.plan[gi] : 0, uF + lrc * N, uG + lrc * N);
            }
            __syncthreads();
        }
    }

    // ---- transposed Lax-Wendroff stencil on rows 1 .. TR, its spin terms and
    // the source derivatives; thread (segment, column) marches down its rows
    double2 cA = zero, cr = zero;
    double spin = 0.0;
    const int top = Nr - g0 < TR + 1 ? Nr - g0 : TR + 1;   // first tile row past the output rows
    if (src || srcu) {
        // Source derivatives, an element a thread: the half node above each
        // output row (adjoint wm from its two nodes) and the node.  The phases,
        // stage lengths and the amplitude are common factors, so the elements
        // only add to sums of the adjoint times the patch (unit and spin
        // derivative); taken element by element they were 180 FP64 instructions
        // each and held the source's tile for 50 us.
        c2 s1 = zero, s1r = zero, s2 = zero, s2r = zero, X1 = zero, Y1 = zero, X2 = zero, Y2 = zero;
        int q0 = p.unit_p0 - g0, q1 = p.unit_p0 + p.unit_np - g0;   // tile rows of the patch
        q0 = q0 < 1 ? 1 : q0;
        q1 = q1 < top ? q1 : top;
        const double zc = p.inv_sig_r2 * p.drs0_dr0;
        for (int lr = q0 + tid / N, j = tid % N; lr < q1;) {
            const int gi = g0 + lr;
            const size_t pr = (size_t)(gi - p.unit_p0) * 2 * N + j;
            const c2 gg = lG[lr * N + j];
            if (gi >= 1 && gi <= Nr - 2) {
                const double u = p.patchu[pr].x, z = (p.rs_min64 + (double)gi * p.drs64 - p.rs0) * zc;
                const c2 t = cscale<c2>(u, gg);
                s2 = cadd(s2, t);
                s2r = caxpy(z, t, s2r);
                if (SPIN && src) {
                    X2 = cfma(conj_c(gg), p.patchd[pr], X2);
                    Y2 = cfma(conj_c(gg), p.patch[pr], Y2);
                }
            }
            if (gi <= Nr - 2) {
                const c2 *q = p.mat.lw + (size_t)gi * kLwStencil * N + j, *n = q + kLwStencil * N;
                const c2 gn = lG[(lr + 1) * N + j];
                const c2 wm = caxpy(q[0].x + q[N].x, gg, cscale<c2>(-(n[0].x + n[N].x), gn));
                const double u = p.patchu[pr + N].x, z = (p.rs_min64 + ((double)gi + 0.5) * p.drs64 - p.rs0) * zc;
                const c2 t = cscale<c2>(u, wm);
                s1 = cadd(s1, t);
                s1r = caxpy(z, t, s1r);
                if (SPIN && src) {
                    const c2 *dq = A.dlw + (size_t)gi * kLwStencil * N + j, *dn = dq + kLwStencil * N;
                    const c2 wd = caxpy(dq[0].x + dq[N].x, gg, cscale<c2>(-(dn[0].x + dn[N].x), gn));
                    const c2 F = p.patch[pr + N];
                    X1 = cfma(conj_c(wm), p.patchd[pr + N], cfma(conj_c(wd), F, X1));
                    Y1 = cfma(conj_c(wm), F, Y1);
                }
            }
            for (j += NT; j >= N; j -= N) ++lr;
        }
        const c2 l1 = cscale<c2>(p.half_dt, s_ph[0]), l2 = cscale<c2>(p.dt, s_ph[1]);
        // d/dA and d/dr0: A (rho dr0*/dr0 - i m Omega' t) times the unit source
        const c2 v1 = cmul(l1, conj_c(s1)), v2 = cmul(l2, conj_c(s2));
        cA = cadd(v1, v2);
        const double z1 = -p.m_dOmega * t1s, z2 = -p.m_dOmega * t2s;
        c2 r = cadd(cmul(l1, conj_c(s1r)), cmul(l2, conj_c(s2r)));
        r = cadd(r, cmk<c2>(-(z1 * v1.y + z2 * v2.y), z1 * v1.x + z2 * v2.x));
        cr = cmul(cmk<c2>(p.amp_re, p.amp_im), r);
        if (SPIN && src) {
            // the source's derivative and its phase's, -i m t (dOmega/da)
            const double m1 = p.m_dOmega_da * t1s, m2 = p.m_dOmega_da * t2s;
            spin = cmul(l1, cadd(X1, cmk<c2>(m1 * Y1.y, -m1 * Y1.x))).x + cmul(l2, cadd(X2, cmk<c2>(m2 * Y2.y, -m2 * Y2.x))).x;
        }
    }
    auto march = [&](int j, int ra, int rb, c2 fm, c2 gm, c2 nf, c2 ng) {
        struct Row {
            c2 a, b, cm, cp;
        };
        auto row = [&](int lr) {
            Row r;
            const int gi = g0 + lr;
            if (gi >= 0 && gi < Nr) {
                const c2 *q = p.mat.lw + (size_t)gi * kLwStencil * N + j;
                r.a = q[0];
                r.b = q[N];
                r.cm = q[2 * N];
                r.cp = q[3 * N];
            } else {
                r.a = r.b = r.cm = r.cp = zero;
            }
            return r;
        };
        // what rows lo and up = lo + 1 send through the difference between them
        auto flux = [&](const Row &lo, c2 fl, c2 gl, const Row &up, c2 fu, c2 gu, c2 &T, c2 &U) {
            T = cfma(conj_c(up.cm), gu, cfnma(conj_c(lo.cp), gl, caxpy(up.a.x, fu, cscale<c2>(lo.a.y, fl))));
            U = caxpy(up.b.x, gu, cscale<c2>(lo.b.y, gl));
        };
        Row cu = row(ra);
        c2 f = lF[ra * N + j], gg = lG[ra * N + j], Tm, Um;
        flux(row(ra - 1), fm, gm, cu, f, gg, Tm, Um);
        for (int lr = ra; lr < rb; ++lr) {
            const int gi = g0 + lr;
            const Row nx = row(lr + 1);
            c2 fn = nf, gn = ng;
            if (lr + 1 < rb) {
                fn = lF[(lr + 1) * N + j];
                gn = lG[(lr + 1) * N + j];
            }
            c2 Tp, Up;
            flux(cu, f, gg, nx, fn, gn, Tp, Up);
            // boundary rows are no output of the step: nothing but the fluxes reaches them
            const bool interior = gi >= 1 && gi <= Nr - 2;
            const c2 wF = cadd(interior ? f : zero, csub(Tp, Tm)), wG = csub(interior ? gg : zero, csub(Up, Um));
            if constexpr (SPIN) {
                if (interior) {
                    const c2 *q = A.dlw + (size_t)gi * kLwStencil * N + j;
                    const c2 a = q[0], b = q[N], cm = q[2 * N], cp = q[3 * N];
                    const int x = lr * N + j;
                    const c2 vb = vF[x], gb = vG[x], dm = csub(vF[x - N], vb), dp = csub(vF[x + N], vb);
                    const c2 dF = caxpy(-a.y, dp, cscale<c2>(a.x, dm));
                    c2 dG = caxpy(b.y, csub(vG[x + N], gb), cscale<c2>(-b.x, csub(vG[x - N], gb)));
                    dG = cfma(cp, dp, cfma(cm, dm, dG));
                    spin = fma(f.x, dF.x, fma(f.y, dF.y, fma(gg.x, dG.x, fma(gg.y, dG.y, spin))));
                }
            }
            lF[lr * N + j] = wF;
            lG[lr * N + j] = wG;
            Tm = Tp;
            Um = Up;
            f = fn;
            gg = gn;
            cu = nx;
        }
    };
    if (N <= NT) {
        const int nseg = NT / N, sl = (top - 1 + nseg - 1) / nseg, sgm = tid / N, j = tid - sgm * N;
        const int ra = 1 + sgm * sl, rb = ra + sl < top ? ra + sl : top;
        const bool work = sgm < nseg && ra < rb;
        c2 fm = zero, gm = zero, nf = zero, ng = zero;
        if (work) {
            fm = lF[(ra - 1) * N + j];
            gm = lG[(ra - 1) * N + j];
            nf = lF[rb * N + j];
            ng = lG[rb * N + j];
        }
        __syncthreads();
        if (work) march(j, ra, rb, fm, gm, nf, ng);
    } else {
        // the march writes its columns in place; the source derivatives above
        // read whatever columns their elements fall on
        __syncthreads();
        for (int j = tid; j < N; j += NT) march(j, 1, top, lF[j], lG[j], lF[top * N + j], lG[top * N + j]);
    }
    __syncthreads();

    // ---- C_h^H on the output rows with the implicit stage's spin terms
    for (int base = 1; base <= TR; base += rpp) {
        if (base + wq > TR) continue;
        const int lr = base + tq, gi = g0 + lr;
        const bool in_tile = lr <= TR && gi < Nr, active = in_tile && gi >= 1 && gi <= Nr - 2;
        const int lrc = in_tile ? lr : 1;
        const double d = row_adjoint<S, SPIN>(K, p.mat, A, lF + lrc * N, lG + lrc * N, uF + lrc * N, uG + lrc * N,
                                              vF + lrc * N, vG + lrc * N, gi, N, active, in_tile, g, G, vec);
        if (active) spin += d;
    }
    __syncthreads();

    // ---- extraction seed g_n C_{dt/2}^H E^H, and the sample's spin term Re conj(g_n) delta . s_n
    if (gseed != nullptr && p.i_ext >= i0 && p.i_ext < i0 + TR && p.i_ext < Nr) {
        const int lx = p.i_ext - g0;
        const double2 gv = *gseed;
        for (int j = tid; j < N; j += NT) {
            lF[lx * N + j] = cfma(gv, p.seed[j], lF[lx * N + j]);
            lG[lx * N + j] = cfma(gv, p.seed[N + j], lG[lx * N + j]);
            if constexpr (SPIN) {
                const c2 sf = tape ? tape[tape_x_off(Nr, N) + j] : sin[(size_t)p.i_ext * N + j];
                const c2 sg = tape ? tape[tape_x_off(Nr, N) + N + j] : sin[((size_t)Nr + p.i_ext) * N + j];
                const c2 d = cfma(A.delta[j], sf, cmul(A.delta[N + j], sg));
                spin = fma(gv.x, d.x, fma(gv.y, d.y, spin));
            }
        }
        __syncthreads();
    }

    // ---- store lam_n
    for (int lr = 1 + tid / N, j = tid % N; lr < top;) {
        const int gi = g0 + lr;
        p.uout[(size_t)gi * N + j] = lF[lr * N + j];
        p.uout[((size_t)Nr + gi) * N + j] = lG[lr * N + j];
        for (j += NT; j >= N; j -= N) ++lr;
    }

    // ---- this CTA's sums (fixed-order reduction)
    double v[kNPart] = {cA.x, cA.y, cr.x, cr.y, spin, 0.0};
#pragma unroll
    for (int c = 0; c < kNPart; ++c)
        for (int o = 16; o > 0; o >>= 1) v[c] += __shfl_xor_sync(0xffffffffu, v[c], o);
    if ((tid & 31) == 0)
        for (int c = 0; c < kNPart; ++c) s_red[tid >> 5][c] = v[c];
    __syncthreads();
    if (tid < kNPart) {
        double acc = 0.0;
        for (int w = 0; w < NT / 32; ++w) acc += s_red[w][tid];
        part[kNPart * tile + tid] = acc;
    }
}

// ---- the planes, once per teuk_adjoint_prepare

// Spin derivatives of the stencil (dlw) and of the implicit operator (dimp),
// a thread per grid element.
__global__ void __launch_bounds__(256) k_adj_planes(const StepParams<double> p, const AdjPlanes A)
{
    typedef double2 c2;
    const int N = p.Nth, Nr = p.Nr;
    const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (long long)Nr * N) return;
    const int i = (int)(idx / N), j = (int)(idx - (long long)i * N);
    c2 *dl = (c2 *)A.dlw + (size_t)i * kLwStencil * N + j, *di = (c2 *)A.dimp + (size_t)i * 3 * N + j;
    if (i < 1 || i > Nr - 2) {
        for (int k = 0; k < kLwStencil; ++k) dl[k * N] = zero_c2<c2>();
        for (int k = 0; k < 3; ++k) di[k * N] = zero_c2<c2>();
        return;
    }
    const double *f = p.stab + (size_t)(2 * i) * NSF, *df = p.dstab + (size_t)(2 * i) * NSF;
    const double S2 = p.thtab[TF_S2 * N + j], C = p.thtab[TF_C * N + j];
    const LwDa<double> n = lw_coef_da<double>(f, df, S2, C), m = lw_coef_da<double>(f - NSF, df - NSF, S2, C),
                       q = lw_coef_da<double>(f + NSF, df + NSF, S2, C);
    const double b = n.beta, db = n.dbeta, bm = m.beta, dbm = m.dbeta, bp = q.beta, dbp = q.dbeta;
    dl[0] = cmk<c2>(db * (0.5 + bm) + b * dbm, db * (0.5 - bp) - b * dbp);
    dl[N] = cmk<c2>(db * (0.5 - bm) - b * dbm, db * (0.5 + bp) + b * dbp);
    auto lin = [](double s, c2 x, double t, c2 y) { return caxpy(s, x, cscale<c2>(t, y)); };
    dl[2 * N] = csub(lin(db, m.kap, b, m.dkap), lin(0.5 + bm, n.dkap, dbm, n.kap));
    dl[3 * N] = cadd(lin(db, q.kap, b, q.dkap), lin(0.5 - bp, n.dkap, -dbp, n.kap));
    const ImpRow<double> r = imp_row(p.full, f);
    double fr[8], dfr[8];
    vload<8>(fr, f);
    vload<8>(dfr, df);
    c2 ddg, dct;
    double dqam, dqap;
    imp_da<double>(r, fr, dfr, S2, C, p.thtab[TF_AM * N + j], p.thtab[TF_A0 * N + j], p.thtab[TF_AP * N + j], ddg, dct, dqam,
                   dqap);
    di[0] = ddg;
    di[N] = dct;
    di[2 * N] = cmk<c2>(dqam, dqap);
}

// d patch / da on the patch rows, from the source's factors and their
// derivatives (src_da).
__global__ void __launch_bounds__(256) k_patch_da(const StepParams<double> p)
{
    const int N = p.Nth, idx = (int)(blockIdx.x * blockDim.x + threadIdx.x);
    if (idx >= p.patch_np * 2 * N) return;
    const int j = idx % N, e = 2 * p.patch_p0 + idx / N;
    if (e > 2 * p.Nr - 2) return;
    const double *f = p.stab + (size_t)e * NSF, *df = p.dstab + (size_t)e * NSF;
    const LwDa<double> l = lw_coef_da<double>(f, df, p.thtab[TF_S2 * N + j], p.thtab[TF_C * N + j]);
    double2 F, dF;
    src_da<double>(f, df, l.sg, l.dsg, p.thtab[TF_GTH * N + j], p.thtab[TF_GA2 * N + j], p.thtab[TF_DGA2 * N + j],
                   make_double2(1.0, 0.0), 0.0, F, dF);
    ((double2 *)p.patchd)[idx] = dF;
}

// Scan levels of the transposed solves (the rule of scan_plan), the products
// pb and the forward segment products af; the lanes of a row as in the step.
template <int S>
__global__ void __launch_bounds__(256) k_adj_plans(const StepParams<double> p, const AdjPlanes A)
{
    typedef double2 c2;
    const int N = p.Nth, Nr = p.Nr, G = p.group, tid = threadIdx.x, g = tid % G;
    const int gi = (int)blockIdx.x * ((int)blockDim.x / G) + tid / G;
    const bool in_grid = gi < Nr, active = in_grid && gi >= 1 && gi <= Nr - 2;
    const int j0 = g * S;
    int len = active ? N - j0 : 0;
    len = len < 0 ? 0 : (len > S ? S : len);
    const size_t o = (size_t)(active ? gi : 1) * N + j0;
    const c2 zero = zero_c2<c2>();
    c2 fm[S], bm[S];
    c2 fkp = zero, ep = zero;   // the element before / this one, walking the segment
    {
        c2 last = len == S ? p.mat.fk[o + S - 1] : zero;
        fkp = shfl_up_c(last, 1, G);
        if (g == 0) fkp = zero;
        const double first = len > 0 ? p.mat.sub[o] : 0.0;
        double sn = __shfl_down_sync(0xffffffffu, first, 1, G);
        if (g == G - 1) sn = 0.0;
        for (int k = 0; k < S; ++k) {
            fm[k] = conj_c(fkp);
            fkp = k < len ? p.mat.fk[o + k] : zero;
            ep = k < len ? conj_c(p.full.piv[o + k]) : zero;
            const double sub = k + 1 < S ? (k + 1 < len ? p.mat.sub[o + k + 1] : 0.0) : sn;
            bm[k] = cscale<c2>(sub, ep);
        }
    }
    const ScanPlan<double> P = scan_plan<double, S>(fm, bm, g, G);
    if (in_grid) {
        if (g == 0) ((int *)A.plan)[gi] = P.nf | (P.nb << 8);
        ((c2 *)A.af)[(size_t)gi * G + g] = P.Af0;
        c2 Q = cmk<c2>(1.0, 0.0);
        for (int k = S - 1; k >= 0; --k) {
            Q = cmul(cmk<c2>(-bm[k].x, -bm[k].y), Q);
            if (j0 + k < N) ((c2 *)A.pb)[(size_t)gi * N + j0 + k] = active ? Q : zero;
        }
    }
}

}  // namespace

size_t adjoint_f64_smem_bytes(int tile_rows, int Nth, bool spin)
{
    return (spin ? 6 : 2) * ((size_t)tile_rows + 2) * Nth * sizeof(double2);
}

template <bool SPIN>
static void (*adjoint_fn(int Nth))(const StepParams<double>, const double2 *, const double2 *, const double2 *,
                                   const AdjPlanes, double *)
{
    const int seg = implicit_seg(Nth);
    return seg == kSegNarrow ? k_adjoint_f64<kSegNarrow, SPIN>
                             : (seg == kSeg ? k_adjoint_f64<kSeg, SPIN> : k_adjoint_f64<kSegWide, SPIN>);
}

cudaError_t launch_adjoint_f64(const StepParams<double> &p, int tile_rows, bool spin, const double2 *sin, const double2 *tape,
                               const double2 *gseed, const AdjPlanes &A, double *part, double *acc, cudaStream_t st)
{
    auto fn = spin ? adjoint_fn<true>(p.Nth) : adjoint_fn<false>(p.Nth);
    cudaError_t e = smem_limit_max((const void *)fn);
    if (e != cudaSuccess) return e;
    StepParams<double> q = p;
    q.tile_rows = tile_rows;
    const int grid = (p.Nr + tile_rows - 1) / tile_rows;
    e = launch_dep(fn, dim3((unsigned)grid), 256, adjoint_f64_smem_bytes(tile_rows, p.Nth, spin), st, q, sin, tape, gseed, A, part);
    if (e != cudaSuccess) return e;
    return launch_part_reduce(part, grid, acc, st);
}

cudaError_t launch_patch_da(const StepParams<double> &p, cudaStream_t st)
{
    k_patch_da<<<(unsigned)((p.patch_np * 2 * p.Nth + 255) / 256), 256, 0, st>>>(p);
    return cudaGetLastError();
}

cudaError_t launch_adjoint_f64_planes(const StepParams<double> &p, const AdjPlanes &A, cudaStream_t st)
{
    const long long n = (long long)p.Nr * p.Nth;
    k_adj_planes<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(p, A);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const int seg = implicit_seg(p.Nth), rows = 256 / p.group;
    auto fn = seg == kSegNarrow ? k_adj_plans<kSegNarrow> : (seg == kSeg ? k_adj_plans<kSeg> : k_adj_plans<kSegWide>);
    fn<<<(p.Nr + rows - 1) / rows, 256, 0, st>>>(p, A);
    return cudaGetLastError();
}

}  // namespace teuk
