// teuk_adjoint.cuh -- device code shared by the adjoint kernels: the source
// term's derivatives.
#pragma once

#include "teuk_dev.cuh"

namespace teuk {
namespace {

// Sums a CTA of the adjoint step with the spin derivative leaves.
constexpr int kNPart = 6;

// Adds conj(lam) * coef * (unit source) * phase to the amplitude sum cA and
// conj(lam) * coef * (source) * (rho d r0*/d r0 - i m Omega' t) to the orbit
// sum cr (rho = (r* - r0*)/sigma_r^2): the derivatives of the source term
// A F_pref G(r*, theta) e^{-i m Omega t} with respect to A and r0.
template <typename T>
__device__ __forceinline__ void source_grad(const StepParams<T> &p, typename V2<T>::t lam, double coef,
                                            typename V2<T>::t u, double2 ph, double rs, double t, double2 &cA,
                                            double2 &cr)
{
    const double lr = (double)lam.x, li = -(double)lam.y;             // conj(lam)
    const double ur = (double)u.x * ph.x - (double)u.y * ph.y, ui = (double)u.x * ph.y + (double)u.y * ph.x;
    const double vr = coef * (lr * ur - li * ui), vi = coef * (lr * ui + li * ur);   // conj(lam) coef U ph
    cA.x += vr;
    cA.y += vi;
    const double fr = p.amp_re * vr - p.amp_im * vi, fi = p.amp_re * vi + p.amp_im * vr;   // times A
    const double zr = (rs - p.rs0) * p.inv_sig_r2 * p.drs0_dr0, zi = -p.m_dOmega * t;
    cr.x += fr * zr - fi * zi;
    cr.y += fr * zi + fi * zr;
}

// The source term of a stage, S = F ph (ph: the scaled phase), as the
// forward step forms it, and dS/da: F = SRC sg (SR2 GTH + GA2) through its
// factors and 1/Sigma^2, the phase through Omega(a) (mdt = m t dOmega/da).
template <typename T>
__device__ __forceinline__ void src_da(const T *f, const T *df, T sg, T dsg, T gth, T ga2, T dga2,
                                       typename V2<T>::t ph, T mdt, typename V2<T>::t &Sv, typename V2<T>::t &dS)
{
    typedef typename V2<T>::t c2;
    const T X = fma(f[SF_SR2], gth, ga2), dX = fma(df[SF_SR2], gth, dga2);
    const c2 src = cmk<c2>(f[SF_SRE], f[SF_SIM]), dsrc = cmk<c2>(df[SF_SRE], df[SF_SIM]);
    const c2 F = cscale<c2>(sg * X, src);
    const c2 dF = cadd(cscale<c2>(sg * X, dsrc), cscale<c2>(fma(dsg, X, sg * dX), src));
    Sv = cmul(F, ph);
    // d/da e^{-i m Omega t} = -i m t (dOmega/da) e^{-i m Omega t}
    dS = cadd(cmul(dF, ph), cmk<c2>(Sv.y * mdt, -Sv.x * mdt));
}

}  // namespace

// acc[c] += the nblk CTAs' sums part[kNPart b + c], c < kNPart, in a fixed
// order (teuk_adjoint.cu).
cudaError_t launch_part_reduce(const double *part, int nblk, double *acc, cudaStream_t st);

// Shared memory of a kernel that solves one row (physical_row, k_seed).
template <typename T>
static inline size_t sample_smem_bytes(int Nth)
{
    const size_t row = (size_t)((Nth + 1) & ~1);
    return 2 * row * sizeof(typename V2<T>::t) + ((size_t)NSF + (size_t)NTF * Nth) * sizeof(T) +
           pair_th_bytes(Nth, (int)sizeof(T));
}

}  // namespace teuk
