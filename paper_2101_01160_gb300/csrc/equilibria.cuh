// Device functions of the analytic equilibria (Sec. 3), shared by the
// single-distribution entry points and the batched f_eq stage.
#pragma once

#include <cuda_runtime.h>
#include <math.h>

namespace mdlg {

// One-dimensional equilibrium of a particle uniform in a unit lattice cell
// displaced by a Gaussian of variance var (lattice units), landing u cells
// away: Eq. (feq_gaussian) with a^2 = var, N = a / sqrt(2 pi).  The WSG
// component f^c of Eq. (f_eq_wsg) is this with var = a^2 (c+1)/(lambda+1)
// (N_c^2 = 2 var).
__device__ inline double cell_gauss_1d(double u, double var) {
    const double s = sqrt(2.0 * var);             // a sqrt(2) = N_c
    const double norm = sqrt(var) * 0.39894228040143267794;   // a / sqrt(2 pi)
    const double um = u - 1.0, up = u + 1.0;
    const double e = exp(-(um * um) / (2.0 * var)) - 2.0 * exp(-(u * u) / (2.0 * var)) +
                     exp(-(up * up) / (2.0 * var));
    const double eu = erf(u / s);
    return norm * e + 0.5 * um * (erf(um / s) - eu) + 0.5 * up * (erf(up / s) - eu);
}

// Root of Eq. (lambda_eq) in the printed form: root 1 takes the '+' sign of
// the square root, root 2 (the paper's choice) the '-' sign.
__device__ inline double lambda_root(double mu2, double mu4, int root) {
    const double m22 = mu2 * mu2;
    const double r = sqrt(3.0 * (15.0 * m22 * m22 - 4.0 * m22 * mu4));
    const double num = -9.0 * m22 + 2.0 * mu4 + (root == 1 ? r : -r);
    return num / (2.0 * (3.0 * m22 - mu4));
}

// Poisson terms kept: |c - lambda| <= 12 sqrt(lambda) + 20 (tails < 1e-16).
__host__ __device__ inline int wsg_cmax(double lam) {
    return lam <= 0.0 ? 0 : (int)ceil(lam + 12.0 * sqrt(lam) + 20.0);
}
__host__ __device__ inline int wsg_cmin(double lam) {
    const double c = floor(lam - 12.0 * sqrt(lam) - 20.0);
    return c > 0.0 ? (int)c : 0;
}

// The sum over the window takes every k-th term, k times its weight.  For the
// Poisson weights alone the error is exactly sum_{m=1..k-1} of their
// characteristic function at 2 pi m / k, at most (k - 1) exp(-lambda (1 -
// cos(2 pi / k))) (the roots-of-unity filter); the factors they multiply vary
// over c ~ lambda, slower than the weights' width sqrt(lambda), except near
// c = 0, where the weight is exp(-lambda).  From lambda = 40 on with k =
// floor(0.45 sqrt(lambda)) the sums agree with the full ones to 1e-18 relative
// for probabilities above 1e-25 (40-digit arithmetic, lambda from 40 to 2,000,
// a^2 from 1e-4 to 20, |v| up to 10), and no window holds more than 137 terms,
// where lambda = 1e5 had 7,631.  (From about 1e-40 down the sum leans on its last
// terms and the two part, 1 % at 1e-46; FP64 has nothing there: the differences
// of error functions that a factor is made of are off by 1e-16.)
__host__ __device__ inline int wsg_stride(double lam) {
    return lam >= 40.0 ? (int)floor(0.45 * sqrt(lam)) : 1;
}
constexpr int WSG_MAX_TERMS = 144;

// Terms of the strided window: c = wsg_cmin + j * stride, j = 0 .. terms - 1.
__host__ __device__ inline int wsg_terms(double lam) {
    return (wsg_cmax(lam) - wsg_cmin(lam)) / wsg_stride(lam) + 1;
}

// Poisson weight Pois(c; lambda).  From c = 16 on in the saddle-point form of
// Loader (2000), exp(-delta(c) - D(c, lambda)) / sqrt(2 pi c), delta the
// Stirling series' error and D = c log(c / lambda) + lambda - c, near c =
// lambda by the series of log((1 + v) / (1 - v)), v = (c - lambda) / (c +
// lambda): the plain exponent loses lambda * 2^-53 to cancellation (1e-10 of
// the weight at lambda = 1e5).
__device__ inline double poisson_weight(int c, double lam) {
    if (!(lam > 0.0)) return c == 0 ? 1.0 : 0.0;
    const double x = (double)c;
    if (c < 16) return exp(-lam + x * log(lam) - lgamma(x + 1.0));
    const double i = 1.0 / x, i2 = i * i;
    const double delta = i * (1.0 / 12.0 - i2 * (1.0 / 360.0 - i2 * (1.0 / 1260.0 - i2 * (1.0 / 1680.0 - i2 / 1188.0))));
    const double d = x - lam, v = d / (x + lam);
    double D;
    if (fabs(v) < 0.1) {
        const double v2 = v * v;
        double s = 1.0 / 17.0;
        s = fma(s, v2, 1.0 / 15.0);
        s = fma(s, v2, 1.0 / 13.0);
        s = fma(s, v2, 1.0 / 11.0);
        s = fma(s, v2, 1.0 / 9.0);
        s = fma(s, v2, 1.0 / 7.0);
        s = fma(s, v2, 1.0 / 5.0);
        s = fma(s, v2, 1.0 / 3.0);
        D = d * v + 2.0 * x * v * v2 * s;
    } else {
        D = x * log(x / lam) - d;
    }
    return exp(-delta - D) * rsqrt(6.283185307179586477 * x);
}

}  // namespace mdlg
