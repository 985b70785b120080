// Small dense kernels of the local frames (Sec. 2): the symmetric 3x3
// eigenproblem of a neighbourhood's covariance.
#pragma once

#include <cuda_runtime.h>

namespace mvgd {

// Cyclic Jacobi on a symmetric 3x3 matrix (a, upper part used).  Columns of v
// are the eigenvectors, w the eigenvalues.
__device__ inline void jacobi3(double a[3][3], double v[3][3], double w[3]) {
    for (int r = 0; r < 3; r++)
        for (int c = 0; c < 3; c++) v[r][c] = (r == c) ? 1.0 : 0.0;
    for (int sweep = 0; sweep < 32; sweep++) {
        double off = a[0][1] * a[0][1] + a[0][2] * a[0][2] + a[1][2] * a[1][2];
        double dia = a[0][0] * a[0][0] + a[1][1] * a[1][1] + a[2][2] * a[2][2];
        if (!(off > 1e-40 * dia)) break;
#pragma unroll
        for (int pq = 0; pq < 3; pq++) {
            const int p = pq == 2 ? 1 : 0;
            const int q = pq == 0 ? 1 : 2;
            double apq = a[p][q];
            if (apq == 0.0) continue;
            double tau = (a[q][q] - a[p][p]) / (2.0 * apq);
            double t = copysign(1.0, tau) / (fabs(tau) + sqrt(1.0 + tau * tau));
            double c = rsqrt(1.0 + t * t);
            double s = t * c;
#pragma unroll
            for (int k = 0; k < 3; k++) {
                double akp = a[k][p], akq = a[k][q];
                a[k][p] = c * akp - s * akq;
                a[k][q] = s * akp + c * akq;
            }
#pragma unroll
            for (int k = 0; k < 3; k++) {
                double apk = a[p][k], aqk = a[q][k];
                a[p][k] = c * apk - s * aqk;
                a[q][k] = s * apk + c * aqk;
            }
#pragma unroll
            for (int k = 0; k < 3; k++) {
                double vkp = v[k][p], vkq = v[k][q];
                v[k][p] = c * vkp - s * vkq;
                v[k][q] = s * vkp + c * vkq;
            }
        }
    }
    w[0] = a[0][0];
    w[1] = a[1][1];
    w[2] = a[2][2];
}

// The same cyclic Jacobi in FP32, stopped at FP32 accuracy: the starting
// frame that one or two FP64 sweeps then polish (the FP32 assembly path).
__device__ inline void jacobi3f(float a[3][3], float v[3][3], float w[3]) {
    for (int r = 0; r < 3; r++)
        for (int c = 0; c < 3; c++) v[r][c] = (r == c) ? 1.0f : 0.0f;
    for (int sweep = 0; sweep < 16; sweep++) {
        const float off = a[0][1] * a[0][1] + a[0][2] * a[0][2] + a[1][2] * a[1][2];
        const float dia = a[0][0] * a[0][0] + a[1][1] * a[1][1] + a[2][2] * a[2][2];
        if (!(off > 1e-14f * dia)) break;
#pragma unroll
        for (int pq = 0; pq < 3; pq++) {
            const int p = pq == 2 ? 1 : 0;
            const int q = pq == 0 ? 1 : 2;
            const float apq = a[p][q];
            if (apq == 0.0f) continue;
            const float tau = (a[q][q] - a[p][p]) / (2.0f * apq);
            const float t = copysignf(1.0f, tau) / (fabsf(tau) + sqrtf(1.0f + tau * tau));
            const float c = rsqrtf(1.0f + t * t);
            const float s = t * c;
#pragma unroll
            for (int k = 0; k < 3; k++) {
                const float akp = a[k][p], akq = a[k][q];
                a[k][p] = c * akp - s * akq;
                a[k][q] = s * akp + c * akq;
            }
#pragma unroll
            for (int k = 0; k < 3; k++) {
                const float apk = a[p][k], aqk = a[q][k];
                a[p][k] = c * apk - s * aqk;
                a[q][k] = s * apk + c * aqk;
            }
#pragma unroll
            for (int k = 0; k < 3; k++) {
                const float vkp = v[k][p], vkq = v[k][q];
                v[k][p] = c * vkp - s * vkq;
                v[k][q] = s * vkp + c * vkq;
            }
        }
    }
    w[0] = a[0][0];
    w[1] = a[1][1];
    w[2] = a[2][2];
}

// FP32 tangent of the Jacobi rotation that annihilates apq (d = aqq - app).
__device__ __forceinline__ float jacobi_tan(float apq, float d) {
    if (apq == 0.0f) return 0.0f;
    const float tau = __fdividef(d, 2.0f * apq), u = fabsf(tau);
    const float t = u > 1e9f ? __fdividef(0.5f, u) : __fdividef(1.0f, u + sqrtf(fmaf(u, u, 1.0f)));
    return copysignf(t, tau);
}

// Eigenvectors (columns of e) of a symmetric 3x3 matrix to FP64 accuracy, w the
// eigenvalues (for their order; c is overwritten).  A plain FP64 Jacobi takes five
// or six sweeps and spends most of their instructions in divisions and square
// roots on the FP64 pipe (one instruction in 16 clocks a warp).  Here the sweeps
// that only find the frame run in FP32; its vectors are orthonormalised in FP64,
// the matrix is rotated into them, and FP64 rotations finish.  A rotation need
// not annihilate exactly, it must only be orthogonal: its tangent comes from FP32,
// its cosine from an FP32 root with one cubic Newton step, so an off-diagonal entry
// shrinks by 1e-7 a sweep beside Jacobi's own quadratic rate.  Once the remaining angles are below 2^-27 one first-order
// update is exact to about 2^-49 of a radian.  For general inputs the entries are
// scaled by a power of two first.
__device__ inline void eig3(double (&c)[3][3], double (&e)[3][3], double (&w)[3]) {
    {
        const double m = fmax(fabs(c[0][0]), fmax(fabs(c[1][1]), fabs(c[2][2])));
        const int ex = (__double2hiint(m) >> 20) & 0x7ff;
        if (ex > 0 && ex < 0x7fe) {
            const double sc = __hiloint2double((2046 - ex) << 20, 0);
#pragma unroll
            for (int r = 0; r < 3; r++)
#pragma unroll
                for (int q = r; q < 3; q++) c[q][r] = c[r][q] *= sc;
        }
    }
    float cf[3][3], vf[3][3], wf[3];
#pragma unroll
    for (int r = 0; r < 3; r++)
#pragma unroll
        for (int q = 0; q < 3; q++) cf[r][q] = (float)c[r < q ? r : q][r < q ? q : r];
    jacobi3f(cf, vf, wf);
#pragma unroll
    for (int r = 0; r < 3; r++)
#pragma unroll
        for (int q = 0; q < 2; q++) e[r][q] = (double)vf[r][q];
    // the FP32 vectors have unit length to about 1e-6: 1 / sqrt(1 + x) by its series
    auto unit = [&](int q) {
        const double x = fma(e[0][q], e[0][q], fma(e[1][q], e[1][q], e[2][q] * e[2][q])) - 1.0;
        const double s = fma(x, fma(x, fma(x, -0.3125, 0.375), -0.5), 1.0);
#pragma unroll
        for (int r = 0; r < 3; r++) e[r][q] *= s;
    };
    unit(0);
    const double d01 = fma(e[0][0], e[0][1], fma(e[1][0], e[1][1], e[2][0] * e[2][1]));
#pragma unroll
    for (int r = 0; r < 3; r++) e[r][1] = fma(-d01, e[r][0], e[r][1]);
    unit(1);
    e[0][2] = fma(e[1][0], e[2][1], -(e[2][0] * e[1][1]));
    e[1][2] = fma(e[2][0], e[0][1], -(e[0][0] * e[2][1]));
    e[2][2] = fma(e[0][0], e[1][1], -(e[1][0] * e[0][1]));
    double a[3][3];  // upper part of e^T c e
    {
        double t[3][3];
#pragma unroll
        for (int r = 0; r < 3; r++)
#pragma unroll
            for (int q = 0; q < 3; q++) t[r][q] = fma(c[r][0], e[0][q], fma(c[r][1], e[1][q], c[r][2] * e[2][q]));
#pragma unroll
        for (int r = 0; r < 3; r++)
#pragma unroll
            for (int q = r; q < 3; q++) a[r][q] = fma(e[0][r], t[0][q], fma(e[1][r], t[1][q], e[2][r] * t[2][q]));
    }
#pragma unroll 1
    for (int sweep = 0; sweep < 16; sweep++) {
        const float t01 = jacobi_tan((float)a[0][1], (float)(a[1][1] - a[0][0]));
        const float t02 = jacobi_tan((float)a[0][2], (float)(a[2][2] - a[0][0]));
        const float t12 = jacobi_tan((float)a[1][2], (float)(a[2][2] - a[1][1]));
        if (!(fmaxf(fabsf(t01), fmaxf(fabsf(t02), fabsf(t12))) >= 0x1p-27f)) {
            const double x = (double)t01, y = (double)t02, z = (double)t12;
#pragma unroll
            for (int r = 0; r < 3; r++) {
                const double e0 = e[r][0], e1 = e[r][1], e2 = e[r][2];
                e[r][0] = fma(-x, e1, fma(-y, e2, e0));
                e[r][1] = fma(x, e0, fma(-z, e2, e1));
                e[r][2] = fma(y, e0, fma(z, e1, e2));
            }
            break;
        }
#pragma unroll
        for (int pq = 0; pq < 3; pq++) {
            const int p = pq == 2 ? 1 : 0, q = pq == 0 ? 1 : 2, o = 3 - p - q;
            const double d = a[q][q] - a[p][p];
            const float tf = pq == 0 ? t01 : jacobi_tan((float)a[p][q], (float)d);
            const double t = (double)tf, x = fma(t, t, 1.0);
            const double y0 = (double)rsqrtf(fmaf(tf, tf, 1.0f));
            const double h = fma(-x * y0, y0, 1.0);
            const double cs = fma(y0 * h, fma(0.375, h, 0.5), y0), sn = t * cs;
            const double apq = a[p][q], m = fma(sn, d, -(cs + cs) * apq), g = fma(cs, d, (sn + sn) * apq);
            a[p][p] = fma(sn, m, a[p][p]);
            a[q][q] = fma(-sn, m, a[q][q]);
            a[p][q] = fma(-sn, g, apq);
            double& ap = p < o ? a[p][o] : a[o][p];
            double& aq = q < o ? a[q][o] : a[o][q];
            const double bp = ap, bq = aq;
            ap = fma(cs, bp, -(sn * bq));
            aq = fma(sn, bp, cs * bq);
#pragma unroll
            for (int r = 0; r < 3; r++) {
                const double ep = e[r][p], eq = e[r][q];
                e[r][p] = fma(cs, ep, -(sn * eq));
                e[r][q] = fma(sn, ep, cs * eq);
            }
        }
    }
    w[0] = a[0][0];
    w[1] = a[1][1];
    w[2] = a[2][2];
}

}  // namespace mvgd
