// Per-pair derivative sums and the assembly of a sample's gradient (adjoint.cu, treeadj.cu).
#pragma once

#include "isw_internal.cuh"
#include "pipeline.cuh"

namespace isw {

constexpr int kAcc = 13;
// sums in use: those after the tenth are for dL/dX'
__host__ __device__ constexpr int adj_rows(bool ng9) { return ng9 ? kAcc : 10; }

// Per-pair derivative sums.  With d = n - Xhat, Q = d.d, u = Xdot - (A/B) X', T = u.d / Q and
// eta = 2T/Q, the n-dependent parts of the three gradients are accumulated as vectors along d
// (and n where d does not appear): sums along n and Xhat separately differ by O(1/|d|) from their
// combination and lose that factor of precision for pixels close to the sample.
//   acc[0] = sum g uX/Q (uX = u.Xhat)   acc[1] = sum g/Q   acc[2] = sum g A/(BQ)   acc[3] = sum g T
//   acc[4..6]   = sum g eta d
//   acc[7..9]   = sum g/Q (d + (A Qd/B^2) n)
//   acc[10..12] = sum g/(BQ) (A d + Qd n)       (Qd = X'.d, Pd = Xdot.d)
// FP64 version (the FP64 kernel and the FP32 kernel's near field)
__device__ __forceinline__ void adj_pair64(double nx, double ny, double nz, double g, const Seg64 &s, int ngrad,
                                           double *acc, unsigned &zero)
{
    const double dx = (nx - s.xh[0]) - s.xl[0];
    const double dy = (ny - s.xh[1]) - s.xl[1];
    const double dz = (nz - s.xh[2]) - s.xl[2];
    const double Q = dx * dx + dy * dy + dz * dz;
    if (Q == 0.0) {
        ++zero;
        return;
    }
    const double A = nx * s.xp[0] + ny * s.xp[1] + nz * s.xp[2];
    const double B = 1.0 + (nx * s.xd[0] + ny * s.xd[1] + nz * s.xd[2]);
    const double Pd = s.xd[0] * dx + s.xd[1] * dy + s.xd[2] * dz;
    const double Qd = s.xp[0] * dx + s.xp[1] * dy + s.xp[2] * dz;
    const double iQ = rcp64(Q), iB = rcp64(B);
    const double AB = A * iB;
    const double uX = (s.xd[0] * s.xh[0] + s.xd[1] * s.xh[1] + s.xd[2] * s.xh[2]) -
                      AB * (s.xp[0] * s.xh[0] + s.xp[1] * s.xh[1] + s.xp[2] * s.xh[2]);
    const double T = (Pd - AB * Qd) * iQ;
    const double gq = g * iQ;
    acc[0] += gq * uX;
    acc[1] += gq;
    acc[2] += gq * AB;
    acc[3] += g * T;
    const double ge = 2.0 * g * T * iQ;
    acc[4] += ge * dx;
    acc[5] += ge * dy;
    acc[6] += ge * dz;
    const double v = gq * AB * Qd * iB;
    acc[7] += gq * dx + v * nx;
    acc[8] += gq * dy + v * ny;
    acc[9] += gq * dz + v * nz;
    if (ngrad >= 9) {
        const double gb = gq * iB;
        const double ga = gb * A, gd = gb * Qd;
        acc[10] += ga * dx + gd * nx;
        acc[11] += ga * dy + gd * ny;
        acc[12] += ga * dz + gd * nz;
    }
}

// Gradient rows of one sample from its sums (FP64).  With c = -4 GU eps dsigma / |X| and
// eps = sqrt(X'^2 / (1 - Xdot^2)):
//   dTheta/dX     = (c/|X|) [eta d - (u - Xhat uX)/Q]    (c/|X| from dc/dX and the projection
//                                                          of d(Xhat)/dX; the Xhat T terms cancel)
//   dTheta/dXdot  = c [T Xdot / (1 - Xdot^2) + (d + (A Qd/B^2) n)/Q]
//   dTheta/dX'    = c [T X' / X'^2 - (A d + Qd n)/(BQ)]
//   dTheta/ddsigma = (c / dsigma) T = cu T                  (the term is linear in dsigma)
// Rows: X (3), Xdot (3), then X' (3) when ngrad >= 9 and dsigma when ngrad == 10.
__device__ __forceinline__ void adj_assemble(const Seg64 &s, const double *acc, int ngrad, double *out)
{
    const double cX = s.c / s.X;
    const double om2 = s.om * (2.0 - s.om);   // 1 - |Xdot|^2 = (1 - v)(1 + v)
    const double xp2 = s.xp[0] * s.xp[0] + s.xp[1] * s.xp[1] + s.xp[2] * s.xp[2];
    for (int k = 0; k < 3; ++k) {
        const double xh = s.xh[k] + s.xl[k];
        out[k] = cX * (acc[0] * xh - acc[1] * s.xd[k] + acc[2] * s.xp[k] + acc[4 + k]);
        out[3 + k] = s.c * (acc[3] / om2 * s.xd[k] + acc[7 + k]);
        if (ngrad >= 9) out[6 + k] = s.c * ((xp2 > 0.0 ? acc[3] / xp2 : 0.0) * s.xp[k] - acc[10 + k]);
    }
    if (ngrad == 10) out[9] = s.cu * acc[3];
}

}  // namespace isw
