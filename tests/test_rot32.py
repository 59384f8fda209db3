"""The rotation sub-steps in FP32 pairs (csrc/dem_rot32.cuh), compiled for the
host, against 128-bit arithmetic: no further from it than the same sub-steps in
FP64, over random bodies (spheres and symmetric ones among them), 8 to 400
sub-steps, angular velocities and torques from rest to the limits of
rot32_applies.

Bound: FP64's own error, or 6e-16 where that is smaller: the result is put
together in FP64 (four products and sums of the quaternion, three of the
angular velocity, 2^-53 each), and the pairs' share is below that."""
import os
import platform
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2206_11634_gb300", "csrc")

HARNESS = r"""
#include <cmath>
#include <cstdio>
#include <random>
#include "dem_rot32.cuh"
using namespace lbmmb;
#if defined(__aarch64__)
typedef long double Quad;  // 128 bits there
#else
typedef __float128 Quad;
#endif

// the sub-steps in type T, sine and cosine by their series
template <class T>
void scheme(T q[4], T w[3], T Tb[3], const T cI[3], const T iI[3], T h, int n) {
    const T hh = h / 2;
    for (int k = 0; k < n; k++) {
        T wh[3], s[3], X[3], Y[3], t[3], v[3], c = 1, sc = 1, tc = 1, ts = 1, a2 = 0;
        for (int l = 0; l < 3; l++) {
            wh[l] = w[l] + hh * (cI[l] * w[(l + 1) % 3] * w[(l + 2) % 3] + iI[l] * Tb[l]);
            a2 += hh * hh * wh[l] * wh[l];
        }
        for (int j = 1; j < 14; j++) {
            tc *= -a2 / ((2 * j - 1) * (2 * j));
            ts *= -a2 / ((2 * j) * (2 * j + 1));
            c += tc;
            sc += ts;
        }
        for (int l = 0; l < 3; l++) s[l] = hh * sc * wh[l];
        for (int l = 0; l < 3; l++) X[l] = s[(l + 1) % 3] * Tb[(l + 2) % 3] - s[(l + 2) % 3] * Tb[(l + 1) % 3];
        for (int l = 0; l < 3; l++) Y[l] = s[(l + 1) % 3] * X[(l + 2) % 3] - s[(l + 2) % 3] * X[(l + 1) % 3];
        for (int l = 0; l < 3; l++) Tb[l] += -2 * c * X[l] + 2 * Y[l];
        for (int l = 0; l < 3; l++) t[l] = wh[l] + hh * iI[l] * Tb[l];
        for (int l = 0; l < 3; l++) v[l] = t[l] + hh * cI[l] * wh[(l + 1) % 3] * wh[(l + 2) % 3];
        for (int l = 0; l < 3; l++) w[l] = t[l] + hh * cI[l] * v[(l + 1) % 3] * v[(l + 2) % 3];
        const T r[4] = {q[0] * c - q[1] * s[0] - q[2] * s[1] - q[3] * s[2],
                        q[0] * s[0] + q[1] * c + q[2] * s[2] - q[3] * s[1],
                        q[0] * s[1] - q[1] * s[2] + q[2] * c + q[3] * s[0],
                        q[0] * s[2] + q[1] * s[1] - q[2] * s[0] + q[3] * c};
        for (int i = 0; i < 4; i++) q[i] = r[i];
    }
}
template <class A, class B> double apart(const A *a, const B *b, int n) {
    double e = 0;
    for (int i = 0; i < n; i++) e += std::pow((double)((Quad)a[i] - (Quad)b[i]), 2);
    return std::sqrt(e);
}

int main() {
    std::mt19937_64 g(7);
    std::uniform_real_distribution<double> U(-1, 1), V(0, 1);
    for (int n : {8, 10, 33, 100, 400})
        for (int reg = 0; reg < 6; reg++) {
            double e64[2] = {0, 0}, e32[2] = {0, 0};
            int taken = 0;
            for (int it = 0; it < 300; it++) {
                double m[3] = {1 + 2 * V(g), 1 + 2 * V(g), 0};
                m[2] = std::fabs(m[0] - m[1]) + (m[0] + m[1] - std::fabs(m[0] - m[1])) * V(g);
                if (it % 7 == 0) m[1] = m[2] = m[0];
                if (it % 7 == 1) m[1] = m[0];
                const double scale = std::pow(10, 2 + 2 * V(g)), h = 1.0 / n, hh = h / 2;
                double iI[3], cI[3], imax = 0, cmax = 0;
                for (int l = 0; l < 3; l++) iI[l] = 1 / (m[l] * scale);
                for (int l = 0; l < 3; l++) cI[l] = (m[(l + 1) % 3] - m[(l + 2) % 3]) / m[l];
                for (int l = 0; l < 3; l++) {
                    imax = std::fmax(imax, iI[l]);
                    cmax = std::fmax(cmax, std::fabs(cI[l]));
                }
                const double top = std::fmin(std::ldexp(1, -16) / hh, std::ldexp(1, -9) / (hh * n));
                double W = 0, D = 0;  // angular velocity, and its change by the torque
                if (reg == 0) W = D = 0.45 * top;
                if (reg == 1) D = 0.95 * top;
                if (reg == 2) W = 0.95 * top;
                if (reg == 3) W = 1e-3 * top, D = 0.5 * top;
                if (reg == 4) W = 0.5 * top, D = 1e-3 * top;
                if (reg == 5) W = 1e-6 * std::pow(10, 3 * V(g)), D = 1e-7 * std::pow(10, 3 * V(g));
                double w0[3], T0[3], q0[4], nw = 0, nt = 0, nq = 0;
                for (int l = 0; l < 3; l++) {
                    w0[l] = U(g); T0[l] = U(g);
                    nw += w0[l] * w0[l]; nt += T0[l] * T0[l];
                }
                for (int i = 0; i < 4; i++) { q0[i] = U(g); nq += q0[i] * q0[i]; }
                for (int l = 0; l < 3; l++) { w0[l] *= W / std::sqrt(nw); T0[l] *= D / (std::sqrt(nt) * imax); }
                for (int i = 0; i < 4; i++) q0[i] /= std::sqrt(nq);
                if (!rot32_applies((float)(hh * (W + D)), n, (float)cmax)) continue;
                Rot32 R;
                for (int l = 0; l < 3; l++) {
                    R.cI[l] = rot_split(cI[l]);
                    R.iI[l] = rot_split(iI[l]);
                    R.U0[l] = rot_split(hh * w0[l]);
                    R.t0[l] = rot_split(hh * hh * T0[l]);
                    R.G0[l] = rot_split(hh * hh * T0[l] * iI[l]);
                }
                const Rot32Result r = rot32_run(R, n);
                if (!r.ok) continue;
                taken++;
                double b[3], b2 = 0, w[3];
                for (int l = 0; l < 3; l++) {
                    b[l] = (double)r.beta[l].h + (double)r.beta[l].l;
                    b2 += b[l] * b[l];
                    w[l] = std::fma(2.0 * n, (double)r.delta[l].h + (double)r.delta[l].l, std::fma(iI[l], T0[l], w0[l]));
                }
                const double d = 1.0 - b2 * (0.5 + b2 * (0.125 + b2 * (0.0625 + b2 * 5.0 / 128.0)));
                const double q[4] = {q0[0] * d - q0[1] * b[0] - q0[2] * b[1] - q0[3] * b[2],
                                     q0[0] * b[0] + q0[1] * d + q0[2] * b[2] - q0[3] * b[1],
                                     q0[0] * b[1] - q0[1] * b[2] + q0[2] * d + q0[3] * b[0],
                                     q0[0] * b[2] + q0[1] * b[1] - q0[2] * b[0] + q0[3] * d};
                Quad qx[4], wx[3], tx[3], cx[3], ix[3];
                double qd[4], wd[3], td[3];
                for (int i = 0; i < 4; i++) qx[i] = qd[i] = q0[i];
                for (int l = 0; l < 3; l++) {
                    wx[l] = wd[l] = w0[l];
                    tx[l] = td[l] = T0[l];
                    cx[l] = cI[l];
                    ix[l] = iI[l];
                }
                scheme<Quad>(qx, wx, tx, cx, ix, Quad(1) / n, n);
                scheme<double>(qd, wd, td, cI, iI, h, n);
                double nx = 0;
                for (int l = 0; l < 3; l++) nx += (double)(wx[l] * wx[l]);
                e64[0] = std::fmax(e64[0], apart(qd, qx, 4));
                e32[0] = std::fmax(e32[0], apart(q, qx, 4));
                e64[1] = std::fmax(e64[1], apart(wd, wx, 3) / std::sqrt(nx));
                e32[1] = std::fmax(e32[1], apart(w, wx, 3) / std::sqrt(nx));
            }
            std::printf("%d %d %d %.3e %.3e %.3e %.3e\n", n, reg, taken, e64[0], e32[0], e64[1], e32[1]);
        }
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs g++")
def test_pairs_are_as_accurate_as_fp64(tmp_path):
    assert platform.machine() in ("x86_64", "aarch64")
    src = tmp_path / "rot32.cpp"
    src.write_text(HARNESS)
    exe = tmp_path / "rot32"
    subprocess.run(["g++", "-O1", "-std=gnu++17", "-ffp-contract=off", "-Wno-unknown-pragmas", "-I", CSRC, str(src),
                    "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout
    rows = [line.split() for line in out.splitlines()]
    assert len(rows) == 30
    for n, reg, taken, q64, q32, w64, w32 in rows:
        if reg != "5" or int(n) >= 100:
            assert int(taken) > 250, (n, reg, taken)
        assert float(q32) <= max(float(q64), 6e-16), (n, reg, q64, q32)
        assert float(w32) <= max(float(w64), 6e-16), (n, reg, w64, w32)
