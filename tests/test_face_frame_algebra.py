"""The sweep's face function in the frame of the interface, restated in NumPy
and checked against the oracle's Appendix A vectors and phi_N: projections on
g, h, k, Y_n with Y = X_m - v X_rho, the central flux left unprojected
(sum_m R_m L_m = identity), a_f and a_s from one root, the boost of the
back-projection, and the smoothness indicators as quadratics in one
difference."""
import numpy as np
import pytest

import oracle as ora
from test_face_algebra import GAMMA, random_states


def frame_scalars(w):
    r, vn, v1, v2, Bn, B1, B2, P = w
    gm1, g2 = GAMMA - 1.0, (GAMMA - 2.0) / (GAMMA - 1.0)
    isr = 1.0 / np.sqrt(r)
    cs2, ca2, btm = GAMMA * P * isr * isr, Bn * Bn * isr * isr, B1 * B1 + B2 * B2
    bt2 = btm * isr * isr
    q, aa = cs2 * bt2, ca2 + bt2 - cs2
    sd = np.sqrt(aa * aa + 4.0 * q)
    big, cs, bt = 0.5 * (sd + abs(aa)), np.sqrt(cs2), np.sqrt(btm)
    ab = np.sqrt(big / sd)
    sm = cs * bt * isr / (sd * ab)
    as_, af = (ab, sm) if aa >= 0 else (sm, ab)
    cf2 = cs2 + (big if aa >= 0 else sm * sm * sd)
    cf = np.sqrt(cf2)
    csl = cs * abs(Bn) * isr / cf
    return dict(vn=vn, v1=v1, v2=v2, hv2=0.5 * (vn * vn + v1 * v1 + v2 * v2), gm1=gm1, g2=g2, isr=isr, sr=r * isr, cs=cs,
                cs2=cs2, cf=cf, csl=csl, af=af, as_=as_, b1=B1 / bt, b2=B2 / bt, bt=bt, sg=1.0 if Bn >= 0 else -1.0)


def project(X, e):
    """Fields (fast -, fast +, slow -, slow +, Alfven -, Alfven + without their
    factor sg/2, entropy) of a 7-vector."""
    Yn, Y1, Y2 = X[1] - e["vn"] * X[0], X[2] - e["v1"] * X[0], X[3] - e["v2"] * X[0]
    b1, b2, sg, pre = e["b1"], e["b2"], e["sg"], 0.5 / e["cs2"]
    h, k, x = b1 * X[4] + b2 * X[5], b1 * Y1 + b2 * Y2, b1 * Y2 - b2 * Y1
    g = X[6] - e["hv2"] * X[0] - e["vn"] * Yn - e["v1"] * Y1 - e["v2"] * Y2 - e["bt"] * h
    afcf, ascl, sc = e["af"] * e["cf"], e["as_"] * e["csl"], e["sr"] * e["cs"]
    fc, fs = pre * (e["gm1"] * e["af"] * g + sc * e["as_"] * h), pre * (-afcf * Yn + sg * ascl * k)
    mc, ms = pre * (e["gm1"] * e["as_"] * g - sc * e["af"] * h), pre * (-ascl * Yn - sg * afcf * k)
    o = sg * e["sr"] * (b1 * X[5] - b2 * X[4])
    return fc + fs, fc - fs, mc + ms, mc - ms, x + o, x - o, X[0] - e["gm1"] / e["cs2"] * g


def back(F, e):
    sf, df, ss, ds, sa, da, Fe = F[0] + F[1], F[0] - F[1], F[2] + F[3], F[2] - F[3], F[4] + F[5], F[4] - F[5], F[6]
    af, as_, b1, b2, sg = e["af"], e["as_"], e["b1"], e["b2"], e["sg"]
    afcf, ascl = af * e["cf"], as_ * e["csl"]
    mg = af * sf + as_ * ss
    S1, S2 = mg + Fe, e["cs"] * e["isr"] * (as_ * sf - af * ss)
    hda = 0.5 * da * sg * e["isr"]
    Tn, Tk = -(afcf * df + ascl * ds), sg * (ascl * df - afcf * ds)
    T1, T2 = Tk * b1 - 0.5 * sa * b2, Tk * b2 + 0.5 * sa * b1
    return np.array([S1, S1 * e["vn"] + Tn, S1 * e["v1"] + T1, S1 * e["v2"] + T2, S2 * b1 - hda * b2, S2 * b2 + hda * b1,
                     e["hv2"] * S1 + e["vn"] * Tn + e["v1"] * T1 + e["v2"] * T2 + afcf * e["cf"] * sf
                     + ascl * e["csl"] * ss - e["g2"] * e["cs2"] * mg])


def test_frame_projection_and_back_projection_equal_the_eigenvectors():
    rng = np.random.default_rng(5)
    for w in random_states(200, 21):
        L, R, _ = ora.eigensystem(w, GAMMA)
        e = frame_scalars(w)
        X = rng.normal(size=7)
        want = L @ X
        got = project(X, e)
        half = 0.5 * e["sg"]
        got = np.array([got[0], half * got[4], got[2], got[6], got[3], half * got[5], got[1]])
        np.testing.assert_allclose(got, want, atol=1e-12 * np.abs(L).max())
        F = rng.normal(size=7)                # field fluxes in the kernel's units
        rows = [0, 6, 2, 4, 1, 5, 3]          # the oracle's rows of (fast -+, slow -+, Alfven -+, entropy)
        scale = [1, 1, 1, 1, half, half, 1]
        want = sum(F[i] * scale[i] * R[rows[i]] for i in range(7))
        np.testing.assert_allclose(back(F, e), want, atol=1e-12 * np.abs(R).max())
        # the identity that leaves the central flux unprojected
        np.testing.assert_allclose(back(project(X, e), e), X, atol=1e-12 * np.abs(R).max() * np.abs(L).max())


@pytest.mark.parametrize("variant", [0, 1])
def test_phi_from_one_difference_indicators(variant):
    """phi_N = N / (12 D) with s_k = (eps + IS_k) / 12 in the kernel's form."""
    cfg = ora.make_config(weno_variant=variant)
    eps = (1e-6 if variant == 0 else 1e-40) / 12.0
    rng = np.random.default_rng(6)
    for _ in range(500):
        a, b, c, d = rng.normal(size=4) * 10.0 ** rng.uniform(-3, 1, 4)
        x, y, z = a - b, b - c, c - d
        s = (x * (4 / 3 * x - b) + b * b + eps, y * (4 / 3 * y - b) + b * b + eps, z * (4 / 3 * z + c) + c * c + eps)
        p = (s[1] * s[2], s[0] * s[2], s[0] * s[1])
        Q, t = (s[0] * p[0]) ** 2, s[0] - s[2]
        W = [v * v if variant == 0 else Q + (t * v) ** 2 for v in p]
        Y = W[0] + 6 * W[1]
        N, D = 4 * W[0] * (x - y) + (3 * W[2] - Y) * (y - z), Y + 3 * W[2]
        assert abs(N / (12 * D) - ora.phi_n(a, b, c, d, cfg)) <= 1e-13 * max(map(abs, (a, b, c, d)))
