"""The double-precision kernels' forms of the collision's odd part and of the
neo-Hooke source tensor, restated on the host: both equal the literal formulas
of the oracle (Alg. 1 collision; N = P(H) + Pi(H)) to double rounding.  The GPU
parity tests compare the kernels themselves with the oracle."""
import math

import numpy as np
import pytest

from test_collision_identity import literal


def collide(f, S, cs, tau, dt):
    c = math.sqrt(3.0) * cs
    omega, s9 = 1.0 / tau, c * dt / cs ** 2 / 9
    d13, d24, d57, d68 = f[1] - f[3], f[2] - f[4], f[5] - f[7], f[6] - f[8]
    Q = f[0] - 2 * ((f[1] + f[3]) + (f[2] + f[4])) + 4 * ((f[5] + f[7]) + (f[6] + f[8]))
    X, Y = s9 * S[0], s9 * S[1]
    tx, ty = d13 - 2 * (d57 - d68), d24 - 2 * (d57 + d68)
    bx, by = X - omega / 6 * tx, Y - omega / 6 * ty
    cx, cy = X + omega / 3 * tx, Y + omega / 3 * ty
    b57, b68 = 0.25 * (cx + cy), 0.25 * (cy - cx)
    A1, A5 = Q * omega / 18, -Q * omega / 36
    return np.array([f[0] - omega / 9 * Q, f[1] + A1 + bx, f[2] + A1 + by, f[3] + A1 - bx, f[4] + A1 - by,
                     f[5] + A5 + b57, f[6] + A5 + b68, f[7] + A5 - b57, f[8] + A5 - b68])


@pytest.mark.parametrize("seed", range(20))
def test_collision_form(oracle_mod, seed):
    rng = np.random.default_rng(seed)
    f, S = rng.normal(0.0, 0.1, 9), rng.normal(0.0, 1.0, 2)
    cs, tau, dt = rng.uniform(0.3, 1.5), rng.uniform(0.51, 1.5), rng.uniform(0.01, 0.1)
    ref = literal(oracle_mod, f, S, cs, tau, dt)
    assert np.abs(collide(f, S, cs, tau, dt) - ref).max() <= 1e-14 * max(1.0, np.abs(ref).max())


@pytest.mark.parametrize("strain", [1e-6, 1e-3, 0.2])
def test_neo_hooke_from_differences(oracle_mod, strain):
    rng = np.random.default_rng(1)
    for _ in range(50):
        nu, h = rng.uniform(0.0, 0.4), rng.uniform(10.0, 1000.0)
        mu, lam = 1 / (2 * (1 + nu)), nu / ((1 + nu) * (1 - 2 * nu))
        H = rng.normal(0.0, strain, 4)
        dxx, dyx, dxy, dyy = H / h
        trH = h * (dxx + dyy)
        a = h * h * (dxx * dyy - dyx * dxy) + trH
        m = mu / (1 + a)
        ma, q = m * a, m * (2 + a)
        k = 0.5 * lam / mu * a * q
        d, mah, kh = k + (ma - q * trH), h * ma, h * k
        N = np.array([d + kh * dyy - mah * dxx, -(mah + kh) * dxy, -(mah + kh) * dyx, d + kh * dxx - mah * dyy])
        ref = oracle_mod.first_piola("nh", lam, mu, H).reshape(4) + oracle_mod.pi_of_h(mu, H).reshape(4)
        # the oracle's P and Pi cancel: its rounding is relative to mu |H|
        assert np.abs(N - ref).max() <= 1e-14 * (1 + abs(lam) + mu)
