"""The node functions that the kernels run, compiled for the host
(tests/c/forms_host.cu), against the literal formulas: the source tensor from
displacement differences (one-sided at walls), the collision, and the wall rules
for every combination of walls and edge types.

Bounds: each result is a sum of at most 32 rounded operations (64 for the source
tensor, whose inputs are rounded too) on terms no larger than M, which every
test forms from absolute values; so it lies within 32 (64) rounding units of M.
"""
import os
import subprocess

import numpy as np
import pytest

from test_collision_identity import EX, EY, literal

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
OPP = (0, 3, 4, 1, 2, 7, 8, 5, 6)
W = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4)
LEFT, RIGHT, BOTTOM, TOP = range(4)
TYPE = {"periodic": 0, "dirichlet": 1, "neumann": 2}
EPS = {"double": 2.0 ** -53, "float": 2.0 ** -24}


@pytest.fixture(scope="module")
def forms(tmp_path_factory):
    from paper_2502_00920_gb300 import build
    exe = str(tmp_path_factory.mktemp("forms") / "forms_host")
    r = subprocess.run([build.nvcc(), *build.ARCH, *build.FLAGS, "-I", build.CSRC,
                        os.path.join(ROOT, "tests", "c", "forms_host.cu"), "-o", exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr

    def call(real, what, cases):
        text = "\n".join(" ".join(repr(float(v)) for v in c) for c in cases)
        r = subprocess.run([exe, real, what, str(len(cases))], input=text, capture_output=True, text=True, timeout=60)
        assert r.returncode == 0
        return np.array([[float(v) for v in line.split()] for line in r.stdout.splitlines()])

    return call


def as_real(x, real):
    """The inputs as the compute type holds them."""
    return np.asarray(x, dtype=np.float64 if real == "double" else np.float32).astype(np.float64)


@pytest.mark.parametrize("real", ["double", "float"])
@pytest.mark.parametrize("model", ["nh", "svk", "le"])
def test_source_tensor(forms, oracle_mod, model, real):
    rng = np.random.default_rng(1)
    cases, want, bound = [], [], []
    for strain in (1e-6, 1e-3, 0.1):
        for onex in (0, 1):
            for oney in (0, 1):
                for _ in range(20):
                    nu, dx = rng.uniform(0.0, 0.4), 1 / rng.uniform(10.0, 1000.0)
                    mu, lam = 1 / (2 * (1 + nu)), nu / ((1 + nu) * (1 - 2 * nu))
                    H = np.clip(rng.normal(0.0, strain, 4), -2 * strain, 2 * strain)  # H11, H12, H21, H22
                    sx, sy = dx if onex else 2 * dx, dx if oney else 2 * dx
                    D = as_real([H[0] * sx, H[2] * sx, H[1] * sy, H[3] * sy], real)  # dxx, dxy, dyx, dyy
                    H = np.array([D[0] / sx, D[2] / sy, D[1] / sx, D[3] / sy])
                    cases.append([dict(svk=0, nh=1, le=2)[model], lam, mu, dx, *D, onex, oney])
                    want.append(oracle_mod.first_piola(model, lam, mu, H).reshape(4)
                                + oracle_mod.pi_of_h(mu, H).reshape(4))
                    h = 2 * np.abs(H).max()
                    J = (1 + H[0]) * (1 + H[3]) - H[1] * H[2] if model == "nh" else 1.0
                    M = (lam + 2 * mu) * h * (1 + h) ** 2 / J
                    # (the oracle's own sum of P and Pi, which cancel, rounds relative to 1 + lam + mu)
                    bound.append(64 * EPS[real] * M + 1e-14 * (1 + lam + mu))
    got = forms(real, "stress", cases)
    assert got.shape == (len(cases), 4)
    assert (np.abs(got - np.array(want)) <= np.array(bound)[:, None]).all()


@pytest.mark.parametrize("real", ["double", "float"])
def test_collision(forms, oracle_mod, real):
    rng = np.random.default_rng(2)
    cases, want, bound = [], [], []
    for _ in range(200):
        f, S = as_real(rng.normal(0.0, 0.1, 9), real), as_real(rng.normal(0.0, 1.0, 2), real)
        cs, tau, dt = rng.uniform(0.3, 1.5), rng.uniform(0.51, 1.5), rng.uniform(0.01, 0.1)
        sigma = np.sqrt(3.0) * cs * dt / cs ** 2
        cases.append([1 / tau, sigma, *f, *S])
        want.append(literal(oracle_mod, f, S, cs, tau, dt))
        # the even relaxation's sum of all populations has weights up to 4, times omega / 9
        bound.append(32 * EPS[real] * (4 * np.abs(f).sum() + sigma * np.abs(S).sum()) + 1e-15)
    got = forms(real, "collision", cases)
    assert got.shape == (len(cases), 9)
    assert (np.abs(got - np.array(want)) <= np.array(bound)[:, None]).all()


def wall_rule(q, xw, yw, kind, T, cs, wn, g):
    """(value, M) of population q at a node on the walls xw, yw (-1: none) by
    Eq. bbcon and abbcon, None where nothing is replaced: the link opp(q)
    crosses a wall where q's source lies beyond it."""
    c = np.sqrt(3.0) * cs
    ax = xw if xw >= 0 and EX[q] == (1 if xw == LEFT else -1) else None
    ay = yw if yw >= 0 and EY[q] == (1 if yw == BOTTOM else -1) else None
    crossed = [w for w in (ax, ay) if w is not None]
    if not crossed:
        return None
    clamped = [w for w in crossed if kind[w] == TYPE["dirichlet"]]
    if clamped:
        j = sum(T[w] for w in clamped) / len(clamped)
        k = 2 / cs ** 2 * W[q] * c
        return g[OPP[q]] + k * (EX[q] * j[0] + EY[q] * j[1]), abs(g[OPP[q]]) + k * np.abs(j).sum()
    pxx, pxy, pyy = (c * c * (e * g).sum() for e in (EX * EX, EX * EY, EY * EY))
    mxx = mxy = myy = c * c * np.abs(g).sum()
    shear = []
    if ax is not None:
        s = 1.0 if ax == RIGHT else -1.0
        pxx, mxx = wn[0] - s * T[ax][0], abs(wn[0]) + abs(T[ax][0])
        shear.append((wn[1] - s * T[ax][1], abs(wn[1]) + abs(T[ax][1])))
    if ay is not None:
        s = 1.0 if ay == TOP else -1.0
        pyy, myy = wn[2] - s * T[ay][1], abs(wn[2]) + abs(T[ay][1])
        shear.append((wn[3] - s * T[ay][0], abs(wn[3]) + abs(T[ay][0])))
    pxy, mxy = np.mean(shear, axis=0)
    r, cs2 = g.sum(), cs ** 2
    cx, cy = c * EX[q], c * EY[q]
    contr = (pxx - r * cs2) * (cx * cx - cs2) + 2 * pxy * (cx * cy) + (pyy - r * cs2) * (cy * cy - cs2)
    M = abs(g[OPP[q]]) + 2 * W[q] * (7 * np.abs(g).sum() + (3 * mxx + 6 * mxy + 3 * myy) / cs2)
    return -g[OPP[q]] + 2 * W[q] * (r + contr / (2 * cs2 * cs2)), M


@pytest.mark.parametrize("real", ["double", "float"])
def test_wall_rules(forms, real):
    rng = np.random.default_rng(3)
    cases, want, bound = [], [], []
    for xw in (-1, LEFT, RIGHT):
        for yw in (-1, BOTTOM, TOP):
            if xw < 0 and yw < 0:
                continue
            for kx in ("dirichlet", "neumann") if xw >= 0 else ("periodic",):
                for ky in ("dirichlet", "neumann") if yw >= 0 else ("periodic",):
                    kind = [TYPE[kx]] * 2 + [TYPE[ky]] * 2
                    for _ in range(8):
                        cs = rng.uniform(0.3, 1.5)
                        T, wn, g = (as_real(rng.normal(0.0, 0.1, n), real) for n in ((4, 2), 4, 9))
                        cases.append([xw, yw, *kind, *T.ravel(), 1 / cs ** 2, np.sqrt(3.0) / cs, *wn, *g])
                        rules = [wall_rule(q, xw, yw, kind, T, cs, wn, g) for q in range(9)]
                        want.append([0.0 if r is None else r[0] for r in rules])
                        bound.append([0.0 if r is None else 32 * EPS[real] * r[1] + 1e-15 for r in rules])
    got = forms(real, "walls", cases)
    assert got.shape == (len(cases), 9)
    assert (np.abs(got - np.array(want)) <= np.array(bound)).all()
    assert (np.array(bound) > 0).any(axis=1).all()


@pytest.mark.parametrize("dx", [2.0 ** -530, 1e-150, 1e-100, 1e100, 1e150, 2.0 ** 530])
def test_neo_hooke_at_any_spacing(forms, oracle_mod, dx):
    """The double-precision form squares 1 / (2 dx) where that stays in range."""
    rng = np.random.default_rng(4)
    mu, lam = 0.4, 0.3
    H = rng.normal(0.0, 0.05, (20, 4))
    got = forms("double", "stress", [[1, lam, mu, dx, *(np.array([h[0], h[2], h[1], h[3]]) * 2 * dx), 0, 0] for h in H])
    for h, n in zip(H, got):
        want = oracle_mod.first_piola("nh", lam, mu, h).reshape(4) + oracle_mod.pi_of_h(mu, h).reshape(4)
        m = 2 * np.abs(h).max()
        J = (1 + h[0]) * (1 + h[3]) - h[1] * h[2]
        assert np.abs(n - want).max() <= 64 * EPS["double"] * (lam + 2 * mu) * m * (1 + m) ** 2 / J + 1e-14 * (1 + lam + mu)
