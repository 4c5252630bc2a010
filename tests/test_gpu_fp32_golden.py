"""Single-precision fields against recorded values (tests/golden/fp32_fields.txt), in cells that amplify a rounding: a
dilute, boosted fringe, where the time derivative of u~^tau is a difference of nearly equal numbers and enters pi~^{00}
times gamma^2.  There the same sums in another order move a field by 3e-4 to 7e-3 of its largest value within six steps.

Tolerance: 16 roundings of the field's largest value, 16 x 2^-24 = 1e-6 of it.
Inputs are sums and products only (no library functions), so that every machine has the same."""
import os

import numpy as np
import pytest

from paper_1802_04449_gb300 import clv
from paper_1802_04449_gb300 import inputs as I

pytestmark = pytest.mark.gpu

GOLDEN = os.path.join(os.path.dirname(__file__), "golden", "fp32_fields.txt")
FIELDS = clv.FIELDS[:18]
CASES = ["minijet", "minijet_conformal", "flow", "options", "lambda1", "direct", "batch"]


def _numbers(seed, n, lo, hi):
    """n numbers in [lo, hi) from a linear congruential generator."""
    out, x = [], 2 * seed + 1
    for _ in range(n):
        x = (x * 6364136223846793005 + 1442695040888963407) % 2 ** 64
        out.append(lo + (hi - lo) * ((x >> 40) / 2 ** 24))
    return np.array(out)


def _grid(shape, d):
    return np.meshgrid(*((np.arange(n) - (n - 1) / 2) * a for n, a in zip(shape, d)), indexing="ij")


def _spots(shape, d, seed, n):
    """Energy density of n spots (steep power-law tails) and two more sums of them, weighted by velocities below 1."""
    X, Y, Z = _grid(shape, d)
    half = [a * (m - 1) / 2 for m, a in zip(shape, d)]
    x, y, z = (_numbers(seed + k, n, -0.9 * half[k], 0.9 * half[k]) for k in range(3))
    v, t = _numbers(seed + 3, n, 0.95, 0.998), _numbers(seed + 4, n, -3.0, 3.0)
    e, mx, my = np.zeros(shape), np.zeros(shape), np.zeros(shape)
    for k in range(n):
        f = 1.0 / (1.0 + (X - x[k]) * (X - x[k]) + (Y - y[k]) * (Y - y[k]) + (Z - z[k]) * (Z - z[k]))
        for _ in range(4):
            f = f * f
        e = e + f
        mx = mx + f * (v[k] * (1 - t[k] * t[k]) / (1 + t[k] * t[k]))
        my = my + f * (v[k] * 2 * t[k] / (1 + t[k] * t[k]))
    s = 55.0 / e.max()
    return e * s, mx * s, my * s


def _flow(shape, d, seed):
    """A flowing state with a shear tensor that is transverse and traceless to first order in the velocity."""
    X, Y, Z = _grid(shape, d)
    e = 4.0 * _spots(shape, d, seed, 40)[0] / 55.0
    u = np.stack([0.25 * X, 0.3 * Y, 0.1 * Z])
    p = 0.03 * e
    pi = np.zeros((10,) + shape)
    pi[4], pi[7], pi[9] = p, p, -2 * p
    pi[1], pi[2], pi[3] = p * u[0], p * u[1], -2 * p * u[2]
    return e, u, pi


def compute(name):
    """Fields (18 or more, flat cells) of a case, in FP32."""
    shape, d = (37, 35, 13), (0.12, 0.12, 0.15)
    if name == "batch":
        cs = []
        for k, sh in enumerate([(25, 23, 9), (31, 29, 14), (19, 21, 7)]):
            e = _spots(sh, d, 11 * k, 20)[0]
            z = np.zeros_like(e)
            cs.append(I.HydroCase("event", *sh, *d, 0.4, 0.005, (0.16, 0.0, 0.08)[k], I.crossover_eos(), e, z, z, z, 0))
        b = clv.Batch(cs, clv.CLV_FP32)
        for k, c in enumerate(cs):
            b.set_event(k, c.eps, c.ux, c.uy, c.ueta)
        b.step(8)
        got = [b.get_event(k, FIELDS) for k in range(len(cs))]
        return np.stack([np.concatenate([g[f].ravel() for g in got]) for f in FIELDS])
    table = None if name == "minijet_conformal" else I.crossover_eos()
    more = {"options": dict(charge=True, zeta_over_s=0.05), "lambda1": dict(lambda1_hat=-2.0),
            "direct": dict(kernel=1)}.get(name, {})
    tau0 = 2.5 if name == "flow" else 0.4
    h = clv.Hydro(*shape, *d, tau0, 0.005, 0.16, table, clv.CLV_FP32, **more)
    if name == "flow":
        e, u, pi = _flow(shape, d, 3)
        h.set_initial(e, *u, pi)
    else:
        e, mx, my = _spots(shape, d, 5, 16)
        h.set_initial_T(np.stack([e, mx, my, np.zeros_like(e)]))
    names = list(FIELDS)
    if name == "options":
        h.set_initial_n(0.02 * e)
        names += ["Nt", "Pi"]
    h.step(6)
    f = h.get(names)
    return np.stack([f[k].ravel() for k in names])


def _recorded():
    """{case: (cells, largest value of each field, values (field, cell))}"""
    out = {}
    for line in open(GOLDEN):
        if line.startswith("#") or not line.strip():
            continue
        name, what, *v = line.split()
        cells, top, rows = out.setdefault(name, ([], [], []))
        if what == "largest":
            top.extend(float.fromhex(x) for x in v)
        else:
            cells.append(int(what))
            rows.append([float.fromhex(x) for x in v])
    return {k: (c, np.array(t), np.array(r).T) for k, (c, t, r) in out.items()}


@pytest.mark.parametrize("name", CASES)
def test_single_precision_fields_are_the_recorded_ones(name):
    cells, top, want = _recorded()[name]
    got = compute(name)[:, cells]
    off = np.abs(got - want).max(1) / np.where(top > 0, top, 1.0)
    assert np.all(off <= 16 * 2.0 ** -24), (name, off.max(), int(off.argmax()))
