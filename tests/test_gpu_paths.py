"""Edges of the kernels' dispatch: tile shapes at the limits of their task lists, transfers of subnormal and signed-zero
floats, the FP64 root solve over the range of the EOS table and beyond its top, and the initial T~ after the first-step predictor.

Tolerances: tiles are a schedule, so fields agree bit for bit; a float widened to a double is that float; a root that
the solve accepts reproduces E and |M| within its own rounding, a few eps (2.2e-16) times the 1/(1 - v^2) < 500 by which
eps = E - M v amplifies it: 1e-12."""
import numpy as np
import pytest

from paper_1802_04449_gb300 import clv
from paper_1802_04449_gb300 import inputs as I

pytestmark = pytest.mark.gpu

FIELDS = ["eps", "ux", "uy", "ueta", "Ttt", "pixx", "piee"]


@pytest.mark.parametrize("prec,shapes", [
    (clv.CLV_FP64, [(1, 1), (1, 45), (2, 13), (8, 16), (10, 14), (30, 3), (37, 2)]),
    (clv.CLV_FP32, [(1, 1), (1, 45), (8, 41), (6, 45), (28, 11), (37, 7)])])
@pytest.mark.parametrize("eta_over_s", [0.0, 0.08])
def test_tiles_at_the_limits_of_their_tasks(prec, shapes, eta_over_s):
    case = I.hotspot_event(nx=9, ny=37, neta=45, n_spots=60, seed=5, eta_over_s=eta_over_s)

    def run(shape):
        g = clv.from_case(case, prec)
        g.set_initial(case.eps, case.ux, case.uy, case.ueta)
        if shape:
            g.set_tile(*shape, 0)
        g.step(2)
        return g.get(FIELDS if eta_over_s else FIELDS[:5])

    ref = run(None)
    for shape in shapes:
        got = run(shape)
        for k in ref:
            assert np.array_equal(got[k], ref[k]), (shape, k)


def test_exports_are_the_floats_that_the_solver_holds():
    """Initial velocities with zeros of both signs, subnormal and ordinary floats, on a ragged grid and past one block."""
    shape = (13, 11, 9)
    rng = np.random.default_rng(2)
    u = rng.normal(size=shape)
    u.flat[::7], u.flat[1::7], u.flat[2::7], u.flat[3::7] = 0.0, -0.0, 1e-42, -3e-39
    h = clv.Hydro(*shape, 0.2, 0.2, 0.2, 0.6, 0.01, 0.0, None, clv.CLV_FP32)
    h.set_initial(np.ones(shape), u, np.zeros(shape), -u)
    f = h.get(["ux", "ueta"])
    d = h.get_device(["ux", "ueta"])
    for k, x in (("ux", u), ("ueta", -u)):
        want = x.astype(np.float32).astype(np.float64)
        assert np.array_equal(f[k].view(np.int64), want.view(np.int64)), k
        assert np.array_equal(d[k].cpu().numpy().view(np.int64), want.view(np.int64)), k


def test_fp64_root_solve_over_the_table():
    """eps from the vacuum cut to above the last node, at nodes and between them, v from 0 to 0.997."""
    eos = I.crossover_eos()
    lne0, dlne, n = eos["lne0"], eos["dlne"], len(eos["P"])
    x = np.concatenate([np.linspace(-30, -1, 8), np.arange(0, n - 1, 97.0), np.arange(0, n - 1, 101.5), [n - 1.0, n + 9.0]])
    x = x[lne0 + x * dlne > np.log(2e-7)]
    e = np.exp(lne0 + x * dlne)
    v = np.array([0.0, 1e-3, 0.3, 0.9, 0.99, 0.997])
    e, v = (a.ravel() for a in np.meshgrid(e, v, indexing="ij"))

    def P_of(e):
        y = (np.log(e) - lne0) / dlne
        k = np.clip(np.floor(y), 0, n - 2).astype(int)
        P = eos["P"][k] + (y - k) * (eos["P"][k + 1] - eos["P"][k])
        top = np.exp(lne0 + (n - 1) * dlne)
        return np.where(y < 0, eos["P"][0] * e / np.exp(lne0), np.where(y >= n - 1, eos["P"][-1] + (e - top) / 3, P))

    g2 = 1 / (1 - v * v)
    E, M = (e + P_of(e)) * g2 - P_of(e), (e + P_of(e)) * g2 * v
    pad = -len(e) % 4
    shape = ((len(e) + pad) // 4, 2, 2)
    T = np.zeros((4,) + shape)
    T[0].flat[:len(e)], T[2].flat[:len(e)] = E, M
    T[0].flat[len(e):] = 1.0
    h = clv.Hydro(*shape, 0.2, 0.2, 0.2, 0.6, 0.01, 0.0, eos, clv.CLV_FP64)
    h.set_initial_T(T)
    f = h.get(["eps", "uy"])
    eg, uy = f["eps"].ravel()[:len(e)], f["uy"].ravel()[:len(e)]
    g2 = 1 + uy * uy
    assert np.all(np.abs((eg + P_of(eg)) * g2 - P_of(eg) - E) <= 1e-12 * E)
    assert np.all(np.abs((eg + P_of(eg)) * np.sqrt(g2) * uy - M) <= 1e-12 * E)


@pytest.mark.parametrize("prec,tol", [(clv.CLV_FP64, 1e-14), (clv.CLV_FP32, 1e-13)])
def test_initial_T_is_kept_by_the_predictor(prec, tol):
    """T~^{tau mu} right after a viscous initial state without pi~ is the ideal tensor of its primitives (FP32: formed
    in FP64 from the stored floats, kept to 48 bits), with the pressure read back through T~^{tau tau}."""
    case = I.hotspot_event(nx=13, ny=11, neta=7, n_spots=30, seed=9, eta_over_s=0.08)
    h = clv.from_case(case, prec)
    rng = np.random.default_rng(4)
    u = 0.3 * rng.normal(size=(3,) + case.eps.shape)
    h.set_initial(case.eps, *u)
    f = h.get(["eps", "ux", "uy", "ueta", "Ttt", "Ttx", "Tty", "Tte"])
    ut2 = 1 + f["ux"] ** 2 + f["uy"] ** 2 + f["ueta"] ** 2
    live = f["eps"] > 0
    # T~^{tau i} = tau w u^tau u^i and T~^{tau tau} = tau (w u^tau^2 - P): the enthalpy w from one gives the others
    w = f["Ttx"] / (case.tau0 * np.sqrt(ut2) * np.where(live, f["ux"], 1.0))
    P = w - f["eps"]
    for k, want in (("Tty", case.tau0 * w * np.sqrt(ut2) * f["uy"]), ("Tte", case.tau0 * w * np.sqrt(ut2) * f["ueta"]),
                    ("Ttt", case.tau0 * (w * ut2 - P))):
        assert np.all(np.abs(f[k] - want)[live] <= tol * 50 * np.abs(f["Ttt"])[live]), k


@pytest.mark.parametrize("refused", [False, True])
@pytest.mark.parametrize("prec", [clv.CLV_FP64, clv.CLV_FP32])
def test_padding_stays_vacuum_through_an_initial_T(prec, refused):
    """Rows of 9 cells have a pitch of 12: in a checkpoint taken before the first step the padding of T~ and pi~ is 0 and that of
    the previous step's primitives equals that of the current ones, vacuum -- also after an initial T that was refused."""
    case = I.hotspot_event(nx=15, ny=13, neta=9, n_spots=30, seed=2, eta_over_s=0.08)
    h = clv.from_case(case, prec)
    T = np.stack([case.eps, 0.3 * case.eps, -0.2 * case.eps, 0.1 * case.eps])
    if refused:
        with pytest.raises(clv.ClvError):
            h.set_initial_T(np.where(np.arange(9) == 4, np.nan, T))
        h.set_initial(case.eps, case.ux, case.uy, case.ueta)
    else:
        h.set_initial_T(T)
    R = np.float64 if prec == clv.CLV_FP64 else np.float32
    f = np.frombuffer(bytes(h.get_state()), R, offset=88).reshape(-1, 15, 13, 12)[..., 9:]
    assert len(f) == (26 if prec == clv.CLV_FP64 else 30)
    assert np.all(f[:-12] == 0) and np.all(f[-12:-8] == 0)
    assert np.array_equal(f[-6:], f[-12:-6])


@pytest.mark.parametrize("shape", [(81, 2), (82, 2), (84, 2), (124, 1), (125, 1), (127, 1)])
def test_long_tiles_whose_threads_stage_two_vectors(shape):
    """FP64 tiles of one or two columns have up to 264 four-cell vectors in a plane for 256 threads (81 x 2 and 124 x 1 are the
    last with one or none for each).  Fields agree with the default tile's bit for bit."""
    case = I.hotspot_event(nx=7, ny=129, neta=5, n_spots=60, seed=6, eta_over_s=0.0)

    def run(tile):
        g = clv.from_case(case, clv.CLV_FP64)
        g.set_initial(case.eps, case.ux, case.uy, case.ueta)
        if tile:
            g.set_tile(*tile, 0)
            assert g.tile()["TJ"] == tile[0]
        g.step(3)
        return g.get(FIELDS[:5])

    ref, got = run(None), run(shape)
    for k in ref:
        assert np.array_equal(got[k], ref[k]), k

def test_logarithm_of_the_fp64_lookup():
    """P(eps) of the table on both sides of the edges and in the middle of the 64 intervals of the mantissa that the logarithm
    is tabulated over, for every binary exponent of the table, read back through T~^{tau x} = tau (eps + P) u~^tau u~^x.

    Tolerance: P varies by at most d ln P / d ln eps < 2 times an error of ln eps.  ln eps - ln eps_0 < 26 is rounded three
    times here and there, 26 x 6 x 1.1e-16 = 1.7e-14; with T~ and the division by u~ (3 x 1.1e-16 of eps + P < 12 P): 4e-14."""
    eos = I.crossover_eos()
    lne0, dlne, n = eos["lne0"], eos["dlne"], len(eos["P"])
    edge = 1 + np.arange(64) / 64
    m = np.concatenate([edge, np.nextafter(edge, 0), np.nextafter(edge, 2), edge + 1 / 128])
    e = (m[None] * 2.0 ** np.arange(-22, 13)[:, None]).ravel()
    e = e[(e > np.exp(lne0) * 1.01) & (e < np.exp(lne0 + (n - 1) * dlne) * 0.99)]
    e = e[:len(e) // 4 * 4]
    shape = (len(e) // 4, 2, 2)
    x = (np.log(e) - lne0) / dlne
    k = np.clip(np.floor(x), 0, n - 2).astype(int)
    P = eos["P"][k] + (x - k) * (eos["P"][k + 1] - eos["P"][k])
    assert np.all(e / P < 11) and np.max(np.diff(np.log(eos["P"])) / dlne) < 2
    h = clv.Hydro(*shape, 0.2, 0.2, 0.2, 1.0, 0.01, 0.0, eos, clv.CLV_FP64)
    z = np.zeros(shape)
    h.set_initial(e.reshape(shape), z + 0.75, z, z)   # u~^tau = 1.25
    got = h.get(["Ttx"])["Ttx"].ravel() / (1.25 * 0.75) - e
    assert np.all(np.abs(got - P) <= 4e-14 * P), float(np.max(np.abs(got - P) / P))


@pytest.mark.parametrize("prec", [clv.CLV_FP64, clv.CLV_FP32])
@pytest.mark.parametrize("shape", [(152, 128, 64), (151, 131, 63)])
def test_exports_on_both_sides_of_the_small_launch(prec, shape):
    """One field of 152 x 128 x 64 cells is the last export with a cell for each thread; two fields of it, and one of a ragged
    grid with a few cells more, take four a thread: the values are those that were set."""
    import torch
    assert shape[0] * shape[1] * shape[2] - 152 * 128 * 64 in (0, 1019)
    g = torch.Generator(device="cuda").manual_seed(4)
    e, u = (torch.rand(shape, generator=g, dtype=torch.float64, device="cuda") + 0.5 for _ in range(2))
    e, u = e.float().double(), u.float().double()
    z = torch.zeros_like(e)
    h = clv.Hydro(*shape, 0.2, 0.2, 0.2, 0.5, 0.01, 0.0, None, prec)
    h.set_initial(e, u, z, z)
    for names in (["eps"], ["ux"], ["eps", "ux"]):
        f = h.get_device(names)
        for k in names:
            assert torch.equal(f[k].reshape(shape), e if k == "eps" else u), (names, k)
