"""The FP64 contractions by exact digit products on the tensor cores, at the
edges of their tiles (128 rows, 16/32/64 real columns, K in stages of 32
reals and slices of 64), against plain FP64."""
import numpy as np
import pytest
import scipy.linalg as sla

from paper_2403_04351_gb300 import Context
from synth import make_dv, make_system, tiny_config

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_aux,n_s", [(16, 9), (33, 16), (128, 17), (129, 32), (145, 33), (300, 64), (97, 70)])
def test_series_of_many_states(n_aux, n_s):
    """theta' = exp(-i HH dt) theta for states of very different norms and for
    a zero column.  The digits' cut (2^-54 of the norm per factor and term,
    sqrt(2 n) entries, about 15 terms) stays below 2e-14 of a column's norm;
    the reference's own rounding is of the same size."""
    s = make_system(tiny_config(n_g=max(n_aux, 60), n_s=n_s, n_aux=n_aux, n_k=2, kgrid=(2, 1, 1)))
    rng = np.random.default_rng(n_aux)
    ctx = Context(s, graph_steps=1)
    a = np.array([[1.0, -2.0, 3.0], [0.5, 4.0, 0.0]])
    want = []
    for k in range(2):
        th = rng.standard_normal((n_aux, n_s)) + 1j * rng.standard_normal((n_aux, n_s))
        th *= 10.0 ** rng.integers(-30, 30, n_s)[None, :]
        th[:, 1] = 0.0
        th[:, 2] = np.eye(n_aux)[:, n_aux - 1]
        ctx.set_state(k, th)
        _, eps, pp = ctx.get_aux(k)
        for v in a:
            h = np.diag(eps + v @ v / (2 * s["c_light"] ** 2)) + np.tensordot(v / s["c_light"], pp, 1)
            th = sla.expm(-1j * s["dt"] * h) @ th
        want.append(th)
    ctx.step(a)
    for k in range(2):
        got = ctx.get_state(k)
        assert np.all(got[:, 1] == 0.0)
        norm = np.linalg.norm(want[k], axis=0)
        norm[1] = 1.0
        assert np.max(np.linalg.norm(got - want[k], axis=0) / norm) < 4e-14
    ctx.close()


@pytest.mark.parametrize("n_g,n_s,n_atoms", [(40, 1, 1), (128, 8, 2), (129, 9, 1), (255, 17, 3), (300, 33, 2), (65, 64, 0)])
@pytest.mark.parametrize("route", ["toeplitz", "fft"])
def test_operator_and_projection(n_g, n_s, n_atoms, route):
    """FP64 operator on columns of very different sizes (and a zero one), and
    the expansion and projection of a step, against the explicit matrices.
    The cut is 2^-54 of a row's and of a column's largest entry: entrywise
    2^-53 sqrt(K) of their product and below, here 1e-13 of the row's and
    column's norms with the three products in a row."""
    from oracle.rttddft_oracle import explicit_operators, hamiltonian
    from systems import free_electron_system
    if n_atoms:
        s = make_system(tiny_config(n_g=n_g, n_atoms=n_atoms, lmax=2, n_lo_per_atom=3, n_s=n_s, n_aux=max(n_s, 12)))
    else:
        s = free_electron_system(n_g=n_g, n_s=n_s, n_aux=n_s)
    rng = np.random.default_rng(n_g)
    ctx = Context(s, interstitial=route)
    ops = explicit_operators(s, 0)
    nb = ops["nb"]
    x = rng.standard_normal((nb, n_s + 1)) + 1j * rng.standard_normal((nb, n_s + 1))
    x *= 10.0 ** rng.integers(-100, 100, n_s + 1)[None, :]
    x[:, 0] = 0.0
    a = np.array([0.4, -0.9, 1.3])
    hx, sx = ctx.apply(0, x, a)
    h = hamiltonian(ops, a, s["c_light"])
    assert np.all(hx[:, 0] == 0.0) and np.all(sx[:, 0] == 0.0)
    size = np.linalg.norm(x[:, 1:], axis=0)
    assert np.max(np.abs(hx - h @ x)[:, 1:] / (np.linalg.norm(h, axis=1)[:, None] * size)) < 1e-13
    assert np.max(np.abs(sx - ops["S"] @ x)[:, 1:] / (np.linalg.norm(ops["S"], axis=1)[:, None] * size)) < 1e-13
    if n_s > 1:
        x[1, 1] = np.nan
        assert np.all(np.isnan(ctx.apply(0, x, a)[0][:, 1]))
    ctx.step(a[None, :])
    o = ctx.observables()
    th, c = ctx.get_state(0, with_c=True)
    cc = ctx.get_aux(0)[0]
    e = 2.0 * np.real(np.vdot(cc @ th, h @ (cc @ th)))
    assert abs(o["energy"][0] - e) < 1e-12 * max(1.0, abs(e))
    assert o["resid"][0] < 1e-12 and o["norm_dev"][0] < 1e-12
    ctx.close()


@pytest.mark.parametrize("prec,tol", [("fp64", 1e-11), ("fp32", 1e-5)])
@pytest.mark.parametrize("n_aux,n_s,n_atoms,n_k", [(12, 1, 1, 1), (65, 17, 2, 2), (130, 33, 3, 1)])
def test_rebuilt_potential_change(prec, tol, n_aux, n_s, n_atoms, n_k):
    """dVV rebuilt over four steps, with the pattern replaced after two, against
    the explicit matrices (the FP32 form's T carries FP32 accuracy)."""
    from oracle import Oracle
    from synth import dv_scale_samples, make_dv, pulse_samples
    s = make_system(tiny_config(n_g=200, n_atoms=n_atoms, lmax=2, n_lo_per_atom=3, n_s=n_s, n_aux=n_aux, n_k=n_k,
                                kgrid=(n_k, 1, 1)))
    a, sc = pulse_samples(s, n_steps=4, a0=5.0), dv_scale_samples(4, s["dt"], freq=3.0)
    pats = make_dv(s, amp=0.3), make_dv(s, amp=0.2, seed_offset=3)
    ctx = Context(s, precision=prec, graph_steps=2)
    th = None
    for i, dv in enumerate(pats):
        r = Oracle(s, dv=dv).run(a[2 * i:2 * i + 2], s["dt"], dv_scale=sc[2 * i:2 * i + 2], thetas=th)
        th = r["theta"]
        ctx.set_dv(dv)
        ctx.step(a[2 * i:2 * i + 2], sc[2 * i:2 * i + 2])
    o = ctx.observables()
    for k in range(n_k):
        d = ctx.get_state(k) - th[k]
        assert np.linalg.norm(d) / np.linalg.norm(th[k]) < tol
    assert np.max(np.abs(o["energy"][2:] - r["E"]) / np.abs(r["E"])) < tol
    ctx.close()


@pytest.mark.parametrize("n_aux,n_s,n_k", [(3, 1, 1), (16, 2, 2), (129, 3, 1), (200, 4, 3), (256, 5, 1), (257, 8, 1), (400, 7, 1),
                                           (470, 3, 1), (90, 8, 8)])
@pytest.mark.parametrize("prop", ["chebyshev", "cn"])
def test_series_of_few_states(n_aux, n_s, n_k, prop):
    """The cooperative integer series (and, past its rows, the digit products
    with few columns): states of very different norms, a zero column, 12 steps
    in graphs of three.  Its cut (2^-59 of the norm per factor and term) stays
    far below the reference's rounding; 4e-14 of a column's norm over the run."""
    s = make_system(tiny_config(n_g=max(n_aux, 60), n_s=n_s, n_aux=n_aux, n_k=n_k, kgrid=(n_k, 1, 1)))
    rng = np.random.default_rng(n_aux)
    ctx = Context(s, propagator=prop, graph_steps=3)
    a = rng.standard_normal((12, 3)) * 3.0
    want = []
    for k in range(n_k):
        th = rng.standard_normal((n_aux, n_s)) + 1j * rng.standard_normal((n_aux, n_s))
        th *= 10.0 ** rng.integers(-200, 200, n_s)[None, :]
        if n_s > 2:
            th[:, 1] = 0.0
            th[:, 2] = np.eye(n_aux)[:, n_aux - 1]
        ctx.set_state(k, th)
        _, eps, pp = ctx.get_aux(k)
        one = np.eye(n_aux)
        for v in a:
            h = np.diag(eps + v @ v / (2 * s["c_light"] ** 2)) + np.tensordot(v / s["c_light"], pp, 1)
            if prop == "cn":
                th = np.linalg.solve(one + 0.5j * s["dt"] * h, (one - 0.5j * s["dt"] * h) @ th)
            else:
                lam, u = np.linalg.eigh(0.5 * (h + h.conj().T))
                th = u @ (np.exp(-1j * s["dt"] * lam)[:, None] * (u.conj().T @ th))
        want.append(th)
    ctx.step(a)
    for k in range(n_k):
        got, size = ctx.get_state(k), np.max(np.abs(want[k]), axis=0)
        assert np.all(got[:, size == 0.0] == 0.0)
        size[size == 0.0] = 1.0
        assert np.max(np.linalg.norm((got - want[k]) / size, axis=0) / np.maximum(np.linalg.norm(want[k] / size, axis=0), 1.0)) < 4e-14
    ctx.close()


@pytest.mark.parametrize("n_aux,n_s", [(130, 3), (33, 4), (60, 12)])
def test_a_k_point_that_is_not_finite_stays_alone(n_aux, n_s):
    """A potential change whose norm leaves FP64's range for one k-point only, at scale
    0: that k-point's interval is not a number, the other's steps are those without
    the change (the same operator; the rounding of a different interval, 1e-12)."""
    from oracle import explicit_dv
    s = make_system(tiny_config(n_g=max(n_aux, 60), n_s=n_s, n_aux=n_aux, n_k=2, kgrid=(2, 1, 1)))
    a = np.random.default_rng(5).standard_normal((3, 3))
    plain = Context(s, graph_steps=1)
    plain.step(a)
    want = [plain.get_state(k) for k in range(2)]
    dv = make_dv(s, amp=0.3)
    norm = []
    for k in range(2):
        cc = plain.get_aux(k)[0]
        norm.append(np.linalg.norm(cc.conj().T @ explicit_dv(s, k, dv) @ cc))
    plain.close()
    assert abs(norm[0] / norm[1] - 1.0) > 1e-6
    big = np.sqrt(np.finfo(float).max / (norm[0] * norm[1]))
    keep = int(np.argmin(norm))
    ctx = Context(s, graph_steps=1)
    ctx.set_dv(dict(dh=[d * big for d in dv["dh"]], dvtab=dv["dvtab"] * big))
    ctx.step(a, np.zeros(3))
    assert np.linalg.norm(ctx.get_state(keep) - want[keep]) < 1e-12 * np.sqrt(n_s)
    assert np.all(np.isnan(ctx.get_state(1 - keep)))
    ctx.close()


@pytest.mark.parametrize("n_g,n_s", [(512, 2), (700, 16), (2600, 2)])
def test_coherent_digits(n_g, n_s):
    """Constant operands (every digit of one sign) and columns whose leading digits
    cancel while the low ones add up, in the direct sum: H x = |G|^2/2 x + c sum x for a
    table that is c everywhere.  2 N_G products a part, each with at most 2^-53 from the
    cut and 2^-51.6 from the accumulators: below 2^-49 of N_G |c| max|x|."""
    from systems import free_electron_system
    s = free_electron_system(n_g=n_g, n_s=n_s, n_aux=n_s)
    rng = np.random.default_rng(n_g)
    sign = np.where(np.arange(n_g) % 2 == 0, 1.0, -1.0)
    sign[-1] = 0.0 if n_g % 2 else sign[-1]
    for _ in range(4):
        c = rng.uniform(0.1, 1.0)
        s["vtab"] = np.full_like(s["vtab"], c)
        z = rng.uniform(-1, 1, 16) + 1j * rng.uniform(-1, 1, 16)
        x = np.outer(np.ones(n_g), z)
        x[:, 8:] = np.outer(sign, z[8:]) + rng.uniform(0, 1, 8) * 2.0 ** -rng.integers(1, 40, 8)
        ctx = Context(s)
        got = ctx.apply(0, x)[0]
        ctx.close()
        kin = 0.5 * np.sum(s["gk"][0].astype(np.longdouble) ** 2, axis=1)
        xl = x.astype(np.clongdouble)
        want = kin[:, None] * xl + np.longdouble(c) * np.sum(xl, axis=0)
        err = np.abs(got - want).astype(float)
        size = n_g * c * np.max(np.abs(x), axis=0) + kin.astype(float)[:, None] * np.abs(x)
        assert np.max(err / size) < 2.0 ** -49
