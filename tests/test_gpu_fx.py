"""The FP64 FFT route in fixed point, at the edges of what it stores: columns
of very different sizes, zero columns, sparse ones (whole planes and chunks of
zeros), subnormal and non-finite entries, grids of 2, 3 and 5 radices and a
potential change alone and added."""
import numpy as np
import pytest

from oracle import explicit_dv, explicit_operators, hamiltonian
from paper_2403_04351_gb300 import Context
from synth import make_dv, make_system, tiny_config
from systems import free_electron_system

pytestmark = pytest.mark.gpu


def plane_waves_in_a_potential(n_g, n_s, n_aux):
    s = free_electron_system(n_g=n_g, n_s=n_s, n_aux=n_aux)
    s["vtab"] = make_system(tiny_config(n_g=n_g, n_s=n_s, n_aux=n_aux, seed=5))["vtab"]
    return s


@pytest.mark.parametrize("launches", ["5", "3"])
@pytest.mark.parametrize("n_g,dv", [(7, False), (25, False), (130, False), (900, False), (60, True), (400, True)])
def test_columns_of_any_size(n_g, dv, launches, monkeypatch):
    """Every pass keeps 53 bits or more below the largest value of a block and
    there are six, so a column is good to about 1e-15 of its largest entry; the
    bound is the 1e-13 at which the FFT route has to agree with the direct sum."""
    monkeypatch.setenv("RTTDDFT_FFT_LAUNCHES", launches)
    if dv:
        s = make_system(tiny_config(n_g=n_g, n_atoms=1, lmax=1, n_lo_per_atom=1, n_s=2, n_aux=8))
    else:
        s = plane_waves_in_a_potential(n_g, 1, 4)
    rng = np.random.default_rng(n_g)
    nb, ng = int(s["n_g"][0]) + int(np.sum(s["n_lo"])), int(s["n_g"][0])
    x = rng.standard_normal((nb, 9)) + 1j * rng.standard_normal((nb, 9))
    x[:, 1] = 0.0
    x[:, 2] *= 1e-200
    x[:, 3] *= 1e150
    x[: ng - 1, 4] = 0.0  # one plane wave
    x[:, 5] *= 10.0 ** rng.uniform(-30, 0, nb)
    x[: ng // 2, 6] *= 1e-290
    x[:, 7] = 1.0
    ctx = Context(s, interstitial="fft")
    ops = explicit_operators(s, 0)
    h = hamiltonian(ops, np.zeros(3), s["c_light"])
    scales = [0.0]
    if dv:
        d = make_dv(s)
        ctx.set_dv(d)
        scales = [0.0, 0.7, -1e-20, 1e6]
    for sc in scales:
        want = h if sc == 0.0 else hamiltonian(ops, np.zeros(3), s["c_light"], explicit_dv(s, 0, d), sc)
        hx, _ = ctx.apply(0, x, np.zeros(3), sc)
        assert np.all(hx[:, 1] == 0.0)
        ref = want @ x
        bound = np.max(np.abs(want)) * np.max(np.abs(x), axis=0)
        bound[1] = 1.0
        assert np.max(np.max(np.abs(hx - ref), axis=0) / np.maximum(np.max(np.abs(ref), axis=0), bound)) < 1e-13
    ctx.close()


@pytest.mark.parametrize("launches", ["5", "3"])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_non_finite_columns_stay_their_own(bad, launches, monkeypatch):
    monkeypatch.setenv("RTTDDFT_FFT_LAUNCHES", launches)
    s = plane_waves_in_a_potential(60, 3, 6)
    rng = np.random.default_rng(3)
    x = rng.standard_normal((60, 3)) + 1j * rng.standard_normal((60, 3))
    ctx = Context(s, interstitial="fft")
    want, _ = ctx.apply(0, x, np.zeros(3), 0.0)
    x[17, 1] = bad
    got, _ = ctx.apply(0, x, np.zeros(3), 0.0)
    assert np.array_equal(got[:, [0, 2]], want[:, [0, 2]])
    assert not np.any(np.isfinite(got[:, 1]))
    ctx.close()


@pytest.mark.parametrize("route", ["toeplitz", "fft"])
@pytest.mark.parametrize("n_s,n_cols", [(7, 9), (7, 17), (16, 19), (17, 18)])
def test_last_columns_of_an_fp32_block(n_s, n_cols, route):
    """Blocks that the states do not divide: the last columns alone (16 states and
    fewer) or padded, at the FP32 form's 1e-5 (|H||x|)."""
    s = make_system(tiny_config(n_g=150, n_atoms=2, lmax=2, n_lo_per_atom=3, n_s=n_s, n_aux=24))
    rng = np.random.default_rng(n_cols)
    nb = int(s["n_g"][0]) + int(np.sum(s["n_lo"]))
    x = rng.standard_normal((nb, n_cols)) + 1j * rng.standard_normal((nb, n_cols))
    a_vec = np.array([3.0, -1.0, 2.0])
    ctx = Context(s, precision="fp32", interstitial=route)
    hx, sx = ctx.apply(0, x, a_vec, 0.0)
    ops = explicit_operators(s, 0)
    h = hamiltonian(ops, a_vec, s["c_light"])
    assert np.max(np.abs(hx - h @ x) / (np.abs(h) @ np.abs(x))) < 1e-5
    assert np.max(np.abs(sx - ops["S"] @ x) / (np.abs(ops["S"]) @ np.abs(x))) < 1e-5
    ctx.close()
