"""Amplitudes that a weak field excites keep FP64's relative accuracy, as small
as they are: theta from the ground state against the same steps in extended
precision, over every form of the series (cluster, grid, digit products)."""
import numpy as np
import pytest

from paper_2403_04351_gb300 import Context
from synth import make_system, tiny_config

pytestmark = pytest.mark.gpu

STEPS = 6


def extended_step(eps, pp, a, c, dt, theta):
    """exp(-i dt HH) theta by its Taylor series, in long double."""
    ld, cd = np.longdouble, np.clongdouble
    a = a.astype(ld)
    h = np.tensordot((a / ld(c)).astype(cd), pp.astype(cd), 1)
    h[np.diag_indices(len(eps))] += eps.astype(ld) + (a @ a) / (2 * ld(c) * ld(c))
    parts = int(np.ceil(dt * np.max(np.sum(np.abs(h), axis=0)))) or 1
    f = cd(-1j) * ld(dt) / parts
    for _ in range(parts):
        term = out = theta
        for n in range(1, 28):
            term = (f / n) * (h @ term)
            out = out + term
        theta = out
    return theta


@pytest.mark.parametrize("a0", [0.05, 1e-4, 1e-6])
@pytest.mark.parametrize("n_aux,n_s,n_k", [(16, 1, 2), (64, 1, 1), (32, 2, 1), (40, 4, 1), (33, 8, 2), (130, 7, 1), (200, 2, 1), (270, 2, 1), (60, 12, 1), (40, 10, 2), (129, 17, 1)])
def test_excited_amplitudes_of_a_weak_field(n_aux, n_s, n_k, a0):
    """The root-mean-square of the amplitudes outside the occupied block.  A
    step has about 20 terms of a few roundings each, so STEPS steps keep
    STEPS 20 2^-53 = 1.3e-14 times a small factor: 1e-13."""
    s = make_system(tiny_config(n_g=max(n_aux, 60), n_s=n_s, n_aux=n_aux, n_k=n_k, kgrid=(n_k, 1, 1)))
    ctx = Context(s, graph_steps=2)
    a = a0 * np.random.default_rng(n_aux).standard_normal((STEPS, 3))
    ctx.step(a)
    for k in range(n_k):
        _, eps, pp = ctx.get_aux(k)
        th = np.eye(n_aux, n_s).astype(np.clongdouble)
        for v in a:
            th = extended_step(eps, pp, v, s["c_light"], s["dt"], th)
        got = ctx.get_state(k)
        diff = (got - th).astype(np.complex128)[n_s:]
        size = np.linalg.norm(th.astype(np.complex128)[n_s:])
        assert size < a0  # the excited part is small
        assert np.linalg.norm(diff) < 1e-13 * size, np.linalg.norm(diff) / size
    ctx.close()
