"""Calls made while the device memory is nearly full: what a call that ran out
of it leaves behind, and what runs without the memory for the digits."""
import numpy as np
import pytest

from paper_2403_04351_gb300 import Context, RttddftError
from synth import make_dv, make_system, pulse_samples, dv_scale_samples, tiny_config

pytestmark = pytest.mark.gpu

MIB = 1 << 20


class Full:
    """All of the device memory taken but `left` bytes (to the driver's granularity)."""

    def __init__(self, left):
        import torch
        torch.cuda.empty_cache()
        torch.cuda.synchronize()
        self.hold = []
        for part in (4096 * MIB, 256 * MIB, 32 * MIB, 4 * MIB):
            while torch.cuda.mem_get_info()[0] > left + part:
                try:
                    n = (torch.cuda.mem_get_info()[0] - left) // part
                    self.hold.append(torch.empty(int(n) * part, dtype=torch.uint8, device="cuda"))
                except torch.OutOfMemoryError:  # not in one piece
                    try:
                        self.hold.append(torch.empty(part, dtype=torch.uint8, device="cuda"))
                    except torch.OutOfMemoryError:
                        break

    def __enter__(self):
        return self

    def __exit__(self, *_):
        import torch
        self.hold.clear()
        torch.cuda.empty_cache()


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_set_dv_after_one_that_ran_out_of_memory(prec):
    """The first call fails in the transform's columns, the last buffers it
    takes.  The same call with the memory free again gives the dVV of a context
    that never failed: the states bit for bit, since both run the same launches."""
    s = make_system(tiny_config(n_g=2500, n_atoms=2, lmax=3, n_lo_per_atom=4, n_s=3, n_aux=200))
    dv = make_dv(s, amp=0.3)
    a, sc = pulse_samples(s, n_steps=3, a0=5.0), dv_scale_samples(3, s["dt"], freq=3.0)

    def steps(ctx):
        ctx.step(a, sc)
        return ctx.get_state(0), ctx.observables()["energy"]

    ctx = Context(s, precision=prec, interstitial="fft", graph_steps=3)
    ctx.set_dv(dv)
    want = steps(ctx)
    ctx.close()
    ctx = Context(s, precision=prec, interstitial="fft", graph_steps=3)
    for _ in range(2):
        with Full(48 * MIB):
            with pytest.raises(RttddftError) as e:
                ctx.set_dv(dv)
        assert e.value.code == -6
    ctx.set_dv(dv)
    got = steps(ctx)
    ctx.close()
    assert np.array_equal(got[0], want[0])
    assert np.array_equal(got[1], want[1])


def test_set_dv_fits_where_its_buffers_do():
    """The digits of the rebuild are optional: they come after the buffers that the call
    cannot do without (the transform's 97 MiB among 112), not before them.  Same states
    with and without them, to FP64's 1e-11 over three steps."""
    s = make_system(tiny_config(n_g=2500, n_atoms=2, lmax=3, n_lo_per_atom=4, n_s=3, n_aux=200))
    dv = make_dv(s, amp=0.3)
    a, sc = pulse_samples(s, n_steps=3, a0=5.0), dv_scale_samples(3, s["dt"], freq=3.0)
    want = None
    for left in (None, 200, 128):
        ctx = Context(s, interstitial="fft", graph_steps=3)
        if left is None:
            ctx.set_dv(dv)
        else:
            with Full(left * MIB):
                ctx.set_dv(dv)
        ctx.step(a, sc)
        th = ctx.get_state(0)
        ctx.close()
        want = th if want is None else want
        assert np.linalg.norm(th - want) < 1e-11 * np.linalg.norm(want)


def _names(ctx, a, sc=None):
    return {n for n, _ in ctx.trace(a, sc)}


@pytest.mark.parametrize("route", ["toeplitz", "fft"])
@pytest.mark.parametrize("n_s", [3, 12])
def test_fp64_form_without_the_memory_for_its_digits(route, n_s):
    """Set-up and a potential change in memory that the digits do not fit into: the FP64
    kernels run, with the record and the states of the digit products to their
    common rounding (1e-11 of E and of the states' norm over four steps, the bound
    that both have against the oracle)."""
    s = make_system(tiny_config(n_g=2500, n_atoms=2, lmax=3, n_lo_per_atom=4, n_s=n_s, n_aux=200))
    dv = make_dv(s, amp=0.3)
    a, sc = pulse_samples(s, n_steps=4, a0=5.0), dv_scale_samples(4, s["dt"], freq=3.0)

    def run(ctx):
        ctx.set_dv(dv)
        ctx.step(a, sc)
        hx, sx = ctx.apply(0, x, np.array([1.0, -2.0, 3.0]), 0.7)
        names = _names(ctx, a[:1], sc[:1])
        out = ctx.observables()["energy"], ctx.get_state(0), hx, sx
        ctx.close()
        return names, out

    rng = np.random.default_rng(1)
    nb = int(s["n_g"][0]) + int(np.sum(s["n_lo"]))
    x = rng.standard_normal((nb, n_s + 2)) + 1j * rng.standard_normal((nb, n_s + 2))
    names, want = run(Context(s, interstitial=route, graph_steps=2))
    assert "split_reduce_forward" not in names and "gemm_forward" in names
    with Full((230 if route == "fft" else 110) * MIB):
        names, got = run(Context(s, interstitial=route, graph_steps=2))
    assert "split_reduce_forward" in names or "tc_backprojection" not in names
    for g, w in zip(got, want):
        assert np.max(np.abs(g - w)) < 1e-11 * np.linalg.norm(w)


def test_error_flag_starts_clear():
    """A context that takes its basis as given reads no flag of the memory's last owner:
    contexts of other shapes come and go between, and none of its waits has run out."""
    from oracle import Oracle
    s = make_system(tiny_config(n_g=300, n_atoms=1, lmax=1, n_lo_per_atom=1, n_s=3, n_aux=20))
    kp = Oracle(s).kp[0]
    a = pulse_samples(s, n_steps=2, a0=5.0)
    for n in (200, 400, 800):
        other = Context(make_system(tiny_config(n_g=n, n_atoms=1, lmax=1, n_lo_per_atom=1, n_s=5, n_aux=30)), precision="bf16x3")
        other.close()
        ctx = Context(s, aux_mode="given", caux=[kp["caux"]], eps=[kp["eps"]])
        ctx.step(a)
        assert len(ctx.observables()["t"]) == 2
        ctx.close()


def test_adjoint_without_the_memory_for_its_history():
    """The Chebyshev vectors of a whole segment (22 MiB) are optional: without them the
    sweep forms one step's at a time.  Gradients to 1e-9 of the largest, the bound of
    both against the oracle."""
    s = make_system(tiny_config(n_g=300, n_atoms=1, lmax=1, n_lo_per_atom=1, n_s=8, n_aux=200))
    a = pulse_samples(s, n_steps=60, a0=5.0)
    g = np.array([0.3, -0.5, 0.8])
    ctx = Context(s)
    with Full(16 * MIB):
        got, dmu = ctx.adjoint(a, g, ckpt_every=60)
    ctx.close()
    ctx = Context(s)
    want, dmu_want = ctx.adjoint(a, g, ckpt_every=60)
    ctx.close()
    assert np.max(np.abs(got - want)) < 1e-9 * np.max(np.abs(want))
    assert np.max(np.abs(dmu - dmu_want)) < 1e-9 * np.max(np.abs(dmu_want))
