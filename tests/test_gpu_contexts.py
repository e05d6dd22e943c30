"""What a context does is settled by its inputs and switches, not by the calls before: when the work of a new
configuration is done, and which kernels run after a switch is changed."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1211_1214_gb300 import binding, synth

pytestmark = pytest.mark.gpu


def context(dims=(8, 8, 8, 8), l=4, seed=3):
    ctx = binding.Context(dims, (l,) * 4)
    ctx.load_gauge(synth.gauge_field(dims, 0.3, seed=seed))
    ctx.set_params(1.4, 0.12, 0.07)
    return ctx


def launches(ctx, call):
    ctx.profile(True)
    call()
    n = ctx.profile_read(12)[0]
    ctx.profile(False)
    return n


@pytest.mark.parametrize("m", [0.0, 0.3])  # the mass of a field loaded before the parameters, and another
def test_inverses_of_a_used_mass_are_made_by_load_gauge(m):
    """A mass that was used once has its in-block inverses made by every load, also when a configuration in between
    did not use it: its next solve launches what a repeat of that solve launches."""
    ctx, b = context(), synth.spinor_field((8, 8, 8, 8), seed=9)
    x = np.zeros_like(b)
    ctx.set_solver(binding.FP64, tol_outer=1e-11, tol_block=1e-12)
    ctx.use_graphs(False)
    ctx.solve_D(m, b, x)
    for seed in (11, 12):
        ctx.load_gauge(synth.gauge_field((8, 8, 8, 8), 0.3, seed=seed))
    first = launches(ctx, lambda: ctx.solve_D(m, b, x))
    assert first == launches(ctx, lambda: ctx.solve_D(m, b, x))
    y = np.zeros_like(b)
    ctx.apply_D(m, x, y)
    assert np.linalg.norm(y - b) <= 1.01e-11 * np.linalg.norm(b)
    ctx.close()
