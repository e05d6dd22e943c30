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


@pytest.mark.parametrize("dims,l,nrhs", [((8, 8, 8, 8), 4, 4), ((12, 12, 12, 12), 6, 1), ((16, 16, 16, 16), 8, 1)])
@pytest.mark.parametrize("prec", [binding.FP64, binding.MIXED_FP32])
def test_block_solves_have_the_same_bits_in_every_context(dims, l, nrhs, prec):
    """Two contexts, one of them with the autotuner off, give the same bits: the block solver's launch shape follows
    from the sizes (these have few blocks, where the shapes differ most)."""
    b = torch.from_numpy(synth.spinor_field(dims, seed=21, nrhs=nrhs)).cuda()
    xs = []
    for tune in (True, False, True):
        ctx = context(dims, l)
        if not tune:
            ctx.autotune(False)
        ctx.set_solver(prec, tol_outer=1e-10, tol_block=1e-12)
        for colour in (0, 1):
            x = torch.zeros_like(b)
            torch.cuda.synchronize()
            ctx.solve_block(colour, 0.07, b, x, nrhs=nrhs)
            xs.append(x)
        ctx.close()
    for k in (2, 3, 4, 5):
        assert torch.equal(xs[k], xs[k % 2])


def test_hard_fp64_solves_keep_their_step_counts():
    """Solves of thousands of BiCGStab steps (a mass beyond the critical one), where ||s|| exceeds ||r|| by orders of
    magnitude and an inner product known only relative to ||s|| costs steps.  Steps of sixteen solves: 122e3 with
    rho and beta from (rh, r), 85e3 with rho alone from it, 174e3 with both from (rh, s) - omega (rh, t); the bar is
    halfway between the last two."""
    dims, steps = (8, 8, 8, 8), 0
    for seed in range(1, 17):
        ctx = binding.Context(dims, (4,) * 4)
        ctx.load_gauge(synth.gauge_field(dims, 0.25, seed=seed))
        ctx.set_params(1.5, -0.105, -0.11)
        ctx.set_solver(binding.FP64, tol_outer=1e-11, tol_block=1e-12, maxiter=4000)
        b = synth.spinor_field(dims, seed=70 + seed)
        steps += ctx.solve_D(-0.11, b, np.zeros_like(b))["iters_outer"]
        ctx.close()
    assert steps <= 130e3


def test_block_config_reaches_captured_estimates():
    """A launch shape pinned after an estimate was captured whole is used by the next estimate: the bits of a context
    on which it was pinned before.  (The shapes add in different orders, so their bits differ.)"""
    e = {}
    for forms in ((0, 2), (2,)):
        ctx = context()
        ctx.set_solver(binding.FP64, tol_outer=1e-11, tol_block=1e-12)
        ctx.use_graphs(1)
        for form in forms:
            ctx.block_config(form)
            for _ in range(3):  # eager, captured, replayed
                e[forms, form] = np.asarray(ctx.estimate(4, seed=5)[0])
        ctx.close()
    assert np.array_equal(e[(0, 2), 2], e[(2,), 2])
    assert not np.array_equal(e[(0, 2), 0], e[(0, 2), 2])


@pytest.mark.parametrize("nrhs,fused", [(1, True), (8, False)])  # 2^15 x 8 sites are beyond the rule's 2^17
def test_fuse_reductions_returns_to_the_size_rule(nrhs, fused):
    """After an explicit setting, -1 chooses by size again (the report lists the stencil shapes that ran)."""
    ctx = context((16, 16, 16, 16))
    ctx.set_solver(binding.MIXED_FP32, tol_outer=1e-10, tol_block=1e-12)
    b = torch.from_numpy(synth.spinor_field((16, 16, 16, 16), seed=5, nrhs=nrhs)).cuda()
    x = torch.zeros_like(b)
    torch.cuda.synchronize()
    ran = []
    for switch in (None, False, True, -1):
        ctx.autotune(True)  # an empty list of shapes
        if switch is not None:
            ctx.fuse_reductions(switch)
        ctx.solve_D(0.12, b, x, nrhs=nrhs)
        ran.append("red=2" in ctx.autotune_report())
    assert ran == [fused, False, True, fused]
    ctx.close()


@pytest.mark.parametrize("prec", [binding.FP64, binding.MIXED_FP32])
def test_force_scratch(prec):
    """The link force takes no more device memory beyond the mass derivative's than its six 3x3 matrices per site
    (864 bytes), the allocator's rounding and the code of its kernels (16 MB for both)."""
    dims = (16, 16, 16, 16)
    ctx = context(dims, 8)
    ctx.set_solver(prec, tol_outer=1e-8, tol_block=1e-8)
    dU = torch.empty((ctx.V, 4, 8), dtype=torch.float64, device="cuda")
    ctx.force(1, seed=5)
    free = torch.cuda.mem_get_info()[0]
    ctx.force(1, seed=5, dU=dU)
    assert free - torch.cuda.mem_get_info()[0] <= 864 * ctx.V + (16 << 20)
    ctx.close()


def test_report_names_the_launches_that_ran():
    """The fully rolled residual stencil (form 11) has CTAs of at most 128 threads, and no larger one is reported."""
    dims = (8, 8, 8, 8)
    ctx = context(dims)
    ctx.set_solver(binding.MIXED_FP32, tol_outer=1e-10, tol_block=1e-12)
    for _ in range(4):
        ctx.autotune(True)
        for nrhs in range(1, 9):
            b = synth.spinor_field(dims, seed=5, nrhs=nrhs)
            x = np.zeros_like(b)
            ctx.solve_block(0, 0.12, b, x, nrhs=nrhs)
            ctx.solve_D(0.12, b, x, nrhs=nrhs)
        lines = [line for line in ctx.autotune_report().splitlines() if "roll=11" in line]
        assert lines and not any("nt=256" in line for line in lines)
    ctx.close()


def test_masses_of_changing_parameters():
    """Solves after changes of the parameters, before and after loads, with masses that were used, that were only the
    context's, and 0 (the mass before the parameters): every residual, by the operator."""
    dims = (8, 8, 8, 8)
    ctx, b = context(dims), synth.spinor_field(dims, seed=9)
    ctx.set_solver(binding.MIXED_FP32, tol_outer=1e-11, tol_block=1e-12)

    def check(*masses):
        for m in masses:
            x, y = np.zeros_like(b), np.zeros_like(b)
            ctx.solve_D(m, b, x)
            ctx.apply_D(m, x, y)
            assert np.linalg.norm(y - b) <= 1.01e-11 * np.linalg.norm(b), m

    for step, (m1, m2) in enumerate([(0.12, 0.07), (0.2, 0.2), (0.07, 0.3), (0.4, 0.0), (0.2, 0.12)]):
        ctx.set_params(1.4, m1, m2)
        if step % 2:
            ctx.load_gauge(synth.gauge_field(dims, 0.3, seed=20 + step))
        if step != 1:  # 0.2 is only the context's at first
            check(m1, m2, 0.25)
    check(0.0, 0.2, 0.07, 0.3, 0.12, 0.25)
    ctx.close()
