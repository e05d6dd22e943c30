"""Calls that choose among several kernels by size, alignment or layout, each compared with the general path
or the oracle.

The FP64 routes order the same sums of about 100 products differently: 1e-13 of the field's norm is about
ten times what 100 roundings of 1.1e-16 can add up to.  A log determinant of a 192 x 192 block of condition
number below 1e3 is known to 192 * 1e3 * 1.1e-16 = 2e-11; the bar is 1e-10.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import core as oc
from paper_1211_1214_gb300 import binding, synth

pytestmark = pytest.mark.gpu

TOL = 1e-13


def context(dims, l, seed=3, antiperiodic=False):
    ctx = binding.Context(dims, (l,) * 4)
    ctx.load_gauge(synth.gauge_field(dims, 0.3, seed=seed))
    ctx.set_params(1.4, 0.12, 0.07, antiperiodic_t=antiperiodic)
    return ctx


def rel(a, b):
    return float(torch.linalg.vector_norm(a - b) / torch.linalg.vector_norm(b))


# sites times right-hand sides on both sides of the split kernel's 12000, every block length, odd counts
@pytest.mark.parametrize("dims,l,nrhs", [((4, 4, 4, 4), 2, 1), ((12, 8, 4, 4), 2, 3), ((8, 8, 8, 8), 4, 2), ((8, 8, 8, 8), 4, 3),
                                         ((12, 12, 12, 12), 6, 1), ((16, 16, 16, 16), 8, 1)])
@pytest.mark.parametrize("antiperiodic", [False, True])
def test_apply_D_layouts_and_block_hops(dims, l, nrhs, antiperiodic):
    ctx = context(dims, l, antiperiodic=antiperiodic)
    x = torch.from_numpy(synth.spinor_field(dims, seed=4, nrhs=nrhs)).cuda()
    n = x.numel()
    calls = [lambda a, o: ctx.apply_D(0.07, a, o, nrhs=nrhs)]
    for rows in (0, 1):
        for cols in (0, 1):
            calls.append(lambda a, o, r=rows, c=cols: ctx.apply_block(r, c, 0.07, a, o, nrhs=nrhs))
    for call in calls:
        ctx.stencil_config(1, 64, 1, 0)  # the general path: internal copies and one thread per site
        want = torch.zeros_like(x)
        call(x, want)
        ctx.stencil_config()
        got = torch.zeros_like(x)
        call(x, got)
        assert rel(got, want) <= TOL
        # in place, and from and to addresses that are multiples of 8 bytes only
        same = x.clone()
        call(same, same)
        assert rel(same, want) <= TOL
        a = torch.empty(2 * n + 1, dtype=torch.float64, device="cuda")[1:]
        o = torch.empty(2 * n + 1, dtype=torch.float64, device="cuda")[1:]
        a.copy_(torch.view_as_real(x).reshape(-1))
        call(a, o)
        assert rel(torch.view_as_complex(o.clone().reshape(*x.shape, 2)), want) <= TOL
    ctx.close()


@pytest.mark.parametrize("dims,m", [((4, 4, 4, 4), 0.2), ((4, 8, 4, 12), -0.3)])
def test_determinants_of_2x2x2x2_blocks(dims, m):
    U = synth.gauge_field(dims, 0.3, seed=7)
    ctx = binding.Context(dims, (2,) * 4)
    ctx.load_gauge(U)
    ctx.set_params(1.4, 0.12, 0.07, antiperiodic_t=True)
    ld, sg = ctx.block_logdet(m)
    lat = oc.Lattice(dims, (2,) * 4, U, 1.4)
    col = lat.colour()
    shape = synth.spinor_field(dims, seed=1).shape[-3:]
    x = np.indices(dims).reshape(4, -1)
    blk = np.zeros(x.shape[1], dtype=int)
    loc = np.zeros(x.shape[1], dtype=int)
    for mu in range(4):
        blk = blk * (dims[mu] // 2) + x[mu] // 2
        loc = loc * 2 + x[mu] % 2
    nblk = blk.max() + 1
    dense = np.zeros((nblk, 192, 192), dtype=complex)
    for j in range(192):
        e = np.zeros((col.size, 12), dtype=complex)
        e[loc == j // 12, j % 12] = 1.0
        for c in (0, 1):
            out = lat.apply(m, np.where((col.reshape(-1) == c)[:, None], e, 0).reshape(shape), rows=c, cols=c).reshape(-1, 12)
            for s in np.flatnonzero(col.reshape(-1) == c):
                dense[blk[s], 12 * loc[s]:12 * loc[s] + 12, j] = out[s]
    sign, want = np.linalg.slogdet(dense)
    assert np.max(np.abs(np.sort(ld) - np.sort(want))) <= 1e-10
    assert np.prod(sg) == np.round(np.prod(sign).real)
    ctx.close()


def test_inverses_of_a_mass_after_a_new_configuration():
    """A mass used before load_gauge finds its in-block inverses made for the new links."""
    dims, b = (8, 8, 8, 8), synth.spinor_field((8, 8, 8, 8), seed=9)
    old, new = context(dims, 4, seed=3), context(dims, 4, seed=11)
    its = []
    for ctx in (old, new):
        x = np.zeros_like(b)
        ctx.set_solver(binding.FP64, tol_outer=1e-11, tol_block=1e-12)
        if ctx is old:
            for m in (0.3, 0.2):
                ctx.solve_D(m, b, x)
            ctx.load_gauge(synth.gauge_field(dims, 0.3, seed=11))
        for m in (0.3, 0.12, 0.2):
            its.append(ctx.solve_D(m, b, x)["iters_outer"])
            y = np.zeros_like(b)
            ctx.apply_D(m, x, y)
            assert np.linalg.norm(y - b) <= 1.01e-11 * np.linalg.norm(b)
    assert its[:3] == its[3:]
    old.close()
    new.close()


@pytest.mark.parametrize("prec", [binding.FP64, binding.MIXED_FP32, binding.MIXED_FP16])
@pytest.mark.parametrize("dims,l", [((4, 4, 4, 4), 2), ((12, 12, 12, 12), 6), ((16, 16, 16, 16), 4)])
def test_residuals_with_a_zero_right_hand_side(dims, l, prec):
    """Five right-hand sides, one of them zero, one tiny: each reaches its own tolerance, as the operator sees it
    (whose rounding is below 1e-14), with the inner products fused, separate and as the context chooses."""
    ctx = context(dims, l)
    b = synth.spinor_field(dims, seed=13, nrhs=5)
    b[1] = 0
    b[3] *= 2.0 ** -40
    ctx.set_solver(prec, tol_outer=1e-10, tol_block=1e-12)
    for fuse in (None, True, False):
        if fuse is not None:
            ctx.fuse_reductions(fuse)
        x, y = np.ones_like(b), np.zeros_like(b)
        ctx.solve_D(0.12, b, x, nrhs=5)
        ctx.apply_D(0.12, x, y, nrhs=5)
        for r in range(5):
            assert np.linalg.norm(y[r] - b[r]) <= (1e-10 + 1e-14) * np.linalg.norm(b[r])
        assert np.max(np.abs(x[1])) == 0.0
    ctx.close()


@pytest.mark.parametrize("dims,l,n", [((4, 4, 4, 8), 2, 3), ((8, 8, 8, 8), 4, 1), ((12, 12, 12, 12), 6, 2), ((16, 16, 16, 16), 8, 1)])
def test_force_block_solves_of_every_length(dims, l, n):
    """The force with FP32 inner solves against FP64 ones: block residuals of 1e-12, magnified by 1 / (m1 - m2) = 20 and
    a condition number of order ten."""
    ctx = context(dims, l)
    dU = []
    for prec, tol in ((binding.MIXED_FP32, 1e-12), (binding.FP64, 1e-13)):
        ctx.set_solver(prec, tol_outer=1e-11, tol_block=tol)
        u = torch.empty((int(np.prod(dims)), 4, 8), dtype=torch.float64, device="cuda")
        ctx.force(n, seed=5, dU=u)
        dU.append(u.clone())
    assert rel(dU[0], dU[1]) <= 1e-9
    ctx.close()


@pytest.mark.parametrize("antiperiodic", [False, True])
def test_apply_D_one_thread_per_site_on_2x2x2x2_blocks(antiperiodic):
    """12288 site updates: beyond the split kernel's range with the smallest blocks."""
    test_apply_D_layouts_and_block_hops((8, 8, 8, 8), 2, 3, antiperiodic)


# half lattices that are multiples of 256 sites: the size rule fuses all of these
@pytest.mark.parametrize("dims,l,nrhs", [((8, 8, 8, 8), 2, 3), ((24, 12, 12, 12), 6, 5), ((16, 16, 16, 16), 8, 1)])
def test_fused_inner_products_of_every_block_length(dims, l, nrhs):
    """The fused stencils ran (the report of tuned shapes lists them), and the solves reach their tolerance as the
    operator sees it."""
    ctx = context(dims, l)
    b = synth.spinor_field(dims, seed=13, nrhs=nrhs)
    ctx.set_solver(binding.MIXED_FP32, tol_outer=1e-10, tol_block=1e-12)
    for fuse in (-1, False, True):
        ctx.autotune(True)
        ctx.fuse_reductions(fuse)
        x, y = np.zeros_like(b), np.zeros_like(b)
        ctx.solve_D(0.12, b, x, nrhs=nrhs)
        ctx.apply_D(0.12, x, y, nrhs=nrhs)
        for r in range(nrhs):
            assert np.linalg.norm(y[r] - b[r]) <= (1e-10 + 1e-14) * np.linalg.norm(b[r])
        report = ctx.autotune_report()
        assert ("red=1" in report and "red=2" in report) == (fuse is not False)
    ctx.close()


@pytest.mark.parametrize("l", [2, 4])
def test_determinants_of_a_nan_link_and_of_singular_blocks(l):
    """Shared memory (l = 2) and dense (l = 4) determinants answer both with DDRW_ENUMERIC."""
    dims = (8, 8, 8, 8)
    U = synth.gauge_field(dims, 0.3, seed=3)
    U[100, 2, 1, 1] = np.nan
    for links, csw, m in ((U, 1.4, 0.1), (synth.gauge_field(dims, 0.3, seed=3), 0.0, -4.0)):  # A = 4 + m = 0
        ctx = binding.Context(dims, (l,) * 4)
        ctx.load_gauge(links)
        ctx.set_params(csw, 0.12, 0.07)
        with pytest.raises(binding.DDRWError) as e:
            ctx.block_logdet(m)
        assert e.value.status == 5
        ctx.close()
