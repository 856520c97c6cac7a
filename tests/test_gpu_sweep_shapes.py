"""V-cycles at the edges of the column sweep's shapes, against the oracle, element by element.

The FP32 sweep of levels of 800k cells or more runs on tensor-copy tiles of up to 32 columns of
a row (8 to 80 levels, two groups of chunks); smaller levels and columns of more than 80 levels run
on register chunks of 5, 8 or 10 levels, FP64 sweeps on chunks of 5, 10 or 16.  Tolerances as for the other large levels: 1e-6 of the
largest element in FP32 (rounding reaches the V-cycle at a few 1e-7), 1e-11 in FP64."""
import numpy as np
import pytest

import synthetic as syn

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def mg():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2002_00756_gb300.build import build
    build()
    import paper_2002_00756_gb300 as m
    m.load()
    return m


@pytest.mark.parametrize("n,nlev,levels,precision", [
    (66, 35, 2, "fp32"),     # ragged tiles (24, 24, 18 columns), odd level count, odd coarse n
    (130, 8, 2, "fp32"),     # fewest levels of the tiles, five tiles to a row
    (44, 71, 2, "fp32"),     # more than 70 levels: chunks of 8
    (48, 80, 3, "fp32"),     # most levels of the tiles
    (33, 81, 1, "fp32"),     # taller columns: register chunks of 8; odd n, no coarse level
    (20, 128, 2, "fp64"),
    (90, 41, 2, "fp64"),     # FP64 chunks of 10
    (90, 41, 2, "fp32_p64"),
    (92, 40, 2, "fp32_p64"),
])
def test_vcycle_shapes(mg, n, nlev, levels, precision):
    from oracle.problem import pressure_hierarchy
    cfg = syn.small_config(n, nlev, levels=levels, seed=syn.BASE_SEED + 700 + n)
    inp = syn.make_inputs(cfg)
    ref = pressure_hierarchy(cfg, inp).vcycle(inp["rhs"], cfg.omega, cfg.n_pre, cfg.n_post, cfg.n_coarse).ravel()
    h = mg.mg_setup_config(cfg, inp, precision=precision)
    x = torch.full((cfg.ncell,), float("nan"), dtype=torch.float64, device="cuda")
    mg.vcycle(h, torch.from_numpy(inp["rhs"]).cuda(), x)
    err = float(np.max(np.abs(x.cpu().numpy() - ref)) / np.max(np.abs(ref)))
    print(f"C{n}L{nlev} {precision} V-cycle: worst element {err:.3e} of max")
    assert err <= (1e-11 if precision == "fp64" else 1e-6)
    h.destroy()


@pytest.mark.parametrize("precision", ["fp32", "fp32_p64", "fp32_bf16"])
@pytest.mark.parametrize("n,nlev", [(24, 30), (20, 9), (66, 35)])
def test_both_forms_of_the_sweep_agree_bit_for_bit(mg, n, nlev, precision):
    """Tensor-copy tiles and register chunks round alike: whichever the tuner picks per level, the
    V-cycle's bits stay (n not a multiple of 4 or 8, odd level counts, prolongation across edges)."""
    cfg = syn.small_config(n, nlev, levels=2, seed=syn.BASE_SEED + 730 + n)
    inp = syn.make_inputs(cfg)
    h = mg.mg_setup_config(cfg, inp, precision=precision)
    b = torch.from_numpy(inp["rhs"]).cuda()
    x0, x1 = torch.empty_like(b), torch.empty_like(b)
    mg.vcycle(h, b, x0)
    for _ in range(2):
        mg.mg_autotune(h)
        mg.vcycle(h, b, x1)
        assert torch.equal(x0, x1)
    h.destroy()


@pytest.mark.parametrize("n,nlev,levels", [(2, 1, 1), (5, 3, 1), (10, 19, 2), (44, 71, 2)])
def test_recurred_residual_is_the_true_one(mg, n, nlev, levels):
    """The fused apply's units (32 columns by up to 18 levels; one level, a ragged last group of
    columns, a ragged last run of levels) add up: the solve's own residual norm is that of b - A x.
    They drift apart by a few eps ||A|| ||x|| per iteration, ||A|| ~ 1e3 here: 1e-10 of ||b|| at most."""
    cfg = syn.small_config(n, nlev, levels=levels, seed=syn.BASE_SEED + 760 + n)
    inp = syn.make_inputs(cfg)
    h = mg.mg_setup_config(cfg, inp)
    b = torch.from_numpy(inp["rhs"]).cuda()
    x, y = torch.empty_like(b), torch.empty_like(b)
    for tol in (1e-3, 1e-7):
        info = mg.pressure_solve(h, b, x, tol)
        mg.helmholtz_apply(h, x, y)
        true = float((b - y).norm() / b.norm())
        assert info.converged and abs(true - info.rel_res) <= 1e-10, (info, true)
    h.destroy()


@pytest.mark.parametrize("n,nlev,levels,rotation", [(10, 19, 1, 0.0), (10, 19, 1, 7.292e-5), (44, 37, 2, 7.292e-5)])
def test_recurred_mixed_residual_is_the_true_one(mg, n, nlev, levels, rotation):
    """The fused mixed operator (units of 32 faces or cells by a run of levels) and its sums: the solve's own
    residual norm is that of b - A x, with ||A|| ~ 2e3 again within 1e-10 of ||b||."""
    cfg = syn.small_config(n, nlev, levels=levels, seed=syn.BASE_SEED + 780 + n, mixed=True,
                           consistent_mass=rotation != 0.0, rotation=rotation)
    inp = syn.make_inputs(cfg)
    h = mg.mg_setup_config(cfg, inp)
    b = [torch.from_numpy(inp[k]).cuda().ravel() for k in ("rhs_u", "rhs_p")]
    x, y = [torch.empty_like(v) for v in b], [torch.empty_like(v) for v in b]
    for tol in (1e-3, 1e-7):
        info = mg.mixed_solve(h, *b, *x, tol=tol)
        mg.mixed_apply(h, *x, *y)
        true = float(torch.cat([v - w for v, w in zip(b, y)]).norm() / torch.cat(b).norm())
        assert info.converged and abs(true - info.rel_res) <= 1e-10, (info, true)
    h.destroy()


def test_degenerate_right_hand_sides_leave_no_trace(mg):
    """A solve launches its first iteration before it knows <b, b>: a zero right-hand side still converges
    at once with x = 0, a NaN still breaks down, and the next solve gives the bits of the first."""
    cfg = syn.small_config(10, 19, levels=2, seed=syn.BASE_SEED + 790)
    inp = syn.make_inputs(cfg)
    h = mg.mg_setup_config(cfg, inp)
    b = torch.from_numpy(inp["rhs"]).cuda().ravel()
    ref, x = torch.empty_like(b), torch.empty_like(b)
    first = mg.pressure_solve(h, b, ref, 1e-9)
    assert first.converged
    for bad in (torch.zeros_like(b), torch.where(torch.arange(b.numel(), device="cuda") == 5, float("nan"), b)):
        x.fill_(1.0)
        info = mg.pressure_solve(h, bad, x, 1e-9)
        assert info.converged == bool(torch.all(bad == 0)) and info.iters == 0 and float(x.abs().max()) == 0.0
        info = mg.pressure_solve(h, b, x, 1e-9)
        assert (info.status, info.iters, info.rel_res) == (first.status, first.iters, first.rel_res)
        assert torch.equal(x, ref)
    h.destroy()


@pytest.mark.parametrize("side", [0, 3, 4])
@pytest.mark.parametrize("factor,ok", [(1 + 3e-11, True), (1 - 9e-11, True), (1 + 1.2e-10, False), (1 - 1e-9, False),
                                       (0.0, False), (-1.0, False), (float("inf"), False), (float("nan"), False)])
def test_flux_symmetry_is_held_to_1e_10(mg, side, factor, ok):
    """Products within 2^18 units in the last place (5.8e-11) pass on their words, others by comparison: either
    way 1e-10 of the larger decides, and signs and non-finite values are refused."""
    from oracle.problem import pressure_hierarchy
    cfg = syn.small_config(4, 6, seed=syn.BASE_SEED + 795)
    inp = syn.make_inputs(cfg)
    a = np.array(pressure_hierarchy(cfg, inp).levels[0].couplings())
    a[side, 2, 5] *= factor
    h = mg.mg_setup_config(cfg, inp)
    if ok:
        mg.mg_set_coefficients(h, torch.from_numpy(a).cuda())
    else:
        with pytest.raises(mg.MGError):
            mg.mg_set_coefficients(h, torch.from_numpy(a).cuda())
    h.destroy()


def test_smoothing_of_misaligned_vectors(mg):
    """Vectors that start on an odd double (8-byte alignment only) give what aligned ones give."""
    cfg = syn.small_config(20, 9, levels=3, seed=syn.BASE_SEED + 720)
    inp = syn.make_inputs(cfg)
    h = mg.mg_setup_config(cfg, inp)
    buf = [torch.zeros(cfg.ncell + 1, dtype=torch.float64, device="cuda") for _ in range(4)]
    b, x = torch.from_numpy(inp["rhs"]).cuda(), torch.from_numpy(syn.normal(8, 0, cfg.ncell)).cuda()
    buf[0][1:].copy_(b)
    buf[1][1:].copy_(x)
    out = torch.empty_like(b)
    for start, odd in ((None, None), (x, buf[1][1:])):
        mg.mg_smooth(h, 0, b, start, out, 2)
        mg.mg_smooth(h, 0, buf[0][1:], odd, buf[2][1:], 2)
        assert float((out - buf[2][1:]).norm()) <= 1e-13 * float(out.norm())
    nc = h.level_cells(1)
    bc, bo = torch.empty(nc, dtype=torch.float64, device="cuda"), torch.zeros(nc + 1, dtype=torch.float64, device="cuda")
    mg.mg_residual_restrict(h, 0, b, x, bc)
    mg.mg_residual_restrict(h, 0, buf[0][1:], buf[1][1:], bo[1:])
    assert float((bc - bo[1:]).norm()) <= 1e-13 * float(bc.norm())
    h.destroy()
