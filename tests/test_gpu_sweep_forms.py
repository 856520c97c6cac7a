"""The launch forms of the column kernels: what the autotuner keeps, and that every form agrees."""
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


def setup(mg, n, nlev, levels, precision, **kw):
    cfg = syn.small_config(n, nlev, levels=levels, seed=syn.BASE_SEED + 850 + n, **kw)
    inp = syn.make_inputs(cfg)
    return cfg, inp, mg.mg_setup_config(cfg, inp, precision=precision), torch.from_numpy(inp["rhs"]).cuda().ravel()


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_tuning_does_not_slow_the_restriction_down(mg, precision):
    """C48L30, whose built-in restriction takes one level per thread (half the time of eight): the tuner
    keeps it, unless one of its own numbers measures faster.  Times within 25 % (events around launches
    of some 10 us)."""
    _, _, h, b = setup(mg, 48, 30, 3, precision)
    x = torch.empty_like(b)

    def restrictions():
        out = []
        for level in (0, 1):
            mg.mg_profile_start(h, 256, "restrict", level)
            for _ in range(60):
                mg.vcycle(h, b, x)
            out.append(float(np.median([r["ms"] for r in mg.mg_profile_stop(h)])))
        return out

    restrictions()
    before = restrictions()
    mg.mg_autotune(h)
    after = restrictions()
    assert all(t <= 1.25 * s for s, t in zip(before, after)), (before, after)
    h.destroy()


@pytest.mark.parametrize("omega", [0.0, 1e-310, 1e-200, 1e300])
def test_line_relaxation_has_its_own_omega(mg, omega):
    """The FP64 factors hold the V-cycle's relaxation factor; a pressure solver with another one gives what a
    handle set up with that one gives, also where the quotient of the two is out of range.  Three roundings
    per level of 9: 1e-13 of the largest element."""
    cfg = syn.small_config(10, 9, levels=2, seed=syn.BASE_SEED + 860)
    inp = syn.make_inputs(cfg)
    x = []
    for om in (0.8, omega):
        h = mg.mg_setup(cfg.n, cfg.nlev, inp["z_if"], inp["g"], levels=2, omega=om)
        mg.mg_set_pressure_solver(h, "jacobi", omega=0.8, sweeps=3)
        b = torch.from_numpy(inp["rhs"]).cuda().ravel()
        x.append(torch.empty_like(b))
        mg.helmholtz_solve(h, b, x[-1])
        h.destroy()
    assert float((x[0] - x[1]).abs().max()) <= 1e-13 * float(x[0].abs().max())


def vcycle_time(mg, n, nlev):
    _, _, h, b = setup(mg, n, nlev, 3, "fp32")
    x, t = torch.empty_like(b), []
    for _ in range(12):
        e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
        e[0].record()
        mg.vcycle(h, b, x)
        e[1].record()
        torch.cuda.synchronize()
        t.append(e[0].elapsed_time(e[1]))
    h.destroy()
    return float(np.median(t))


def test_short_columns_cost_no_more_than_longer_ones(mg):
    """C256L6 in chunks cut to its columns against twice the levels (0.8 of
    its time; 1.37 with chunks of 10)."""
    assert vcycle_time(mg, 256, 6) <= 1.0 * vcycle_time(mg, 256, 12)


def test_tall_columns_run_on_tiles(mg):
    """C128L100 against C128L80, 1.25 times the cells: no change to a form of half the rate (1.4
    times the time; 2.0 on register chunks)."""
    assert vcycle_time(mg, 128, 100) <= 1.7 * vcycle_time(mg, 128, 80)


@pytest.mark.parametrize("precision", ["fp64", "fp32", "fp32_p64"])
@pytest.mark.parametrize("n,nlev", [(10, 20), (12, 3), (96, 41), (24, 90)])
def test_a_cycle_of_one_sweep_is_one_launch(mg, n, nlev, precision):
    """One level, one sweep from zero: FP64 in, FP64 out, no copy of b and no conversion."""
    from oracle.problem import pressure_hierarchy
    cfg, inp, h, b = setup(mg, n, nlev, 1, precision, n_coarse=1)
    x = torch.full_like(b, float("nan"))
    mg.mg_profile_start(h, 16)
    mg.vcycle(h, b, x)
    assert [r["kind"] for r in mg.mg_profile_stop(h)] == ["sweep"]
    ref = pressure_hierarchy(cfg, inp).vcycle(inp["rhs"], cfg.omega, cfg.n_pre, cfg.n_post, 1).ravel()
    err = float(np.max(np.abs(x.cpu().numpy() - ref)) / np.max(np.abs(ref)))
    assert err <= (1e-11 if precision == "fp64" else 1e-6), err
    h.destroy()


def launch_times(mg, n, nlev, kind, variant=0, **kw):
    _, _, h, b = setup(mg, n, nlev, 2, "fp32", **kw)
    x, t = torch.empty_like(b), []
    mg.vcycle(h, b, x)
    mg.mg_profile_start(h, 4096, kind, 0)
    for _ in range(15):
        mg.vcycle(h, b, x)
    t = [r["ms"] for r in mg.mg_profile_stop(h) if r["variant"] == variant]
    h.destroy()
    return float(np.median(t))


def test_prolongation_onto_a_level_without_sweeps(mg):
    """C192L60 without any sweeps on the finest level: the prolongation writes 9 bytes per cell, the restriction of
    b reads 5; 1.3 times its time (2.7 with a thread per cell, each with the divisions that find its parent)."""
    kw = dict(n_pre=0, n_post=0)
    assert launch_times(mg, 192, 60, "prolong", **kw) <= 1.9 * launch_times(mg, 192, 60, "restrict", **kw)


@pytest.mark.parametrize("n,nlev", [(10, 9), (96, 20)])
@pytest.mark.parametrize("n_pre,n_post", [(0, 0), (2, 0), (0, 2)])
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_cycles_without_sweeps_on_one_side(mg, n, nlev, n_pre, n_post, precision):
    """The levels' plain copies and prolongations, one level per thread and eight, against the oracle."""
    from oracle.problem import pressure_hierarchy
    cfg, inp, h, b = setup(mg, n, nlev, 2, precision, n_pre=n_pre, n_post=n_post)
    ref = pressure_hierarchy(cfg, inp).vcycle(inp["rhs"], cfg.omega, n_pre, n_post, cfg.n_coarse).ravel()
    x = torch.full_like(b, float("nan"))
    mg.vcycle(h, b, x)
    err = float(np.max(np.abs(x.cpu().numpy() - ref)) / np.max(np.abs(ref)))
    assert err <= (1e-11 if precision == "fp64" else 1e-6), err
    h.destroy()


def test_a_sweep_from_the_prolongation_alone_runs_on_tiles(mg):
    """C128L70 without sweeps before the coarse correction: the first sweep after it reads less than a plain one
    and takes about its time (twice that on register chunks)."""
    first, plain = (launch_times(mg, 128, 70, "sweep", v, n_pre=0) for v in (3, 0))
    assert first <= 1.3 * plain, (first, plain)


def test_short_columns_that_chunks_hold_without_waste(mg):
    """C256L8 in registers (a chunk of 4 per half) against C256L10 on tiles: 0.7 of its time (as much of it on tiles,
    whose chunks of 7 would be half empty)."""
    assert launch_times(mg, 256, 8, "sweep") <= 0.85 * launch_times(mg, 256, 10, "sweep")


def forced(mg, h, form, kc=0):
    mg.mg_apply_choices(h, [(form, kc, 0)] * h.levels)


# n not a multiple of 4 or 8, single tiles and several; 8 levels, both ends of the chunks of 7, 8 and 10,
# short columns (chunks of 1 to 4, four groups a block), levels above and below 2M cells
FORMS = [(2, 8, 1), (6, 8, 2), (10, 9, 2), (20, 30, 2), (24, 70, 3), (50, 71, 2), (33, 80, 1), (26, 81, 2), (34, 128, 2), (92, 41, 2),
         (66, 80, 2), (64, 128, 2)]


@pytest.mark.parametrize("precision", ["fp32", "fp32_p64", "fp32_bf16"])
@pytest.mark.parametrize("n,nlev,levels", FORMS)
def test_tiles_and_register_chunks_agree_bit_for_bit(mg, n, nlev, levels, precision):
    """Each form forced on every level: the same rounding, so the same V-cycle (sweeps from zero, plain,
    with prolongation across panel edges); and any number of levels per thread of the restriction."""
    _, _, h, b = setup(mg, n, nlev, levels, precision)
    x, y = torch.full_like(b, float("nan")), torch.full_like(b, float("nan"))
    forced(mg, h, 64)
    mg.vcycle(h, b, x)
    forced(mg, h, 128, 3)
    mg.vcycle(h, b, y)
    assert torch.equal(x, y)
    forced(mg, h, 0)
    mg.vcycle(h, b, y)
    assert torch.equal(x, y)
    h.destroy()
    _, _, h, b = setup(mg, n, nlev, levels, precision, n_pre=0)   # (a sweep from the prolongation alone)
    forced(mg, h, 64)
    mg.vcycle(h, b, x)
    forced(mg, h, 128)
    mg.vcycle(h, b, y)
    assert torch.equal(x, y)
    h.destroy()


@pytest.mark.parametrize("n,nlev,levels,precision,kw", [
    (92, 41, 2, "fp64", {}),                   # FP64 chunks of 10, uneven: products of 8 and 9 levels
    (96, 43, 2, "fp64", {}),
    (96, 41, 2, "fp32", dict(n_pre=0)),        # chunks in registers, from a prolongation alone
    (80, 81, 2, "fp32", {}),                   # tall tiles
    (52, 128, 2, "fp32", {}),
    (8, 1, 2, "fp32", {}), (6, 2, 1, "fp32_p64", {}), (10, 3, 2, "fp32", {}), (12, 4, 2, "fp32_p64", {}),
    (10, 5, 2, "fp32_p64", {}), (6, 6, 1, "fp32", {}), (14, 7, 2, "fp32", {}), (10, 8, 2, "fp32_p64", {}),
])
def test_vcycle_against_the_oracle(mg, n, nlev, levels, precision, kw):
    """1e-6 of the largest element in FP32, 1e-11 in FP64, as for the other shapes."""
    from oracle.problem import pressure_hierarchy
    cfg, inp, h, b = setup(mg, n, nlev, levels, precision, **kw)
    ref = pressure_hierarchy(cfg, inp).vcycle(inp["rhs"], cfg.omega, cfg.n_pre, cfg.n_post, cfg.n_coarse).ravel()
    if kw:
        forced(mg, h, 64)
    x = torch.full_like(b, float("nan"))
    mg.vcycle(h, b, x)
    err = float(np.max(np.abs(x.cpu().numpy() - ref)) / np.max(np.abs(ref)))
    assert err <= (1e-11 if precision == "fp64" else 1e-6), err
    h.destroy()


def test_choices_are_checked(mg):
    _, _, h, b = setup(mg, 8, 9, 2, "fp32")
    for bad in ((32, 0, 0), (64, -1, 0), (64, 129, 0), (0, 2 ** 31 - 1, 0)):
        with pytest.raises(mg.MGError):
            mg.mg_apply_choices(h, [(0, 0, 0), bad])
    with pytest.raises(ValueError):
        mg.mg_apply_choices(h, [(0, 0, 0)])
    mg.mg_apply_choices(h, mg.mg_autotune(h))
    h.destroy()


@pytest.mark.parametrize("a", [0.0, 1.0, 1e20, 1e29, 1e31, 1e40, 1e200])
def test_pivots_of_any_size(mg, a):
    """One level of C1, whose six cells are alike and whose couplings all equal a: a sweep from zero is
    omega b / (1 + 4 a).  Seven roundings (weights, sum, reciprocal, products) and the weights' own: 1e-15,
    below and above the range in which the reciprocal starts from FP32 (1e30)."""
    h = mg.mg_setup(1, 1, [0.0, 1000.0], np.ones(6), levels=1)
    coef = torch.zeros((6, 6), dtype=torch.float64, device="cuda")
    coef[:4] = a
    mg.mg_set_coefficients(h, coef.ravel())
    b = torch.from_numpy(syn.normal(5, 0, 6)).cuda()
    x = torch.empty_like(b)
    mg.mg_smooth(h, 0, b, None, x, 1)
    ref = 0.8 * b.cpu().numpy() / (1.0 + 4.0 * a)
    assert np.max(np.abs(x.cpu().numpy() / ref - 1.0)) <= 1e-15
    h.destroy()
