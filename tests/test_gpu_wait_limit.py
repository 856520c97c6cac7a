"""The bounded waits of the tensor-copy sweeps, made to run out by a limit of a few polls (no copy is
dropped and nothing hangs: a sweep that gives up goes on without new copies, yields NaN and waits for
those in flight before it ends)."""
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


def setup(mg, n, nlev, precision):
    cfg = syn.small_config(n, nlev, levels=2, seed=syn.BASE_SEED + 810 + n)
    inp = syn.make_inputs(cfg)
    return mg.mg_setup_config(cfg, inp, precision=precision), torch.from_numpy(inp["rhs"]).cuda().ravel()


# finest levels on tiles: several tiles a block, full chunks (70 levels) and short ones
TILED = [(66, 35, "fp32"), (96, 70, "fp32"), (66, 41, "fp32_bf16"), (66, 41, "fp32_p64"), (64, 80, "fp32")]


@pytest.mark.parametrize("n,nlev,precision", TILED)
def test_a_wait_that_runs_out_gives_nan_and_a_status(mg, n, nlev, precision):
    h, b = setup(mg, n, nlev, precision)
    ref, x = torch.empty_like(b), torch.zeros_like(b)
    mg.vcycle(h, b, ref)
    lib = mg.load()
    assert lib.mg_inject_wait_limit(h.ptr, 0) == mg.MG_OK
    mg.vcycle(h, b, x)
    assert bool(torch.isnan(x).all())
    with pytest.raises(mg.MGError) as e:
        mg.pressure_solve(h, b, x, 1e-8)
    assert e.value.status == mg.MG_ERR_TIMEOUT
    # a single poll: some copies are late, others are not, and no late one goes unseen
    assert lib.mg_inject_wait_limit(h.ptr, 1) == mg.MG_OK
    for _ in range(3):
        mg.vcycle(h, b, x)
        assert bool(torch.isnan(x).any()) or torch.equal(x, ref)
    assert lib.mg_inject_wait_limit(h.ptr, -1) == mg.MG_OK
    mg.vcycle(h, b, x)
    assert torch.equal(x, ref)
    h.destroy()


def test_every_kind_of_solve_reports_it_and_the_next_one_is_clean(mg):
    h, b = setup(mg, 66, 35, "fp32")
    h2, b2 = setup(mg, 10, 9, "fp32")   # (no level on tiles: no copy to wait for)
    ref, x, x2 = torch.empty_like(b), torch.empty_like(b), torch.empty_like(b2)
    first = mg.pressure_solve(h, b, ref, 1e-8)
    mg.mg_set_pressure_solver(h, "bicgstab_mg", eps=1e-6)
    lib = mg.load()
    assert lib.mg_inject_wait_limit(h.ptr, 0) == mg.MG_OK
    e = mg.Ensemble([h2, h], [b2, b], [x2, x], 1e-8)
    for call in (lambda: mg.pressure_solve(h, b, x, 1e-8), lambda: mg.pressure_solve_adjoint(h, b, x, 1e-8),
                 lambda: mg.helmholtz_solve(h, b, x), lambda: e.solve(),
                 lambda: mg.ensemble_pressure_solve([h2, h], [b2, b], [x2, x], 1e-8)):
        with pytest.raises(mg.MGError) as err:
            call()
        assert err.value.status == mg.MG_ERR_TIMEOUT
    e.destroy()
    assert lib.mg_inject_wait_limit(h.ptr, -1) == mg.MG_OK
    # a breakdown of its own (the FP32 V-cycle overflows) is called one, in every kind of solve
    e = mg.Ensemble([h2, h], [b2, b * 1e100], [x2, x], 1e-8)
    assert [i.status for i in e.solve()] == [mg.MG_OK, mg.MG_ERR_BREAKDOWN]
    e.destroy()
    assert mg.pressure_solve(h, b * 1e100, x, 1e-8).status == mg.MG_ERR_BREAKDOWN
    assert mg.helmholtz_solve(h, b * 1e100, x).status == mg.MG_ERR_BREAKDOWN
    again = mg.pressure_solve(h, b, x, 1e-8)
    assert (again.status, again.iters, again.rel_res) == (first.status, first.iters, first.rel_res)
    assert torch.equal(x, ref)
    h.destroy()
    h2.destroy()
