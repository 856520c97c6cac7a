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
