"""A zero right-hand side costs no iteration."""
import time

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


@pytest.mark.parametrize("mixed", [False, True])
def test_zero_right_hand_side(mg, mixed):
    """Its only work is the start of the solve: one recorded launch, and less than
    half the time of one iteration of an ordinary solve (C96L70, mixed C48L30: 0.15 and 0.3 of one)."""
    cfg = syn.small_config(48 if mixed else 96, 30 if mixed else 70, levels=4, seed=syn.BASE_SEED + 890, mixed=mixed)
    inp = syn.make_inputs(cfg)
    h = mg.mg_setup_config(cfg, inp, precision="fp32")
    b = [torch.from_numpy(inp[k]).cuda().ravel() for k in (("rhs_u", "rhs_p") if mixed else ("rhs",))]
    zero, x = [torch.zeros_like(v) for v in b], [torch.empty_like(v) for v in b]
    solve = mg.mixed_solve if mixed else mg.pressure_solve

    def run(rhs):
        t = []
        for _ in range(15):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            info = solve(h, *rhs, *x, tol=1e-8)
            torch.cuda.synchronize()
            t.append(time.perf_counter() - t0)
        return info, float(np.median(t))

    full, t_full = run(b)
    none, t_none = run(zero)
    assert full.converged and none.converged and none.iters == 0 and all(float(v.abs().max()) == 0.0 for v in x)
    mg.mg_profile_start(h, 256)
    solve(h, *zero, *x, tol=1e-8)
    assert len(mg.mg_profile_stop(h)) == 1
    assert t_none < 0.5 * t_full / full.iters + 30e-6, (t_none, t_full / full.iters)
    again, _ = run(b)
    assert (again.iters, again.rel_res) == (full.iters, full.rel_res)
    h.destroy()
