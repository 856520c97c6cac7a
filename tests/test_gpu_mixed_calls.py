"""Single calls on the mixed system: rounding, and results in place of operands."""
import numpy as np
import pytest
import scipy.sparse as sp

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


def test_the_face_weights_cost_one_unit_in_the_last_place(mg):
    """A^T [u; 0] = S J A-hat J S^-1 [u; 0] with a unit velocity mass is u in its velocity rows: W (u / W),
    two correctly rounded operations, so within (1 + 2^-53)^2 - 1 < 2^-52 (1 + 2^-53) of u."""
    cfg = syn.small_config(24, 20, levels=1, seed=syn.BASE_SEED + 870, mixed=True, eps=0.0)
    inp = syn.make_inputs(cfg)
    h = mg.mg_setup_config(cfg, inp)
    u = torch.from_numpy(syn.normal(cfg.seed, 0, h.nu)).cuda()
    p = torch.zeros(h.ncell, dtype=torch.float64, device="cuda")
    yu, yp = torch.empty_like(u), torch.empty_like(p)
    mg.mixed_apply_transpose(h, u, p, yu, yp)
    ulps = ((yu - u) / u).abs() / 2.0 ** -52   # (exact difference, a power of two; the quotient rounds once)
    assert float(ulps.max()) <= 1.0 + 1e-15
    h.destroy()


def test_the_transposed_mass_costs_three_roundings(mg):
    """Where a face's transposed mass row meets one non-zero velocity, u = 1, its result is the mass entry
    1 / 6 over W times W, each rounded: within three roundings, whatever the errors of W itself."""
    from oracle.problem import mixed_problem
    cfg = syn.small_config(24, 20, levels=1, seed=syn.BASE_SEED + 875, mixed=True, eps=0.0, consistent_mass=True)
    inp = syn.make_inputs(cfg)
    S, _ = mixed_problem(cfg, inp)
    h = mg.mg_setup_config(cfg, inp)
    nh = S.nh
    u = np.zeros(h.nu)
    u[::97] = 1.0
    uh, uv = u[:nh].reshape(cfg.nlev, -1), u[nh:].reshape(cfg.nlev + 1, -1)
    uv[0] = uv[-1] = 0.0
    off = (S.Mh != 0).astype(float).T - sp.identity(S.nhf)   # faces coupled to each other
    ch = np.stack([off @ uh[k] for k in range(cfg.nlev)])
    cv = np.zeros_like(uv)
    cv[1:-1] = uv[:-2] + uv[2:]
    one = np.concatenate([((ch == 1) & (uh == 0)).ravel(), ((cv == 1) & (uv == 0)).ravel()])
    assert one.sum() > 1000
    d = [torch.from_numpy(a).cuda() for a in (u, np.zeros(h.ncell))]
    yu, yp = torch.empty_like(d[0]), torch.empty_like(d[1])
    mg.mixed_apply_transpose(h, *d, yu, yp)
    got = np.abs(yu.cpu().numpy()[one])
    assert np.max(np.abs(got - 1 / 6)) <= 3 * (1 + 2.0 ** -50) * 2.0 ** -53 / 6
    h.destroy()


@pytest.mark.parametrize("n,nlev,consistent", [(10, 19, False), (48, 30, True)])
def test_pressure_rows_in_place(mg, n, nlev, consistent):
    """mixed_apply with yp = p, and the Schur-complement step in place of its right-hand side, give the bits
    of separate arrays."""
    cfg = syn.small_config(n, nlev, levels=1, seed=syn.BASE_SEED + 880, mixed=True, consistent_mass=consistent)
    inp = syn.make_inputs(cfg)
    h = mg.mg_setup_config(cfg, inp)
    u, p = (torch.from_numpy(inp[k]).cuda().ravel() for k in ("rhs_u", "rhs_p"))
    yu, yp, zu, zp = torch.empty_like(u), torch.empty_like(p), torch.empty_like(u), p.clone()
    mg.mixed_apply(h, u, p, yu, yp)
    mg.mixed_apply(h, u, zp, zu, zp)
    assert torch.equal(yu, zu) and torch.equal(yp, zp)
    mg.schur_precond(h, u, p, yu, yp)
    zu, zp = u.clone(), p.clone()
    mg.schur_precond(h, zu, zp, zu, zp)
    assert torch.equal(yu, zu) and torch.equal(yp, zp)
    h.destroy()
