"""What a handle holds and what its set-up does."""
import threading

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


def device_bytes(mg, n, nlev, precision):
    cfg = syn.small_config(n, nlev, levels=1, seed=syn.BASE_SEED + 900, gcr_restart=1)
    inp = syn.make_inputs(cfg)
    mg.mg_setup_config(cfg, inp, precision=precision).destroy()   # (the module's own memory)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    h = mg.mg_setup_config(cfg, inp, precision=precision)
    used = free - torch.cuda.mem_get_info()[0]
    h.destroy()
    return used, cfg.ncell


def test_padding_of_the_fp32_fields(mg):
    """C64L80 with FP64 elimination, restart 1.  Bytes per cell: faces 24, FP64 iterates 16, operator 56,
    GCR 32, FP64 level data 40; seven FP32 fields and three of FP64 in rows of 96 for 64 cells, 66 rows a
    panel: 52 times 1.547.  248 in all, and 20 allocations of which a 2 MB page may be partly used."""
    used, cells = device_bytes(mg, 64, 80, "fp32_p64")
    assert used <= (24 + 16 + 56 + 32 + 40 + 52 * 1.547) * cells + 20 * 2 ** 21, used / cells


def test_large_fp32_levels_hold_fp64_data_on_demand(mg):
    """C128L30, 2.9M cells, restart 1: 24 + 16 + 56 + 32 bytes per cell and seven FP32 fields padded by 1.27,
    without the 40 of the FP64 level data; 20 allocations as above."""
    used, cells = device_bytes(mg, 128, 30, "fp32")
    assert used <= (24 + 16 + 56 + 32 + 28 * 1.27) * cells + 20 * 2 ** 21, used / cells


@pytest.mark.parametrize("n,nlev", [(24, 30), (128, 30)])
def test_fp64_calls_of_an_fp32_handle(mg, n, nlev):
    """mg_smooth and mg_residual_restrict of an FP32 handle give the bits of an FP64 handle's: at their first call,
    first captured into a graph and called eagerly before and after it is replayed, and after other
    couplings have been set, by the graph as well."""
    cfg = syn.small_config(n, nlev, levels=2, seed=syn.BASE_SEED + 910)
    inp = syn.make_inputs(cfg)
    h = [mg.mg_setup_config(cfg, inp, precision=p) for p in ("fp64", "fp32", "fp32")]
    b, x0 = torch.from_numpy(inp["rhs"]).cuda().ravel(), torch.from_numpy(syn.normal(9, 0, cfg.ncell)).cuda()

    def calls(hd):
        x, bc = torch.empty_like(b), torch.empty(hd.level_cells(1), dtype=torch.float64, device="cuda")
        mg.mg_smooth(hd, 0, b, x0, x, 2)
        mg.mg_residual_restrict(hd, 0, b, x, bc)
        return x, bc

    def same(u, v):
        return all(torch.equal(s, t) for s, t in zip(u, v))

    ref = calls(h[0])
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        out = calls(h[1])
    assert same(calls(h[1]), ref)          # (nothing of the graph has run)
    graph.replay()
    assert same(out, ref) and same(calls(h[1]), ref) and same(calls(h[2]), ref)
    # couplings of another operator: unit ones weighted by the cells' own volumes
    z = np.asarray(inp["z_if"])
    dz = torch.from_numpy(np.diff(z)).cuda()
    area = torch.from_numpy(areas(mg, cfg)).cuda()
    a = torch.zeros((6, cfg.nlev, cfg.ncol), dtype=torch.float64, device="cuda")
    a[:4] = 1e10 / area
    a[4, :-1] = 300.0 / dz[:-1, None]
    a[5, 1:] = 300.0 / dz[1:, None]
    for hd in h:
        mg.mg_set_coefficients(hd, a.ravel())
    other = calls(h[0])
    assert not same(other, ref)
    graph.replay()
    assert same(out, other) and same(calls(h[1]), other) and same(calls(h[2]), other)
    for hd in h:
        hd.destroy()


def areas(mg, cfg):
    from oracle.geometry import Mesh
    return np.asarray(Mesh(cfg.n, syn.make_inputs(cfg)["z_if"], cfg.radius).area).ravel()


@pytest.mark.parametrize("precision", ["fp64", "fp32", "fp32_bf16"])
def test_a_level_takes_few_allocations(mg, precision):
    """Set-up of a small handle is mostly allocations and uploads.  A level's: connectivity, column factors,
    two face forms, FP32 column factors and restriction weights, FP64 level data, and one for all else."""
    lib, count = mg.load(), []
    for levels in (2, 3):
        cfg = syn.small_config(12, 10, levels=levels, seed=syn.BASE_SEED + 920)
        inp = syn.make_inputs(cfg)
        lib.mg_inject_alloc_failure(0)
        h = mg.mg_setup_config(cfg, inp, precision=precision)
        count.append(lib.mg_inject_alloc_failure(0))
        h.destroy()
    assert count[1] - count[0] <= 8, count


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_a_refused_set_of_couplings_leaves_no_trace(mg, precision):
    """The check's flag is cleared by the call that found it set, not at the start of every call."""
    cfg = syn.small_config(6, 5, levels=2, seed=syn.BASE_SEED + 930)
    inp = syn.make_inputs(cfg)
    h = mg.mg_setup_config(cfg, inp, precision=precision)
    good = torch.zeros((6, cfg.nlev, cfg.ncol), dtype=torch.float64, device="cuda")
    b = torch.from_numpy(inp["rhs"]).cuda().ravel()
    ref, x = torch.empty_like(b), torch.empty_like(b)
    mg.vcycle(h, b, ref)
    for s, k, c in ((0, 2, 5), (4, 4, 3), (5, 0, 7)):
        bad = good.clone()
        bad[s, k, c] = 1.0      # a flux from one side only, through the lid, through the surface
        with pytest.raises(mg.MGError) as e:
            mg.mg_set_coefficients(h, bad.ravel())
        assert e.value.status == mg.MG_ERR_ARG
        mg.vcycle(h, b, x)
        assert torch.equal(x, ref)
    mg.mg_set_coefficients(h, good.ravel())
    mg.helmholtz_apply(h, b, x)
    assert torch.equal(x, b)
    h.destroy()


def test_one_fp64_scratch_array_is_enough_for_smoothing(mg):
    """C160L60, restart 1, FP32: 24 + 8 + 56 + 32 bytes per cell and seven FP32 fields padded by 1.215 (9.2M
    cells; a second scratch array would be 74 MB)."""
    used, cells = device_bytes(mg, 160, 60, "fp32")
    assert used <= (24 + 8 + 56 + 32 + 28 * 1.215) * cells + 20 * 2 ** 21, used / cells


@pytest.mark.parametrize("gamma2", [0.0, 0.25])
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("sweeps", [0, 1, 2, 3, 4])
def test_smoothing_in_place(mg, sweeps, precision, gamma2):
    """x_in == x_out, x_in kept, x_in NULL and x_out full of NaN: the same bits as sweep by sweep."""
    cfg = syn.small_config(10, 9, levels=2, seed=syn.BASE_SEED + 940, gamma2=gamma2)
    inp = syn.make_inputs(cfg)
    h = mg.mg_setup_config(cfg, inp, precision=precision)
    for level in range(2):
        n = h.level_cells(level)
        b, x0 = (torch.from_numpy(syn.normal(s, 0, n)).cuda() for s in (3, 4))
        for start in (None, x0):
            ref = torch.zeros_like(b) if start is None else start.clone()
            for i in range(sweeps):
                y = torch.full_like(b, float("nan"))
                mg.mg_smooth(h, level, b, None if i == 0 and start is None else ref, y, 1)
                ref = y
            x = torch.full_like(b, float("nan"))
            mg.mg_smooth(h, level, b, start, x, sweeps)
            assert torch.equal(x, ref)
            if start is not None:
                x = start.clone()
                mg.mg_smooth(h, level, b, x, x, sweeps)
                assert torch.equal(x, ref)
    h.destroy()


def test_first_fp64_calls_on_several_streams_and_threads(mg):
    """Calls on other streams and from other threads than the one that packs an FP32 handle's FP64 data: the
    first one's stream is busy, so that what it enqueued would come last."""
    cfg = syn.small_config(128, 30, levels=2, seed=syn.BASE_SEED + 950)
    inp = syn.make_inputs(cfg)
    h = [mg.mg_setup_config(cfg, inp, precision=p) for p in ("fp64", "fp32", "fp32")]
    b, x0 = torch.from_numpy(inp["rhs"]).cuda().ravel(), torch.from_numpy(syn.normal(9, 0, cfg.ncell)).cuda()
    ref = torch.empty(h[0].level_cells(1), dtype=torch.float64, device="cuda")
    mg.mg_residual_restrict(h[0], 0, b, x0, ref)
    torch.cuda.synchronize()
    busy = torch.empty(4096, 4096, device="cuda")
    for hd, threads in ((h[1], False), (h[2], True)):
        streams = [torch.cuda.Stream() for _ in range(4)]
        out = [torch.empty_like(ref) for _ in streams]
        torch.cuda.synchronize()
        with torch.cuda.stream(streams[0]):
            for _ in range(20):
                busy = busy @ busy
        start, status = threading.Barrier(len(streams)), [None] * len(streams)

        def call(i):
            if threads:
                start.wait()
            status[i] = mg.load().mg_residual_restrict(hd.ptr, 0, b.data_ptr(), x0.data_ptr(), out[i].data_ptr(),
                                                       streams[i].cuda_stream)

        ts = [threading.Thread(target=call, args=(i,)) for i in range(len(streams))]
        for t in ts:
            t.start()
            if not threads:
                t.join()
        for t in ts:
            t.join()
        torch.cuda.synchronize()
        assert status == [mg.MG_OK] * len(streams)
        for o in out:
            assert torch.equal(o, ref)
    for hd in h:
        hd.destroy()
