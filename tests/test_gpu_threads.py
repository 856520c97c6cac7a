"""Calls on different handles from different host threads."""
import threading

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


def test_tiled_sweeps_of_different_heights_from_two_threads(mg):
    """The tensor-copy sweep's shared memory depends on the column's height, its limit belongs to the
    kernel: neither thread's launches may fail, and the results are those of one thread."""
    work = []
    for n, nlev in ((48, 69), (48, 41)):   # (chunks of 7, not full: one kernel)
        cfg = syn.small_config(n, nlev, levels=1, seed=syn.BASE_SEED + 830 + nlev)
        inp = syn.make_inputs(cfg)
        h = mg.mg_setup_config(cfg, inp, precision="fp32")
        b = torch.from_numpy(inp["rhs"]).cuda().ravel()
        ref = torch.empty_like(b)
        mg.vcycle(h, b, ref)
        work.append((h, b, ref, torch.empty_like(b)))
    torch.cuda.synchronize()
    lib, failed = mg.load(), [0, 0]
    start = threading.Barrier(2)

    def run(i):
        h, b, _, x = work[i]
        args = (h.ptr, b.data_ptr(), x.data_ptr(), torch.cuda.Stream().cuda_stream)
        start.wait()
        for k in range(4000):   # (the library call itself runs without the interpreter's lock)
            failed[i] += lib.vcycle(*args) != mg.MG_OK
            if k % 100 == 99:
                torch.cuda.synchronize()

    ts = [threading.Thread(target=run, args=(i,)) for i in range(2)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    torch.cuda.synchronize()
    assert failed == [0, 0]
    for h, _, ref, x in work:
        assert torch.equal(x, ref)
        h.destroy()
