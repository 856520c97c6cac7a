"""What a handle holds and what its set-up does."""
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
