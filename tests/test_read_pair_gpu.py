"""GPU parity of the memory read on CTA pairs (more tiles of 128 queries x 128 hidden units than SMs): query
counts that end inside the first and the second CTA's half of a tile of 256, one past a tile, and heads of 64
and of 128.  bf16 bound 2e-2 (test_parity_gpu.py)."""
import pytest
import torch

import paper_2608_17616_gb300 as mone
import workloads as wk
from harness import DeviceRun, oracle_chain, oracle_read, record, rel_fro

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2608_17616_gb300 import build
    build.build()
    assert torch.cuda.is_available()
    mone.lib()


@pytest.mark.parametrize("Q,hd,mode", [(1000, 64, wk.PAPER), (1025, 128, wk.PAPER), (513, 64, wk.PLAIN), (900, 128, wk.PLAIN)])
def test_read_of_many_tiles(Q, hd, mode):
    # 10 chains x 4 tiles of hidden units (and of outputs) x ceil(Q / 128) query tiles; more than 4608 query
    # rows, so the input transform takes two a warp (an odd Q leaves a warp with one)
    wl = wk.Workload("read_pair", 14, 2, 5, 256, 512, 512, 512 // (2 * hd), hd, 128, 160, Q, "bf16", mode)
    run = DeviceRun(wl)
    run.ttl_context()
    Xq = wk.query_inputs(wl, "cuda")
    Kg, Vg = run.generate_kv(Xq)
    for c in (0, wl.chains - 1):
        st, _ = oracle_chain(run, c)
        ctx, layer = divmod(c, wl.n_layers)
        Ko, Vo = oracle_read(run, st, c, Xq)
        assert record("read pair", "K", rel_fro(Kg[ctx, layer].float(), Ko), 2e-2) <= 2e-2, c
        assert record("read pair", "V", rel_fro(Vg[ctx, layer].float(), Vo), 2e-2) <= 2e-2, c
    run.close()
