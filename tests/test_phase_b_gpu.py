"""GPU parity of phase B where its column tiles and state ring can go wrong: widths that leave a
128-column tile in W1, tiles of W2 that take half their columns from K and half from V, launches of
more than one tile per CTA (wide and narrow tiles through the same ring), the four ways the ring's slots
are handed back (by tiles a CTA and T; plain mode and CTA pairs as few tiles) and the CTA-pair form.  Bounds as in
test_parity_gpu.py: 2e-2 on the weights and on their change."""
import pytest
import torch

import oracle as O
import paper_2608_17616_gb300 as mone
import workloads as wk
from harness import DeviceRun, oracle_chain, record, rel_fro

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2608_17616_gb300 import build
    build.build()
    assert torch.cuda.is_available()
    mone.lib()


@pytest.mark.parametrize("d_in,d_hid,d_out,T,n_layers,N,mode", [
    (128, 256, 256, 128, 2, 300, wk.PAPER),      # a narrow tile of W1, one of W2 from K and V
    (384, 256, 768, 128, 30, 300, wk.PAPER),     # 256 + 128 columns in W1; 150 tiles a launch, two launches
    (384, 256, 768, 512, 30, 700, wk.PAPER),     # the same in longer segments
    (384, 768, 768, 256, 20, 600, wk.PAPER),     # two tiles a CTA: slots by twos, one store later
    (1152, 2048, 1280, 256, 22, 513, wk.PAPER),  # 11.6 tiles a CTA: slots one by one, three stores later
    (512, 512, 512, 128, 80, 300, wk.PAPER),     # 4.2 tiles a CTA: the same
    (512, 512, 512, 512, 168, 513, wk.PAPER),    # 8.8 tiles a CTA at T = 512: slots by twos, three stores later
    (384, 256, 256, 4096, 204, 4096 + 5, wk.PAPER),  # 4.03 tiles a CTA at T = 4096: slots by fours, two stores later
    (640, 256, 256, 256, 3, 513, wk.PLAIN),      # W alone in the ring; a last segment of one token
    (512, 256, 512, 1024, 3, 1024 + 65, wk.PAPER),  # CTA pairs
    (512, 256, 768, 1024, 3, 1024 + 65, wk.PAPER),  # CTA pairs, a tile from K and V
    (640, 256, 768, 1024, 3, 1024 + 65, wk.PAPER),  # T = 1024 with a narrow tile: one-CTA tiles
])
def test_phase_b_tiles(d_in, d_hid, d_out, T, n_layers, N, mode):
    wl = wk.Workload("phase_b", 12, 1, n_layers, d_in, d_hid, d_out, d_out // 128, 64, T, N, 8, "bf16", mode,
                     0.3 if mode == wk.PAPER else 0.05)
    run = DeviceRun(wl)
    run.ttl_context()
    W1, W2, mu1, mu2 = run.state()
    for c in sorted({0, n_layers // 2, n_layers - 1}):
        st, _ = oracle_chain(run, c)
        for name, w, w0, mu in (("W1", W1, run.W1_0, mu1), ("W2", W2, run.W2_0, mu2)):
            ref, start = st.W[name], O.f64(w0[c])
            assert record("phase B", name, rel_fro(w[c], ref), 2e-2) <= 2e-2, c
            assert record("phase B", "d" + name, rel_fro(w[c].double().numpy() - start, ref - start), 2e-2) <= 2e-2, c
            if mode == wk.PAPER:
                assert record("phase B", "mu " + name, rel_fro(mu[c], st.mu[name]), 5e-2) <= 5e-2, c
    run.close()
