"""GPU parity of the fp32 phase kernels over their tile variants: 64 x 64 (phase A) and 128 x 128 (phase B)
tiles on large grids, 32 x 64 and 64 x 64 where a width is an odd multiple of 64, 32 x 64 on small grids; ragged last
segments (rows of a tile absent, a contraction over few tokens) and plain mode; and of the resident kernel
(d_in + d_out <= 512) at widths that end inside a warp's 128 columns, with four and with eight rows a CTA
(more than 152 CTAs of four; 16 or 32 lanes to a token), and a last segment of one token, of one chunk and one token.  fp32 bound 1e-4 on the
weights, their change and the momentum (test_parity_gpu.py)."""
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


@pytest.mark.parametrize("d_in,d_hid,d_out,T,n_layers,N,mode,loss", [
    (512, 512, 512, 256, 8, 2 * 256 + 33, wk.PAPER, "neg_inner"),  # 64 x 64 and 128 x 128 tiles
    (448, 320, 384, 192, 8, 2 * 192 + 1, wk.PAPER, "neg_inner"),   # 32 x 64 and 64 x 64; a last segment of one token
    (576, 64, 128, 64, 1, 3 * 64 + 17, wk.PAPER, "neg_inner"),     # one 32 x 64 tile column
    (384, 256, 256, 128, 2, 2 * 128 + 65, wk.PLAIN, "mse"),        # residual targets, no momentum
    (64, 64, 128, 64, 2, 3 * 64 + 1, wk.PAPER, "neg_inner"),       # resident: W1 in half a warp's columns
    (192, 128, 256, 128, 3, 2 * 128 + 33, wk.PAPER, "neg_inner"),  # resident: W1 ends inside a warp's columns
    (384, 704, 128, 64, 1, 2 * 64 + 32, wk.PLAIN, "neg_inner"),    # resident, eight rows a CTA
    (320, 256, 128, 64, 3, 3 * 64 + 1, wk.PAPER, "neg_inner"),     # resident, eight rows a CTA, W1 ends inside
    (64, 704, 128, 64, 1, 3 * 64 + 1, wk.PAPER, "neg_inner"),      # eight rows, 16 lanes to a token: three pieces a lane
    (192, 256, 128, 192, 3, 2 * 192 + 17, wk.PLAIN, "neg_inner"),  # five, the most
    (128, 256, 128, 128, 3, 2 * 128 + 33, wk.PAPER, "neg_inner"),  # eight rows, 32 lanes (256 columns)
    (64, 256, 384, 64, 3, 3 * 64 + 33, wk.PAPER, "neg_inner"),     # eight rows, 32 lanes again (448 columns)
])
def test_f32_tiles(d_in, d_hid, d_out, T, n_layers, N, mode, loss):
    wl = wk.Workload("f32_tiles", 13, 1, n_layers, d_in, d_hid, d_out, d_out // 128, 64, T, N, 8, "f32", mode,
                     0.3 if mode == wk.PAPER else 1e-2, loss=loss)
    run = DeviceRun(wl)
    run.ttl_context()
    W1, W2, mu1, mu2 = run.state()
    for c in sorted({0, n_layers - 1}):
        st, _ = oracle_chain(run, c)
        for name, w, w0, mu in (("W1", W1, run.W1_0, mu1), ("W2", W2, run.W2_0, mu2)):
            ref, start = st.W[name], O.f64(w0[c])
            assert record("f32 tiles", name, rel_fro(w[c], ref), 1e-4) <= 1e-4, c
            assert record("f32 tiles", "d" + name, rel_fro(w[c].double().numpy() - start, ref - start), 1e-4) <= 1e-4, c
            if mode == wk.PAPER:
                assert record("f32 tiles", "mu " + name, rel_fro(mu[c], st.mu[name]), 1e-4) <= 1e-4, c
    run.close()
