"""GPU parity of one-chain learning, whose kernels chain by programmatic launch and whose phase A splits
a tile's contraction over a cluster: four and two CTAs a tile and neither, uneven shares of the
k-blocks (d_in and d_out not multiples of four blocks), ragged segments, losses, several segments and
calls in a row, both modes.  Bounds of test_parity_gpu.py."""
import numpy as np
import pytest
import torch

import oracle as O
import paper_2608_17616_gb300 as mone
import workloads as wk
from harness import (DeviceRun, oracle_chain, oracle_hyper, oracle_init, oracle_meta, oracle_read, record,
                     rel_fro)

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2608_17616_gb300 import build
    build.build()
    assert torch.cuda.is_available()
    mone.lib()


@pytest.mark.parametrize("d_in,d_hid,d_out,T,N,mode", [
    (256, 256, 256, 128, 4 * 128 + 5, wk.PAPER),       # 2 tiles, four CTAs each
    (640, 512, 768, 512, 2 * 512 + 130, wk.PAPER),     # 16 tiles; ten and twelve k-blocks over four CTAs
    (128, 1024, 256, 384, 3 * 384, wk.PAPER),          # d_in of two blocks: two CTAs a tile (24 tiles, T / 128 odd)
    (896, 1792, 512, 512, 512 + 1, wk.PLAIN),          # 56 tiles: two CTAs each, seven blocks a share
    (256, 2560, 256, 512, 512 + 77, wk.PAPER),         # 80 tiles: not split
])
def test_one_chain_learning(d_in, d_hid, d_out, T, N, mode):
    wl = wk.Workload("few_tiles", 14, 1, 1, d_in, d_hid, d_out, d_out // 128, 64, T, N, 33, "bf16", mode,
                     0.3 if mode == wk.PAPER else 0.02)
    run = DeviceRun(wl)
    S = wl.S
    loss, step = torch.empty(S, 1, device="cuda"), torch.empty(S, 1, device="cuda")
    mone.mone_ttl_context_metrics(run.h, run.X, run.K, run.V, N, loss, step)
    Xq = wk.query_inputs(wl, "cuda")
    Kg, Vg = run.generate_kv(Xq)
    W1, W2, mu1, mu2 = run.state()
    st, losses, trail = oracle_chain(run, 0, return_all=True)
    for name, w, w0, mu in (("W1", W1, run.W1_0, mu1), ("W2", W2, run.W2_0, mu2)):
        ref, start = st.W[name], O.f64(w0[0])
        assert record("few tiles", name, rel_fro(w[0], ref), 2e-2) <= 2e-2
        assert record("few tiles", "d" + name, rel_fro(w[0].double().numpy() - start, ref - start), 2e-2) <= 2e-2
        if mode == wk.PAPER:
            assert record("few tiles", "mu " + name, rel_fro(mu[0], st.mu[name]), 5e-2) <= 5e-2
    # The loss is a mean of y_t . M(u_t), sums of both signs: besides 2e-2 of its value it carries the
    # rounding of the operands, 2^-8 of |y_t| |M(u_t)| per token (bf16 U, Y and W: 2^-9 each, H and R), independent
    # between tokens.
    hp, meta = oracle_hyper(wl), oracle_meta(run, 0)
    for s in range(S):
        sl = slice(s * T, min(N, (s + 1) * T))
        W = trail[s - 1].W if s else oracle_init(wl, run.W1_0[0], run.W2_0[0]).W
        o, _ = O.memory_forward(O.transform_inputs(run.X[0, 0, sl], hp, meta), W, hp)
        y = np.concatenate([O.f64(run.K[0, 0, sl]), O.f64(run.V[0, 0, sl])], axis=1)
        noise = np.linalg.norm(np.linalg.norm(y, axis=1) * np.linalg.norm(o, axis=1)) / len(y)
        bound = 2e-2 * max(1.0, abs(losses[s])) + 2.0**-8 * noise
        assert record("few tiles", "loss/bound", abs(loss[s, 0].item() - losses[s]) / bound, 1.0) <= 1.0
    Ko, Vo = oracle_read(run, st, 0, Xq)
    assert rel_fro(Kg[0, 0].float(), Ko) <= 2e-2 and rel_fro(Vg[0, 0].float(), Vo) <= 2e-2
    run.close()


def test_one_chain_segments_equal_one_context():
    """Segment by segment, back to back without a wait, the state is the context's up to rounding: a
    segment call ends with the rescaled weights rounded to bf16 anew, where the context goes on with the
    unscaled ones, so their operands differ by two roundings of at most 2^-9 each (momentum bound: twice
    their sum)."""
    wl = wk.Workload("few_tiles", 15, 1, 1, 512, 512, 512, 4, 64, 256, 6 * 256, 8, "bf16", wk.PAPER, 0.3)
    a, b = DeviceRun(wl), DeviceRun(wl)
    a.ttl_context()
    for s in range(wl.S):
        sl = slice(s * 256, (s + 1) * 256)
        mone.mone_ttl_segment(b.h, 0, 0, b.X[0, 0, sl], b.K[0, 0, sl], b.V[0, 0, sl], 256)
    mone.mone_mem_sync(b.h)
    for ta, tb, tol in zip(a.state(), b.state(), (1e-3, 1e-3, 2.0**-7, 2.0**-7)):
        assert rel_fro(ta, tb) <= tol
    a.close()
    b.close()
