"""GPU parity of single kernels at the sizes where they can go wrong: edges of tiles, remainders, the smallest and
largest of a dispatch's range.  Oracle, tolerances and comparison as in test_gpu_parity.py."""
import pytest
import torch

from paper_2406_12335_b200 import synth
from tests import parity as P
from tests.test_gpu_parity import _run_case, _small

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,B,F,R,window", [
    (1, 1, 0, 0, 0),            # one token
    (127, 60, 2, 10, 0),
    (128, 64, 0, 8, 0),         # exactly one tile
    (129, 64, 0, 8, 0),         # one row in the second tile
    (256, 100, 2, 10, 0),       # exactly one chunk of streamed tokens
    (1000, 400, 4, 50, 0),      # eight tiles, ragged; the decode step splits a unit over several CTAs
    (600, 250, 2, 10, 200),     # history window that starts inside a tile
])
@pytest.mark.parametrize("call", ["scores", "attention", "lse"])
def test_head_dim_64_on_the_tensor_cores(T, B, F, R, window, call):
    """bf16 with 64 channels through the tensor-core scoring, forward, history-rebuild and decode kernels."""
    _run_case(_small("bf16", 64, T, B, F, R, b=1, h=3, indicator="window" if window else "h2o", window=window, steps=8, cid=80),
              fused_forward=call == "attention", lse_given=call == "lse", recompute_window=bool(window))


def test_head_dim_64_window_leaves_earlier_normalisers_alone():
    """lse_out covers the rows of the history window; what the caller had in the rows before it stays."""
    V = P.vatp()
    wl = _small("bf16", 64, 344, 34, 0, 32, b=1, h=2, indicator="window", window=256, cid=81)
    q, k, v = synth.prefill_inputs(wl, 0, "cuda")
    g = P.GpuPrefill(wl, q, k, v, recompute_window=True)
    g.lse.fill_(7.0)
    V.vatp_prefill_scores(g.p, q, k, v, lse_out=g.lse, attn_acc=g.attn_acc, vnorm=g.vnorm, score=g.score, workspace=g.ws,
                          dev_status=g.status)
    torch.cuda.synchronize()
    assert torch.all(g.lse[..., :344 - 256] == 7.0) and torch.all(g.lse[..., 344 - 256:] != 7.0)
