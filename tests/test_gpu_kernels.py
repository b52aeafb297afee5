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


@pytest.mark.parametrize("b,h,kv,d,B,window", [
    (1, 3, 0, 128, 1, 0),        # one slot besides the incoming token's
    (1, 3, 0, 128, 127, 0),      # ring of fewer units than slots
    (2, 60, 0, 128, 200, 0),     # 120 units: one CTA each, requests by the warps themselves
    (2, 60, 0, 64, 300, 0),      # rings deeper than some warps' rows
    (3, 100, 0, 128, 130, 0),    # 300 units: more than two CTAs per SM hold, the producer warp goes on to a second unit
    (3, 100, 0, 64, 130, 40),    # the same with head_dim 64 and a history window (the state of the next unit is fetched early)
    (5, 8, 2, 128, 600, 0),      # grouped queries split over a cluster
    (2, 640, 160, 64, 90, 0),    # grouped queries, several units per CTA
    (1, 80, 0, 128, 1100, 0),    # a unit over two CTAs, beyond one CTA per SM
    (1, 60, 0, 64, 1900, 0),     # ... over four
    (1, 3, 0, 128, 1030, 0),     # eight CTAs a unit, seven slots beyond their tiles
    (1, 4, 0, 64, 1031, 40),     # ... eight, a history window
    (1, 8, 2, 128, 1025, 0),     # ... two, four heads
    (1, 2, 0, 128, 9000, 0),     # state beyond shared memory
    (1, 300, 0, 128, 2048, 30),  # several units per CTA, their state read from global memory in the tail
])
@pytest.mark.parametrize("grow", [0, 5, 190])       # (less where the budget is smaller)
def test_decode_step_against_float64(b, h, kv, d, B, window, grow):
    """One-step arithmetic of every unit against float64 torch: output rows, indicators, evicted token; grow: the cache
    starts that many tokens short of its budget, so rows requested before the live range is known are dropped."""
    V = P.vatp()
    hk, T = kv or h, 2 * B
    G = h // hk
    grow = min(grow, B - 1)
    p = V.make_params(batch=b, heads=h, kv_heads=kv, seq_len=T, head_dim=d, dtype="bf16", budget=B,
                      indicator="window" if window else "h2o", window=window)
    c, n = V.Cache(p), B - grow
    g = torch.Generator(device="cuda").manual_seed(B + h)
    rnd = lambda *s: torch.randn(*s, generator=g, device="cuda")  # noqa: E731
    c.k_cache[:, :, :n], c.v_cache[:, :, :n] = rnd(b, hk, n, d).bfloat16(), rnd(b, hk, n, d).bfloat16()
    c.pos[:, :, :n] = torch.arange(n, dtype=torch.int32, device="cuda")
    c.vnorm[:, :, :n] = c.v_cache[:, :, :n].float().abs().sum(-1)
    c.len.fill_(n), c.free_slot.fill_(n), c.next_pos.fill_(T)
    if window:
        c.ring[..., :n] = torch.rand(b, hk, window, n, generator=g, device="cuda") / n
        c.acc_fixed[..., :n] = (c.ring[..., :n].double() * 2.0 ** 52).long().sum(2)
        c.acc.copy_((c.acc_fixed.double() / 2.0 ** 52).float())
    else:
        c.acc[:, :, :n] = torch.rand(b, hk, n, generator=g, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    i0, i1 = torch.arange(b, device="cuda")[:, None], torch.arange(hk, device="cuda")[None]
    for s in range(3):
        q, k, v = rnd(b, h, d).bfloat16(), rnd(b, hk, d).bfloat16(), rnd(b, hk, d).bfloat16()
        fs = c.free_slot.long()
        K, W, acc, vn, pos = c.k_cache.double(), c.v_cache.double(), c.acc.double(), c.vnorm.double(), c.pos.clone()
        K[i0, i1, fs], W[i0, i1, fs], vn[i0, i1, fs], pos[i0, i1, fs] = k.double(), v.double(), v.double().abs().sum(-1), T + s
        live = pos >= 0
        logits = torch.einsum("bhd,bhnd->bhn", q.double(), K.repeat_interleave(G, 1)) * d ** -0.5
        prob = torch.softmax(logits.masked_fill(~live.repeat_interleave(G, 1), float("-inf")), -1)
        want = torch.einsum("bhn,bhnd->bhd", prob, W.repeat_interleave(G, 1))
        acc[i0, i1, fs] = 0
        if window:
            old = c.ring[:, :, (T + s) % window].double()
            old[i0, i1, fs] = 0
            acc -= old
        acc += prob.view(b, hk, G, -1).mean(2)
        out, ev = torch.empty_like(q), torch.empty(b, hk, dtype=torch.int32, device="cuda")
        V.vatp_decode_step(p, c, q, k, v, out, evicted_pos=ev, dev_status=status)
        torch.cuda.synchronize()
        assert int(status.item()) == 0
        # bf16 output: half a unit in the last place of the largest value, and the sums' 1e-3
        assert torch.all((out.double() - want).abs() <= 2.0 ** -8 * want.abs() + 1e-3 * want.abs().amax(-1, keepdim=True))
        assert torch.all(((c.acc.double() - acc).abs() <= 1e-3 * acc.abs() + 1e-6)[live])
        assert torch.all(((c.vnorm.double() - vn).abs() <= 1e-5 * vn)[live])
        if n + s < B:
            assert torch.all(ev == -1)
        else:
            imp = (acc * vn).masked_fill(~live, float("inf"))
            got = imp.gather(2, (pos == ev[..., None]).int().argmax(-1, keepdim=True))[..., 0]
            assert torch.all((pos == ev[..., None]).sum(-1) == 1)
            assert torch.all(got <= imp.amin(-1) * (1 + 2e-3) + 1e-9)      # the minimum, up to both sides' tolerance


@pytest.mark.parametrize("units,B,layers", [
    (8, 300, 8),     # eight launches of one CTA per SM fill the machine, of two they do not
    (48, 500, 4),
    (8, 300, 2),     # too few either way
    (90, 1000, 3),   # a unit over two CTAs
])
def test_steps_of_several_caches_side_by_side(units, B, layers):
    """Steps of several caches in turn, with and without leave to overlap: the same bits."""
    V = P.vatp()
    got = []
    for overlap in (False, True):
        g = torch.Generator(device="cuda").manual_seed(B)
        rnd = lambda *s: torch.randn(*s, generator=g, device="cuda").bfloat16()  # noqa: E731
        p = V.make_params(batch=1, heads=units, seq_len=2 * B, head_dim=128, dtype="bf16", budget=B, decode_overlap=overlap)
        caches = [V.Cache(p) for _ in range(layers)]
        for c in caches:
            c.k_cache[:, :, :B], c.v_cache[:, :, :B] = rnd(1, units, B, 128), rnd(1, units, B, 128)
            c.pos[:, :, :B] = torch.arange(B, dtype=torch.int32, device="cuda")
            c.vnorm[:, :, :B] = c.v_cache[:, :, :B].float().abs().sum(-1)
            c.acc[:, :, :B] = torch.rand(1, units, B, generator=g, device="cuda")
            c.len.fill_(B), c.free_slot.fill_(B), c.next_pos.fill_(2 * B)
        qkv = [[rnd(3, 1, units, 128) for _ in range(layers)] for _ in range(6)]
        out = torch.empty(6, layers, 1, units, 128, dtype=torch.bfloat16, device="cuda")
        status = torch.zeros(1, dtype=torch.int32, device="cuda")
        torch.cuda.synchronize()
        for s in range(6):
            for l, c in enumerate(caches):
                V.vatp_decode_step(p, c, *qkv[s][l], out[s, l], dev_status=status)
        torch.cuda.synchronize()
        assert int(status.item()) == 0
        got.append([out] + [t for c in caches for t in (c.k_cache, c.v_cache, c.acc, c.vnorm, c.pos, c.len, c.free_slot)])
    assert all(torch.equal(a, b) for a, b in zip(*got))


@pytest.mark.parametrize("units,B,d,window", [
    (37, 600, 128, 0),       # one CTA per SM resident: a cluster of two
    (64, 600, 64, 300),      # two CTAs per SM, all threads clear a recycled slot's history first
    (30, 1500, 64, 400),     # clusters of eight, a long history: one thread clears it
    (30, 19000, 128, 0),     # split further for the slots' state to fit
    (2, 1, 64, 3),           # one slot besides the incoming token's
])
def test_fp32_decode_step_against_float64(units, B, d, window):
    """The general kernel's steps back to back, each read only at the end, against float64 torch."""
    V = P.vatp()
    p = V.make_params(batch=1, heads=units, seq_len=2 * B, head_dim=d, dtype="f32", budget=B,
                      indicator="window" if window else "h2o", window=window)
    c = V.Cache(p)
    g = torch.Generator(device="cuda").manual_seed(units + B)
    rnd = lambda *s: torch.randn(*s, generator=g, device="cuda")  # noqa: E731
    c.k_cache[:, :, :B], c.v_cache[:, :, :B] = rnd(1, units, B, d), rnd(1, units, B, d)
    c.pos[:, :, :B] = torch.arange(B, dtype=torch.int32, device="cuda")
    c.vnorm[:, :, :B] = c.v_cache[:, :, :B].abs().sum(-1)
    c.len.fill_(B), c.free_slot.fill_(B), c.next_pos.fill_(2 * B)
    if window:
        c.ring[..., :B] = torch.rand(1, units, window, B, generator=g, device="cuda") / B
        c.acc_fixed[..., :B] = (c.ring[..., :B].double() * 2.0 ** 52).long().sum(2)
        c.acc.copy_((c.acc_fixed.double() / 2.0 ** 52).float())
    else:
        c.acc[:, :, :B] = torch.rand(1, units, B, generator=g, device="cuda")
    K, W, pos, n = c.k_cache[0].double(), c.v_cache[0].double(), c.pos[0].clone(), B + 1
    fs = c.free_slot[0].long()
    q, k, v = (rnd(4, 1, units, d) for _ in range(3))
    out, ev = torch.empty_like(q), torch.empty(4, 1, units, dtype=torch.int32, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    for s in range(4):
        V.vatp_decode_step(p, c, q[s], k[s], v[s], out[s], evicted_pos=ev[s], dev_status=status)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    i = torch.arange(units, device="cuda")
    for s in range(4):
        K[i, fs], W[i, fs], pos[i, fs] = k[s, 0].double(), v[s, 0].double(), 2 * B + s
        logits = torch.einsum("hd,hnd->hn", q[s, 0].double(), K) * d ** -0.5
        want = torch.einsum("hn,hnd->hd", torch.softmax(logits.masked_fill(pos < 0, float("-inf")), -1), W)
        # fp32 sums of n terms and exponentials: n * 2^-24 of the largest value, and 2^-20 of slack for exp2f's argument
        assert torch.all((out[s, 0].double() - want).abs() <= (n * 2.0 ** -24 + 2.0 ** -18) * W.abs().amax(1))
        fs = (pos == ev[s, 0][:, None]).int().argmax(1)
        pos[i, fs] = -1
    assert torch.equal(pos[:, :n], c.pos[0, :, :n])
    if window:
        # the windowed sums are the ring's columns added up exactly
        live = c.pos[0] >= 0
        sums = (c.ring[0].double() * 2.0 ** 52).long().sum(1)
        assert torch.equal(sums[live], c.acc_fixed[0][live])


@pytest.mark.parametrize("units", [5, 200])          # CTAs of 1024 and of 512 threads
@pytest.mark.parametrize("n", [1, 2, 3, 5, 30, 31, 1022, 1023, 1024, 1025, 2047, 2051, 7806, 7807])
def test_select_middle_range_of_every_length_and_alignment(units, n):
    """Middle ranges of every residue mod 4 whose first score lies at every alignment (odd prompt lengths, several units),
    some with ties at the boundary: the kept sets bit for bit."""
    from oracle import vatp_oracle as O
    V = P.vatp()
    for F in range(4):
        R, keep = 2 + (n + F) % 2, max(n // 3, 1) - (n == 1)
        T, B = n + F + R, keep + F + R
        if T <= B or B == 0:
            continue
        T += 1 - T % 2 if n > 8 else 0               # odd: the units' rows start at all four alignments
        g = torch.Generator().manual_seed(n + F)
        score = torch.rand(1, units, T, generator=g)
        score[:, ::2] = (score[:, ::2] * 16).floor()
        p = V.make_params(batch=1, heads=units, seq_len=T, head_dim=64, dtype="f32", budget=B, n_sink=F, n_recent=R)
        kept = torch.empty(1, units, B, dtype=torch.int32, device="cuda")
        status = torch.zeros(1, dtype=torch.int32, device="cuda")
        V.vatp_select(p, score.cuda(), kept, dev_status=status)
        torch.cuda.synchronize()
        assert int(status.item()) == 0
        for u in list(range(5)) + [units - 1]:
            assert kept[0, u].cpu().numpy().tolist() == O.select_keep(score[0, u].numpy(), B, F, R).tolist()


def test_select_alignments_on_the_bounds_checking_build():
    """The same on the build that range-checks every staged group before it is read."""
    import os
    import subprocess
    import sys
    from paper_2406_12335_b200 import build
    env = dict(os.environ, VATP_LIBRARY=build.build(debug_bounds=True))
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-m", "pytest", "tests/test_gpu_kernels.py", "-x", "-q", "-m", "gpu", "-k", "every_length_and_alignment",
                        "-p", "no:cacheprovider"], cwd=root, env=env, capture_output=True, text=True)
    assert r.returncode == 0 and " passed" in r.stdout, (r.stdout + r.stderr)[-2000:]


@pytest.mark.parametrize("units,B", [(320, 300), (16, 600)])     # several units per CTA, and one
def test_overlapping_steps_whose_output_lands_in_an_earlier_steps_query(units, B):
    """Steps of several caches over three query / output buffers in turn: a step's output replaces the query of the step
    before it, which its launch may still be reading.  With and without leave to overlap: the same bits."""
    V = P.vatp()
    got = []
    for overlap in (False, True):
        g = torch.Generator(device="cuda").manual_seed(B)
        rnd = lambda *s: torch.randn(*s, generator=g, device="cuda").bfloat16()  # noqa: E731
        p = V.make_params(batch=1, heads=units, seq_len=2 * B, head_dim=128, dtype="bf16", budget=B, decode_overlap=overlap)
        caches = [V.Cache(p) for _ in range(4)]
        for c in caches:
            c.k_cache[:, :, :B], c.v_cache[:, :, :B] = rnd(1, units, B, 128), rnd(1, units, B, 128)
            c.pos[:, :, :B] = torch.arange(B, dtype=torch.int32, device="cuda")
            c.vnorm[:, :, :B] = c.v_cache[:, :, :B].float().abs().sum(-1)
            c.acc[:, :, :B] = torch.rand(1, units, B, generator=g, device="cuda")
            c.len.fill_(B), c.free_slot.fill_(B), c.next_pos.fill_(2 * B)
        buf, kv = [rnd(1, units, 128) for _ in range(3)], [(rnd(1, units, 128), rnd(1, units, 128)) for _ in range(24)]
        status = torch.zeros(1, dtype=torch.int32, device="cuda")
        torch.cuda.synchronize()
        for s in range(24):
            V.vatp_decode_step(p, caches[s % 4], buf[s % 3], *kv[s], buf[(s + 2) % 3], dev_status=status)
        torch.cuda.synchronize()
        assert int(status.item()) == 0
        got.append(buf + [t for c in caches for t in (c.k_cache, c.v_cache, c.acc, c.vnorm, c.pos, c.free_slot)])
    assert all(torch.equal(a, b) for a, b in zip(*got))


def _probabilities(q, k, first, scale):
    """float64 rows first .. T - 1 of the causal attention matrix of one unit ([T, d] each), and their normalisers."""
    s = (q[first:].double() @ k.double().T) * scale
    T = k.shape[0]
    s.masked_fill_(torch.arange(T, device=q.device)[None] > torch.arange(first, T, device=q.device)[:, None], float("-inf"))
    lse = torch.logsumexp(s, -1)
    return torch.exp(s - lse[:, None]), lse


@pytest.mark.parametrize("d,heads,kv", [(64, 1, 0), (128, 2, 1)])
def test_history_of_more_elements_than_32_bits_index(d, heads, kv):
    """A history window times a capacity beyond 2^31 elements (8.6 GB of rows per cache), head_dim 64 and grouped queries."""
    V = P.vatp()
    T, w, B = 300, 65536, 32768
    p = V.make_params(batch=1, heads=heads, kv_heads=kv, seq_len=T, head_dim=d, dtype="bf16", budget=B, indicator="window", window=w)
    g = torch.Generator(device="cuda").manual_seed(d)
    q, k, v = (torch.randn(1, n, T, d, generator=g, device="cuda").bfloat16() for n in (heads, kv or heads, kv or heads))
    rows = [_probabilities(q[0, h], k[0, 0], 0, d ** -0.5) for h in range(heads)]
    want, lse = sum(r[0] for r in rows) / heads, torch.stack([r[1] for r in rows])[None].float().contiguous()
    acc, vnorm = torch.zeros(1, 1, T, device="cuda"), v.float().abs().sum(-1)
    kept = torch.full((1, 1, B), -1, dtype=torch.int32, device="cuda")
    kept[..., :T] = torch.arange(T, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    c = V.Cache(p)
    assert w * c.cap >= 1 << 31
    V.vatp_compact_window(p, q, k, v, lse, acc, vnorm, kept, c, dev_status=status)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    # 32-bit logits and normalisers of size up to 8: each rounding shows as 2^-21 of the probability at most, four of them
    assert torch.all((c.ring[0, 0, :T, :T].double() - want).abs() <= 2.0 ** -19 * want)
    assert torch.all(((c.acc[0, 0, :T].double() - want.sum(0)).abs() <= 2.0 ** -19 * want.sum(0)))
    assert int(torch.count_nonzero(c.ring[0, 0, T:])) == 0 and int(torch.count_nonzero(c.ring[0, 0, :T, T:])) == 0


@pytest.mark.parametrize("call", ["scores", "lse"])
def test_value_norms_of_a_very_long_prompt(call):
    """One token more than 65535 groups of 64: the value norms beside a history window's scoring."""
    V = P.vatp()
    T, w, d = 65535 * 64 + 1, 16, 64
    p = V.make_params(batch=1, heads=1, seq_len=T, head_dim=d, dtype="bf16", budget=64, indicator="window", window=w)
    g = torch.Generator(device="cuda").manual_seed(7)
    q, k, v = (torch.randn(1, 1, T, d, generator=g, device="cuda").bfloat16() for _ in range(3))
    prob, lse = _probabilities(q[0, 0], k[0, 0], T - w, d ** -0.5)
    acc, vnorm, score, given = (torch.zeros(1, 1, T, device="cuda") for _ in range(4))
    given[0, 0, T - w:] = lse.float()
    ws = torch.empty(V.vatp_workspace_bytes(p), dtype=torch.uint8, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    to = dict(attn_acc=acc, vnorm=vnorm, score=score, workspace=ws, dev_status=status)
    if call == "lse":
        V.vatp_prefill_scores_from_lse(p, q, k, v, given, **to)
    else:
        V.vatp_prefill_scores(p, q, k, v, **to)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    norm = v[0, 0].float().abs().sum(-1)
    assert torch.allclose(vnorm[0, 0], norm, rtol=1e-5, atol=0)
    # logits and normalisers (size up to 22 in the log2 domain) rounded to 32 bits, exponentials good to 2^-20
    assert torch.all((acc[0, 0].double() - prob.sum(0)).abs() <= 2.0 ** -17 * prob.sum(0))
    assert torch.equal(score, acc * vnorm)


@pytest.mark.parametrize("w,heads,kv", [(700, 2, 0), (300, 8, 2), (700, 12, 1)])
def test_history_of_several_chunks_and_heads(w, heads, kv):
    """Each chunk of 256 window rows and each head of a group meets its own normalisers: they differ widely from head to head
    and from row to row (scaled queries)."""
    V = P.vatp()
    T, d, B, hk = 800, 128, 200, kv or heads
    p = V.make_params(batch=1, heads=heads, kv_heads=kv, seq_len=T, head_dim=d, dtype="bf16", budget=B, indicator="window", window=w)
    g = torch.Generator(device="cuda").manual_seed(w)
    rnd = lambda n: torch.randn(1, n, T, d, generator=g, device="cuda")  # noqa: E731
    size = (torch.arange(heads, device="cuda")[:, None] % 3 + 1) * (1 + torch.arange(T, device="cuda")[None] // 100 % 2)
    q, k, v = (rnd(heads) * size[None, ..., None]).bfloat16(), rnd(hk).bfloat16(), rnd(hk).bfloat16()
    G, f32 = heads // hk, dict(dtype=torch.float32, device="cuda")
    rows = [_probabilities(q[0, h], k[0, h // G], 0, d ** -0.5) for h in range(heads)]
    lse = torch.stack([r[1] for r in rows])[None].float().contiguous()
    want = torch.stack([r[0] for r in rows]).view(hk, G, T, T).mean(1)[:, T - w:]
    kept = torch.randperm(T, generator=torch.Generator().manual_seed(w))[:B].sort().values.cuda()
    c, status = V.Cache(p), torch.zeros(1, dtype=torch.int32, device="cuda")
    V.vatp_compact_window(p, q, k, v, lse, torch.zeros(1, hk, T, **f32), torch.ones(1, hk, T, **f32), kept.int().repeat(1, hk, 1).contiguous(),
                          c, dev_status=status)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    ring = c.ring[0][:, torch.arange(T - w, T, device="cuda") % w, :B].double()
    want = want[..., kept]
    # 32-bit logits and normalisers of size up to 64 in the log2 domain: a few roundings of 2^-19 each
    assert torch.all((ring - want).abs() <= 2.0 ** -16 * want + 1e-30)


@pytest.mark.parametrize("d,heads,kv,T,w", [(64, 16, 0, 1531, 256), (64, 8, 2, 700, 100), (128, 8, 2, 700, 100), (128, 32, 8, 900, 300)])
def test_history_precision_of_head_dim_64_and_grouped_queries(d, heads, kv, T, w):
    """The rebuilt history against float64 given the normalisers: no coarser than 32-bit arithmetic in natural logarithms."""
    V = P.vatp()
    B, hk = T // 2, kv or heads
    G = heads // hk
    p = V.make_params(batch=1, heads=heads, kv_heads=kv, seq_len=T, head_dim=d, dtype="bf16", budget=B, indicator="window", window=w)
    g = torch.Generator(device="cuda").manual_seed(T + d)
    q, k, v = (torch.randn(1, n, T, d, generator=g, device="cuda").bfloat16() for n in (heads, hk, hk))
    lse = torch.stack([_probabilities(q[0, h], k[0, h // G], 0, d ** -0.5)[1] for h in range(heads)])[None].float().contiguous()
    s = (q.double() @ k.double().repeat_interleave(G, 1).transpose(-1, -2)) * d ** -0.5
    s.masked_fill_(torch.ones(T, T, dtype=torch.bool, device="cuda").triu(1), float("-inf"))
    want = torch.exp(s - lse[..., None].double())[0].view(hk, G, T, T).mean(1)[:, T - w:]
    kept = torch.randperm(T, generator=torch.Generator().manual_seed(w))[:B].sort().values.cuda()
    c, status = V.Cache(p), torch.zeros(1, dtype=torch.int32, device="cuda")
    ones = torch.ones(1, hk, T, device="cuda")
    V.vatp_compact_window(p, q, k, v, lse, ones, ones, kept.int().repeat(1, hk, 1).contiguous(), c, dev_status=status)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    ring, want = c.ring[0][:, torch.arange(T - w, T, device="cuda") % w, :B].double(), want[..., kept]
    sums = want.sum(1)
    # their sums: rounded once to 32 bits (up to 3.4e-8), what is left of the means below 1.5e-8
    assert float((c.acc[0, :, :B].double() - sums).norm() / sums.norm()) <= 3.8e-8
    # exponents of magnitude 8 to 16 rounded once: 2^-20 / sqrt(12) * ln 2 = 1.9e-7 of a probability, 5e-8 for its exponential and
    # the factor; a second rounding of that size (of the normaliser) would give 2.7e-7
    e = float((ring - want).norm() / want.norm())
    print(f"[history precision] d {d} heads {heads}/{hk}: {e:.3e}")
    assert e <= 2.1e-7


@pytest.mark.parametrize("kv", [0, 3])      # (groups of four: the factor of their mean is exact, a third would be 3e-8 off)
@pytest.mark.parametrize("T,window", [(130, 0), (300, 100), (700, 0), (1531, 0), (1531, 256), (3000, 100), (3000, 256)])
def test_head_dim_64_scoring_precision(T, window, kv):
    """Normalisers and indicators against float64, and the mean error of the indicators: as good as 32-bit arithmetic in
    natural logarithms gives them."""
    V = P.vatp()
    h, d, hk = 12, 64, kv or 12
    p = V.make_params(batch=1, heads=h, kv_heads=kv, seq_len=T, head_dim=d, dtype="bf16", budget=T // 2, indicator="window" if window else "h2o",
                      window=window)
    e_lse, e, mean = [], [], []
    for seed in range(3):
        g = torch.Generator(device="cuda").manual_seed(T + seed)
        q, k, v = (torch.randn(1, n, T, d, generator=g, device="cuda").bfloat16() for n in (h, hk, hk))
        acc, vnorm, score = (torch.zeros(1, hk, T, device="cuda") for _ in range(3))
        lse = torch.zeros(1, h, T, device="cuda")
        status, ws = torch.zeros(1, dtype=torch.int32, device="cuda"), torch.empty(V.vatp_workspace_bytes(p), dtype=torch.uint8, device="cuda")
        V.vatp_prefill_scores(p, q, k, v, lse_out=lse, attn_acc=acc, vnorm=vnorm, score=score, workspace=ws, dev_status=status)
        torch.cuda.synchronize()
        assert int(status.item()) == 0
        first = max(T - window, 0) if window else 0
        rows = [_probabilities(q[0, i], k[0, i * hk // h], first, d ** -0.5) for i in range(h)]
        want_lse, want = torch.stack([r[1] for r in rows]), torch.stack([r[0].sum(0) for r in rows]).view(hk, h // hk, T).mean(1)
        e_lse.append(float((lse[0, :, first:].double() - want_lse).norm() / want_lse.norm()))
        e.append(float((acc[0].double() - want).norm() / want.norm()))
        mean.append(float(((acc[0].double() - want) / want).mean()))
    print(f"[scoring precision] T {T} window {window} heads {h}/{hk}: normalisers {sum(e_lse) / 3:.3e} indicators {sum(e) / 3:.3e} mean {sum(mean) / 3:.3e}")
    # values of 3 to 8, the result's and the logarithm's rounding: up to 1.4e-7 of about 4.5 at the least, up to 2.7e-7 of 8 and more
    assert sum(e_lse) / 3 <= 4.2e-8
    # the terms' exponents, of magnitude 4 to 16, are rounded once each (2e-7 of a term, less the more rows are summed) and the sums
    # in sixteen chains: 5e-8 to 8e-8, of which no more than 4e-8 may be common to all tokens
    assert sum(e) / 3 <= 9e-8 and abs(sum(mean) / 3) <= 4e-8


@pytest.mark.parametrize("what", ["select", "select_clusters", "fp32_step", "grouped_step"])
def test_host_threads_with_calls_of_different_sizes(what):
    """Two threads launch the same kernel with different amounts of shared memory, each on a stream of its own."""
    import threading
    V = P.vatp()
    failed, go = [], threading.Barrier(2)

    def calls(size, stream):
        with torch.cuda.stream(stream):
            status = torch.zeros(1, dtype=torch.int32, device="cuda")
            if what.startswith("select"):
                T, B = size
                p = V.make_params(batch=1, heads=2, seq_len=T, head_dim=64, dtype="f32", budget=B)
                score, kept = torch.rand(1, 2, T, device="cuda"), torch.empty(1, 2, B, dtype=torch.int32, device="cuda")
                run = lambda: V.vatp_select(p, score, kept, dev_status=status)  # noqa: E731
            else:
                kv = 2 if what == "grouped_step" else 0
                p = V.make_params(batch=1, heads=32, kv_heads=kv, seq_len=2 * size, head_dim=64, dtype="f32", budget=size)
                c, q = V.Cache(p), torch.zeros(1, 32, 64, device="cuda")
                c.len.zero_(), c.free_slot.zero_()
                k, out = torch.zeros(1, kv or 32, 64, device="cuda"), torch.empty(1, 32, 64, device="cuda")
                run = lambda: V.vatp_decode_step(p, c, q, k, k, out, dev_status=status)  # noqa: E731
            stream.synchronize()
            go.wait()
            try:
                for _ in range(3000):
                    run()
            except V.VatpError as e:
                failed.append(str(e))
            stream.synchronize()
            assert int(status.item()) == 0

    sizes = {"select": ((1500, 100), (8000, 1000)), "select_clusters": ((9000, 1000), (100000, 20000)), "fp32_step": (100, 9000),
             "grouped_step": (64, 1500)}[what]
    threads = [threading.Thread(target=calls, args=(s, torch.cuda.Stream())) for s in sizes]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed, failed


@pytest.mark.parametrize("T", [189000, 192000])      # a cluster's shared memory holds the first in four parts, not the second
def test_select_from_a_very_long_prompt(T):
    from oracle import vatp_oracle as O
    V = P.vatp()
    score = torch.rand(1, 2, T, generator=torch.Generator().manual_seed(T))
    p = V.make_params(batch=1, heads=2, seq_len=T, head_dim=64, dtype="f32", budget=T // 5, n_sink=3, n_recent=100)
    kept, status = torch.empty(1, 2, T // 5, dtype=torch.int32, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
    V.vatp_select(p, score.cuda(), kept, dev_status=status)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    for u in range(2):
        assert kept[0, u].cpu().numpy().tolist() == O.select_keep(score[0, u].numpy(), T // 5, 3, 100).tolist()


@pytest.mark.parametrize("d,units,T,window,call,norm,tile", [
    (64, 49, 700, 0, "scores", "l1", 64),       # 294 rows of 128-row tiles: just below twice 148 SMs
    (64, 50, 700, 0, "scores", "l1", 128),      # 300: the large tiles, the last of a unit ragged
    (128, 49, 769, 0, "scores", "l2", 128),     # one row in the last tile
    (128, 50, 700, 0, "lse", "linf", 128),
    (64, 150, 500, 200, "scores", "l1", 128),   # history window, which starts inside a tile of keys
    (128, 99, 530, 257, "lse", "l1", 128),
    (128, 150, 300, 400, "scores", "l1", 128),  # window longer than the prompt
])
def test_fp32_scoring_tiles_against_float64(d, units, T, window, call, norm, tile):
    """The fp32 passes either side of the line between 64- and 128-row tiles."""
    V = P.vatp()
    rows = window if 0 < window < T else T
    assert (tile == 128) == (units * ((rows + 127) // 128) >= 2 * 148)
    p = V.make_params(batch=1, heads=units, seq_len=T, head_dim=d, dtype="f32", budget=T // 2, indicator="window" if window else "h2o",
                      window=window, norm=norm)
    g = torch.Generator(device="cuda").manual_seed(T + d)
    q, k, v = (torch.randn(1, units, T, d, generator=g, device="cuda") for _ in range(3))
    first = max(T - window, 0) if window else 0
    ref = [_probabilities(q[0, i], k[0, i], first, d ** -0.5) for i in range(units)]
    want, want_lse = torch.stack([r[0].sum(0) for r in ref]), torch.stack([r[1] for r in ref])
    acc, vnorm, score, lse = (torch.zeros(1, units, T, device="cuda") for _ in range(4))
    status, ws = torch.zeros(1, dtype=torch.int32, device="cuda"), torch.empty(V.vatp_workspace_bytes(p), dtype=torch.uint8, device="cuda")
    to = dict(attn_acc=acc, vnorm=vnorm, score=score, workspace=ws, dev_status=status)
    if call == "lse":
        given = torch.zeros_like(lse)
        given[0, :, first:] = want_lse.float()
        V.vatp_prefill_scores_from_lse(p, q, k, v, given, lse_out=lse, **to)
        assert torch.equal(lse, given)
    else:
        V.vatp_prefill_scores(p, q, k, v, lse_out=lse, **to)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    tol = P.TOL["f32"]
    assert torch.all((lse[0, :, first:].double() - want_lse).abs() <= 10 * tol)
    assert torch.all(lse[0, :, :first] == 0)
    assert torch.all((acc[0].double() - want).abs() <= tol * want)
    n = v[0].double().norm(p={"l1": 1, "l2": 2, "linf": float("inf")}[norm], dim=-1)
    assert torch.all((vnorm[0].double() - n).abs() <= tol * n)
    assert torch.equal(score, acc * vnorm)


def _simt_clusters(units, T, window):
    """Tile rows and the two passes' cluster sizes of an fp32 scoring call on 148 SMs."""
    rows = window if 0 < window < T else T
    size = 128 if units * ((rows + 127) // 128) >= 2 * 148 else 64
    qtiles, ktiles = (rows + size - 1) // size, (T + size - 1) // size

    def clusters(tiles, most):
        cs = 1
        while cs < 8 and tiles * units * cs * 2 <= 2 * 148 and cs < most:
            cs *= 2
        return cs
    return size, clusters(qtiles, ktiles), clusters(ktiles, qtiles)


@pytest.mark.parametrize("d,units,kv,T,window,call,plan", [
    (64, 1, 0, 1, 0, "scores", (64, 1, 1)),         # one token
    (64, 1, 0, 64, 0, "scores", (64, 1, 1)),        # one tile
    (64, 3, 0, 66, 0, "scores", (64, 2, 2)),        # two tiles, two rows in the second
    (128, 2, 0, 200, 0, "scores", (64, 4, 4)),
    (64, 2, 0, 514, 0, "scores", (64, 8, 8)),       # more CTAs than the first rows have key tiles
    (128, 1, 0, 700, 33, "scores", (64, 8, 1)),     # a window of less than a tile
    (64, 9, 0, 450, 0, "scores", (64, 4, 4)),
    (64, 8, 0, 700, 0, "scores", (64, 2, 2)),       # up to six tiles per CTA of a cluster
    (64, 50, 0, 700, 0, "scores", (128, 1, 1)),     # the large tiles
    (128, 50, 0, 700, 0, "scores", (128, 1, 1)),
    (64, 8, 2, 514, 0, "scores", (64, 8, 8)),       # grouped queries: four rounds of both passes, on two units each
    (64, 200, 100, 300, 0, "scores", (128, 1, 1)),
    (64, 2, 0, 514, 0, "lse", (64, 8, 8)),          # normalisers given: pass 2 alone
    (64, 50, 0, 700, 0, "lse", (128, 1, 1)),
    (64, 3, 0, 514, 100, "lse", (64, 8, 2)),
])
def test_fp32_scoring_right_behind_a_kernel_that_releases_it_early(d, units, kv, T, window, call, plan):
    """The fp32 passes enqueued right behind the kernel that writes their queries, keys and values and that lets its dependents
    start long before: another scoring call, whose indicators, norms and scores are the inputs.  With clusters of every size and
    both tiles, over and over on the same buffers: an input read too early is the one of the round before."""
    V = P.vatp()
    hk = kv or units
    assert _simt_clusters(hk, T, window) == plan
    f32 = dict(dtype=torch.float32, device="cuda")
    g = torch.Generator(device="cuda").manual_seed(T + d)
    n = units * T * d
    T0 = 128 if n % 128 == 0 else 64                  # the writer: short prompts, as many as it takes
    assert n % T0 == 0
    p0 = V.make_params(batch=1, heads=n // T0, seq_len=T0, head_dim=64, dtype="f32", budget=T0)
    p = V.make_params(batch=1, heads=units, kv_heads=kv, seq_len=T, head_dim=d, dtype="f32", budget=T, scale=0.001,
                      indicator="window" if window else "h2o", window=window)
    first = max(T - window, 0) if window else 0
    sources = [torch.randn(1, n // T0, T0, 64, generator=g, **f32) for _ in range(3)]
    made, ws0 = torch.zeros(3, 1, n // T0, T0, **f32), torch.empty(V.vatp_workspace_bytes(p0), dtype=torch.uint8, device="cuda")
    ws, status = torch.empty(V.vatp_workspace_bytes(p), dtype=torch.uint8, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
    rows = [made[0].view(1, units, T, d)] + [made[i].view(-1)[:hk * T * d].view(1, hk, T, d) for i in (1, 2)]

    def write(src):
        V.vatp_prefill_scores(p0, src, src, src, attn_acc=made[0], vnorm=made[1], score=made[2], workspace=ws0, dev_status=status)

    def score(given):
        lse = torch.zeros(1, units, T, **f32)
        out = torch.zeros(3, 1, hk, T, **f32)
        to = dict(attn_acc=out[0], vnorm=out[1], score=out[2], workspace=ws, dev_status=status)
        if call == "lse":
            return lambda: V.vatp_prefill_scores_from_lse(p, *rows, given, lse_out=lse, **to), lse, out
        return lambda: V.vatp_prefill_scores(p, *rows, lse_out=lse, **to), lse, out

    want = []
    for src in sources:
        write(src)
        torch.cuda.synchronize()
        q, k, v = (x.double() for x in rows)
        s = (q @ k.repeat_interleave(units // hk, 1).transpose(-1, -2)) * p.scale
        s.masked_fill_(torch.ones(T, T, dtype=torch.bool, device="cuda").triu(1), -torch.inf)
        lse = torch.logsumexp(s, -1)
        acc = torch.softmax(s, -1)[..., first:, :].sum(-2).view(1, hk, units // hk, T).mean(2)
        norm = v.abs().sum(-1)
        want.append((lse.float(), lse, acc, norm))
        del s
    calls = [score(want[i % 3][0]) for i in range(9)]
    torch.cuda.synchronize()
    for i, (run, _, _) in enumerate(calls):
        write(sources[i % 3])
        run()
    torch.cuda.synchronize()
    assert int(status) == 0
    tol = P.TOL["f32"]
    for i, (_, lse, out) in enumerate(calls):
        _, want_lse, acc, norm = want[i % 3]
        assert (lse.double() - want_lse)[..., first:].abs().max() <= 10 * tol
        for got, ref in ((out[0], acc), (out[1], norm), (out[2], acc * norm)):
            assert ((got.double() - ref).abs() <= 2 * tol * ref + 1e-30).all()      # (the score: two factors)
        assert torch.equal(out, calls[i % 3][2])
