"""Dispatch branches of the rotation (threads per row segment) and the prefill's overlapped launch, at their borders."""
import numpy as np
import pytest
import torch

import atf_inputs as gen
from oracle import atf_oracle as orc

pytestmark = pytest.mark.gpu


# one, two, four and eight threads a segment (d = 128: from 18913, 9457, 4729 rows down), rows that do not fill a block,
# fewer heads than threads
@pytest.mark.parametrize("H,N,d", [(3, 18945, 128), (2, 18912, 128), (5, 9440, 128), (1, 4700, 128), (9, 33, 128), (3, 1, 64),
                                   (3, 2501, 64), (1, 37889, 64)])
def test_rope_threads_per_segment(H, N, d):
    import paper_2608_02947_b200 as atf
    X = gen.normal_bf16((1, H, N, d), 4242 + N)
    _, theta = orc.window_table(5e5, d, 2.0, N)
    ref = orc.rope_half_split(gen.to_f64(X), theta, pos0=77)  # rounded to bf16 once
    out = gen.to_f64(atf.atf_rope(X.cuda(), theta, pos0=77))
    # fp64 angles on both sides, one rounding: a tie may fall either way, one bf16 unit (2^-7 of the value at most)
    assert np.all(np.abs(out - ref) <= 2.0 ** -7 * np.abs(ref) + 1e-30)
    assert (out != ref).mean() < 1e-4
    f = torch.randn((1, H, N, d), generator=torch.Generator().manual_seed(N))
    ref = orc.rope_half_split(f.double().numpy(), theta, pos0=77, round_bf16=False)
    out = atf.atf_rope_f32(f.cuda(), theta, pos0=77).double().cpu().numpy()
    assert np.all(np.abs(out - ref) <= 2.0 ** -23 * np.abs(ref) + 1e-30)  # one rounding to fp32


@pytest.mark.parametrize("split", [False, True])
def test_prefill_back_to_back_and_captured(split):
    """Calls that follow one another on one workspace, with new inputs each, give what each gives alone, also in a graph."""
    import paper_2608_02947_b200 as atf
    d, N, Nq = 128, 1000, 700
    W, _ = atf.atf_window_table(5e5, d, 2.0, N)
    gen_ = torch.Generator().manual_seed(5)
    kind = torch.float32 if split else torch.bfloat16
    cases = [[torch.randn((1, h, n, d), generator=gen_).to(t).cuda() for h, n, t in ((6, Nq, kind), (2, N, kind), (2, N, torch.bfloat16))]
             for _ in range(3)]
    call = atf.atf_prefill_split if split else atf.atf_prefill
    alone = []
    for q, k, v in cases:
        alone.append([t.clone() for t in call(q, k, v, table=W)])
        torch.cuda.synchronize()
    together = [call(q, k, v, table=W) for q, k, v in cases]
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        captured = [call(q, k, v, table=W) for q, k, v in cases]
    g.replay()
    torch.cuda.synchronize()
    for got in (together, captured):
        for a, b in zip(alone, got):
            assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])


@pytest.mark.parametrize("split", [False, True])
def test_prefill_other_schedule_in_each_call(split):
    """Calls on one workspace whose band schedules differ (table, mode, lengths), Q rotated in place right before each: the
    words that the call before left, or a Q read too early, would show as other bits."""
    import paper_2608_02947_b200 as atf
    d = 128
    rope = atf.atf_rope_f32 if split else atf.atf_rope
    call = atf.atf_prefill_split if split else atf.atf_prefill
    kind = torch.float32 if split else torch.bfloat16
    gen_ = torch.Generator().manual_seed(6)
    forms = [(1700, 1700, 2.0, atf.ATF_MODE_EXACT), (1000, 300, None, atf.ATF_MODE_EXACT), (1700, 900, 0.5, atf.ATF_MODE_COARSE),
             (1700, 1700, 0.25, atf.ATF_MODE_EXACT), (129, 129, 2.0, atf.ATF_MODE_COARSE), (1700, 1700, None, atf.ATF_MODE_EXACT)]
    cases = []
    for N, Nq, k, mode in forms:
        W, theta = atf.atf_window_table(5e5, d, k or 2.0, N)
        q, key, v = [torch.randn((1, h, n, d), generator=gen_).to(t).cuda()
                     for h, n, t in ((6, Nq, kind), (2, N, kind), (2, N, torch.bfloat16))]
        cases.append((q, key, v, None if k is None else W, theta, N - Nq, mode))

    def step(q, key, v, W, theta, pos0, mode):
        q = q.clone()
        return call(rope(q, theta, pos0=pos0), key, v, table=W, mode=mode)

    alone = []
    for c in cases:
        alone.append([t.clone() for t in step(*c)])
        torch.cuda.synchronize()
    order = [0, 1, 2, 3, 4, 5, 3, 0, 4, 1, 5, 2]
    for _ in range(3):
        together = [(i, step(*cases[i])) for i in order]
        torch.cuda.synchronize()
        for i, got in together:
            assert torch.equal(alone[i][0], got[0]) and torch.equal(alone[i][1], got[1])
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        captured = [(i, step(*cases[i])) for i in order]
    g.replay()
    torch.cuda.synchronize()
    for i, got in captured:
        assert torch.equal(alone[i][0], got[0]) and torch.equal(alone[i][1], got[1])


# heads dealt over blocks (few rows; a last block with fewer heads than threads; fp32 up to twelve blocks an SM), a last row
# that does not fill a block, fp32 with the next head on its way (more than 126 MB; heads that do not divide by the threads)
@pytest.mark.parametrize("B,H,N,d,f32", [(8, 24, 1, 128, False), (64, 28, 1, 64, False), (3, 67, 5, 128, False), (2, 9, 440, 64, False),
                                         (8, 24, 1, 128, True), (3, 67, 5, 64, True), (5, 11, 700, 128, True), (1, 6, 9001, 64, True),
                                         (2, 53, 2401, 128, True), (1, 3, 90001, 128, True)])
def test_rope_heads_over_blocks(B, H, N, d, f32):
    import paper_2608_02947_b200 as atf
    _, theta = orc.window_table(5e5, d, 2.0, N)
    X = torch.randn((B, H, N, d), generator=torch.Generator().manual_seed(N))
    if not f32:
        X = X.to(torch.bfloat16)
    out = (atf.atf_rope_f32 if f32 else atf.atf_rope)(X.cuda(), theta, pos0=1234)
    # a head at a time, as the oracle rotates it: fp64, one rounding (a tie may fall either way)
    for b, h in {(0, 0), (0, H - 1), (B - 1, 0), (B - 1, H - 1), (B // 2, H // 2), (B - 1, min(8, H - 1))}:
        ref = orc.rope_half_split(X[b, h].double().numpy(), theta, pos0=1234, round_bf16=not f32)
        got = out[b, h].double().cpu().numpy()
        assert np.all(np.abs(got - ref) <= 2.0 ** (-23 if f32 else -7) * np.abs(ref) + 1e-30)
    # every head is rotated, and once: the length of a pair does not change
    n = d // 2
    was, now = X.cuda().double(), out.double()
    was, now = was[..., :n] ** 2 + was[..., n:] ** 2, now[..., :n] ** 2 + now[..., n:] ** 2
    assert torch.all((was - now).abs() <= 2.0 ** (-21 if f32 else -6) * was + 1e-30)
    if N > 1:
        assert not torch.equal(out[..., 1, :], X.cuda()[..., 1, :])


@pytest.mark.parametrize("d,mode,outlier", [(128, 0, False), (128, 1, False), (64, 0, True), (128, 0, True)])
def test_prefill_output_over_its_queries(d, mode, outlier):
    """O written over Q, also where tiles are run twice (outlier logits read Q again)."""
    import paper_2608_02947_b200 as atf
    N, Nq = 1500, 1100
    g = torch.Generator().manual_seed(d + mode)
    Q, K, V = [torch.randn((2, h, n, d), generator=g) for h, n in ((6, Nq), (2, N), (2, N))]
    W, theta = atf.atf_window_table(5e5, d, 2.0, N)
    if outlier:
        for t in (Q, K):
            t[..., d // 2 - 4:d // 2] *= 8
            t[..., d - 4:] *= 8
    Q, K, V = (t.to(torch.bfloat16).cuda() for t in (Q, K, V))
    O, lse = atf.atf_prefill(Q, K, V, table=W, mode=mode)
    got, lse2 = atf.atf_prefill(Q, K, V, table=W, mode=mode, O=Q)
    assert got.data_ptr() == Q.data_ptr()
    assert torch.equal(got, O) and torch.equal(lse2, lse)


@pytest.mark.parametrize("N", [300, 14817])
def test_prefill_and_decode_in_turn_on_one_workspace(N):
    """The decode's partials lie where the next prefill's schedule is written: 300 layer steps give what the first one gave."""
    import paper_2608_02947_b200 as atf
    Hq, Hkv, d = 14, 2, 64
    W, theta = atf.atf_window_table(1e6, d, 2.0, N)
    table = atf.WindowTable(W)
    g = torch.Generator(device="cuda").manual_seed(N)
    Q, K, V = [torch.randn((1, h, N, d), generator=g, device="cuda").to(torch.bfloat16) for h in (Hq, Hkv, Hkv)]
    cache = atf.new_kcache_groups(1, Hkv, N, d, "cuda")
    atf.atf_rope(Q, theta)
    atf.atf_rope(K, theta)
    q = Q[:, :, -1].contiguous()

    def step():
        O, lse = atf.atf_prefill(Q, K, V, table=table, kcache_groups=cache)
        return O, lse, atf.atf_decode(q, cache, V, table=table)

    first = step()
    other = torch.zeros((), dtype=torch.bool, device="cuda")
    for _ in range(300):
        for a, b in zip(first, step()):
            other |= (a != b).any()
    assert not other.item()
    atf.binding.check_status()
