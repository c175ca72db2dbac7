"""Prefill, exact mode, with widths that reach every key: the form of the kernel without a per-cell finish, at its border
(the narrowest width one below the largest distance takes the other form), and its time."""
import numpy as np
import pytest
import torch

import atf_inputs as gen
from oracle import atf_oracle as orc

pytestmark = pytest.mark.gpu


def _inputs(d, Nq, N, seed):
    g = torch.Generator().manual_seed(seed)
    return [torch.randn((1, h, n, d), generator=g).to(torch.bfloat16).cuda() for h, n in ((4, Nq), (2, N), (2, N))]


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("N,Nq", [(1, 1), (129, 129), (513, 513), (513, 200), (640, 3)])
def test_border_width_against_oracle(d, N, Nq):
    import paper_2608_02947_b200 as atf
    Q, K, V = _inputs(d, Nq, N, N + Nq)
    full = atf.atf_prefill(Q, K, V)
    coarse = atf.atf_prefill(Q, K, V, mode=atf.ATF_MODE_COARSE)
    assert torch.equal(full[0], coarse[0]) and torch.equal(full[1], coarse[1])
    q, k, v = (gen.to_f64(t.cpu()) for t in (Q, K, V))
    for w0 in (N - 1, N - 2):
        if w0 < 0:
            continue
        W = np.full(d // 2, N, dtype=np.int64)
        W[0] = w0
        kept = torch.zeros(4, dtype=torch.int64, device="cuda")
        O, lse = atf.atf_prefill(Q, K, V, table=W, kept_terms=kept)
        assert kept.cpu().tolist() == [orc.kept_terms_interval(W, N - Nq, N)] * 4
        if w0 == N - 1:
            assert torch.equal(O, full[0]) and torch.equal(lse, full[1])
        for h in range(4):
            ref = orc.attention_appended_rows(q[0, h], k[0, h // 2], v[0, h // 2], W, N - Nq)
            err = np.abs(gen.to_f64(O[0, h].cpu()) - ref[0])
            assert err.max() <= 2e-2 and err.mean() <= 2e-3
            assert np.abs(lse[0, h].double().cpu().numpy() - ref[1]).max() <= 1e-3


def test_first_chunk_inside_the_narrowest_window_is_the_single_shot():
    """Chunks whose keys all lie inside every window take the full form, the single shot the windowed one: same bits."""
    import paper_2608_02947_b200 as atf
    N, d = 900, 128
    Q, K, V = _inputs(d, N, N, 9)
    W = np.sort(np.r_[[400, 450, 500, 700], np.full(d // 2 - 4, N)]).astype(np.int64)
    O, lse = atf.atf_prefill(Q, K, V, table=W)
    for n in (1, 100, 257, 401, 402):
        part = atf.atf_prefill(*(t[:, :, :n].contiguous() for t in (Q, K, V)), table=np.minimum(W, n))
        assert torch.equal(part[0], O[:, :, :n]) and torch.equal(part[1], lse[:, :, :n])


def test_full_attention_is_not_slower_than_coarse():
    """Both are one computation: the exact mode's pays for no copy of Q and no release of K by the softmax warps."""
    import paper_2608_02947_b200 as atf
    g = torch.Generator(device="cuda").manual_seed(1)
    Q, K, V = [torch.randn((1, h, 1000, 128), generator=g, device="cuda").to(torch.bfloat16) for h in (24, 8, 8)]

    def us(mode):
        best = float("inf")
        for _ in range(10):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(20):
                atf.atf_prefill(Q, K, V, mode=mode)
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b) / 20 * 1e3)
        return best

    for mode in (atf.ATF_MODE_EXACT, atf.ATF_MODE_COARSE):
        us(mode)
    # 43 against 25 us where the exact form was taken
    assert us(atf.ATF_MODE_EXACT) <= 1.25 * us(atf.ATF_MODE_COARSE)
