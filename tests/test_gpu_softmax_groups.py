"""The prefill's softmax groups take whole key tiles in turn in coarse mode (and in full attention at d = 64): one, odd and even
numbers of tiles, windows that end, and the safe second pass.  Calls that count terms never take turns, so they are the reference,
bit for bit; the oracle is the other."""
import numpy as np
import pytest
import torch

import atf_inputs as gen
from oracle import atf_oracle as orc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["window", "ending", "full"])
@pytest.mark.parametrize("d,N,far", [(128, 100, False), (128, 130, False), (64, 257, True), (128, 400, True), (64, 1153, False), (128, 2500, False),
                                     (64, 2311, True)])
def test_groups_in_turn(d, N, far, kind):
    import paper_2608_02947_b200 as atf
    H, h = 2, d // 2
    rng = np.random.default_rng(N + d)
    Q, K, V = (torch.from_numpy(rng.standard_normal((1, n, N, d))).float() for n in (H, 1, 1))
    if far:  # the oldest keys have logits in the hundreds, past what a reference from the diagonal tile can hold
        K[:, :, :20] *= 40
        Q *= 4
    Q, K, V = (t.to(torch.bfloat16) for t in (Q, K, V))
    W = np.full(h, N, dtype=np.int64)
    if kind != "full":
        W[:10] = [3, 17, 90, 130, 200, 460, 777, 1100, 1500, 1999]
        if kind == "ending":  # keys beyond the widest window are dropped
            W[10:] = 2100
    W = np.minimum(W, N)
    table = torch.from_numpy(W)
    q, k, v = Q.cuda(), K.cuda(), V.cuda()
    O, lse = atf.atf_prefill(q, k, v, table=table, mode=1)
    O1, lse1 = atf.atf_prefill(q, k, v, table=table, mode=1, kept_terms=torch.zeros(H, dtype=torch.int64, device="cuda"))
    atf.binding.check_status()
    assert torch.equal(O, O1) and torch.equal(lse, lse1)
    if kind == "full":
        O1, lse1 = atf.atf_prefill(q, k, v)
        assert torch.equal(O, O1) and torch.equal(lse, lse1)
    n0 = N // 3 + 1  # appended rows: the same bits again (an unaligned cut may choose the other pass)
    if not far:
        O1, lse1 = atf.atf_prefill(q[:, :, n0:].contiguous(), k, v, table=table, mode=1)
        assert torch.equal(O1, O[:, :, n0:]) and torch.equal(lse1, lse[:, :, n0:])
    rows = sorted(set(range(max(0, N - 200), N)) | set(range(0, N, 11)))
    for i in range(H):
        Or, Lr = orc.coarse_attention_rows(gen.to_f64(Q[0, i]), gen.to_f64(K[0, 0]), gen.to_f64(V[0, 0]), W, rows)
        # scores are sums of d exact products in fp32: 2^-18 of the largest logit covers their rounding
        assert np.abs(lse[0, i].double().cpu().numpy()[rows] - Lr).max() <= 1e-3 + 2.0 ** -18 * np.abs(Lr).max()
        err = np.abs(gen.to_f64(O[0, i][rows]) - Or)
        assert err.max() <= 2e-2 and err.mean() <= 2e-3
