"""Exact mode: the per-cell finish adds a pair's term to a score with one rounding to nearest (no bias)."""
import math

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("split", [False, True])
def test_added_pair_is_rounded_to_nearest(d, split):
    import paper_2608_02947_b200 as atf
    H, N, h = 48, 256, d // 2
    # Rows 160..191 see key 86 of the other tile at distances 74..105.  Pair 0 (width 111) is live there and not kept in the
    # matrix product of that quarter of the rows (its middle distance is 112): its term is what the finish adds.
    rows, key = slice(160, 192), 86
    W = torch.full((h,), N, dtype=torch.int64)
    W[0] = 111
    rng = np.random.default_rng(11)
    Q, K = np.zeros((1, H, N, d)), np.zeros((1, H, N, d))
    # The product's part: integers, 2048 <= sum < 4096, exact in fp32.  Every other key has score 0 in these dims.
    rest = [i for i in range(d) if i not in (0, h)]
    Q[0, :, :, rest] = rng.integers(0, 8, (len(rest), H, N)) // (d // 64)
    K[0, :, key, rest] = rng.integers(0, 8, (len(rest), H))
    Q[0, :, :, 1], K[0, :, key, 1] = 64, 32
    # Pair 0: 8-bit values whose products reach five bits below the last place of the sum.
    Q[0, :, :, [0, h]] = rng.integers(128, 256, (2, H, N)) / 128
    K[0, :, key, [0, h]] = rng.integers(128, 256, (2, H)) / 1024
    V = torch.zeros((1, H, N, d), dtype=torch.bfloat16, device="cuda")
    kind = torch.float32 if split else torch.bfloat16
    call = atf.atf_prefill_split if split else atf.atf_prefill
    q, k = torch.from_numpy(Q).to(kind).cuda(), torch.from_numpy(K).to(kind).cuda()
    assert torch.equal(q.double().cpu(), torch.from_numpy(Q)) and torch.equal(k.double().cpu(), torch.from_numpy(K))
    _, lse = call(q, k, V, table=W)
    S = (Q[0, :, rows] * K[0, :, key][:, None]).sum(-1)
    assert S.min() >= 2048 and S.max() < 4096
    # One key holds the whole weight: LSE = S / sqrt(d), times the fp32 constants log2(e) / sqrt(d) and ln 2 of the kernel.
    c = float(np.float32(math.log2(math.e)) / np.sqrt(np.float32(d))) * float(np.float32(math.log(2.0)))
    unit = 2.0 ** -12 * c  # last place of S, as LSE
    bias = ((lse[0, :, rows].double().cpu().numpy() - S * c) / unit).mean()
    # Roundings to nearest average out: S and the two products behind LSE spread by less than 0.7 units, over 1536 rows
    # 0.02.  A sum cut off towards zero is 0.5 units low.
    assert abs(bias) < 0.12, bias
