"""Decode on the group-major cache: heads of a KV group as columns of the products (1 to 8, even and odd), at the edges of a
tile, with the rotation at read and without."""
import numpy as np
import pytest
import torch

import atf_inputs as gen
from oracle import atf_oracle as orc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("G,d,L", [(1, 128, 1), (2, 128, 63), (5, 128, 65), (8, 128, 1000), (1, 64, 127), (4, 64, 129), (7, 64, 2500), (8, 64, 16),
                                   (3, 128, 15), (6, 64, 31)])
def test_heads_of_a_group(G, d, L, mode):
    import paper_2608_02947_b200 as atf
    B, Hkv = 2, 3
    g = torch.Generator().manual_seed(100 * G + L)
    q, K, V = [torch.randn(s, generator=g).to(torch.bfloat16) for s in ((B, G * Hkv, d), (B, Hkv, L, d), (B, Hkv, L, d))]
    W, theta = atf.atf_window_table(1e4, d, 2.0, L)
    W = torch.clamp(W, max=max(1, (3 * L) // 4))  # keys that no pair reaches, too
    tabs = atf.atf_rope_tables(theta, d, L + 100, pos0=3)
    Kg = atf.new_kcache_groups(B, Hkv, L + 100, d, "cuda")
    atf.atf_kcache_pack(K.cuda(), Kg)
    fn = orc.decode if mode == 0 else orc.coarse_decode
    for tables, Kr in ((None, gen.to_f64(K)), (tabs, orc.rope_half_split(gen.to_f64(K), theta.numpy(), 3))):
        O, lse = atf.atf_decode(q.cuda(), Kg, V.cuda(), table=W, mode=mode, return_lse=True, rope_tables=tables)
        Or, Lr = fn(gen.to_f64(q), Kr, gen.to_f64(V), W.numpy())
        err = np.abs(gen.to_f64(O) - Or)
        assert err.max() <= 2e-2 and err.mean() <= 2e-3  # P and O rounded to bf16, values of N(0, 1)
        assert np.abs(lse.double().cpu().numpy() - Lr).max() <= 1e-3
