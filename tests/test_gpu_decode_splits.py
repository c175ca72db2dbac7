"""Decode: the number of splits of a call, at the sizes where the deal of tiles to splits and the merge can go wrong (one
tile, one key over a tile, a last split with fewer tiles, more splits than a merge batch), and with scratch for one."""
import ctypes as C

import numpy as np
import pytest
import torch

import atf_inputs as gen
from oracle import atf_oracle as orc

pytestmark = pytest.mark.gpu
HEADER = 256 + 16384 * 4  # status words and split counters


def _case(B, Hq, Hkv, d, L, seed):
    w = gen.Workload("splits", B, Hq, Hkv, d, L, 5e5, 2.0, gen.LLAMA3_SCALING, gen.SEED0 + seed)
    q, K, V = gen.decode_inputs(w)
    Wo, _ = orc.window_table(w.base, w.d, w.k, w.N, w.scaling)
    return q, K, V, Wo


def _check(O, lse, ref):
    # P and O are rounded to bf16 (2^-9 each): the tolerances of the other decode tests
    err = np.abs(gen.to_f64(O) - ref[0])
    assert err.max() <= 2e-2 and err.mean() <= 2e-3
    if lse is not None:
        assert np.abs(lse.double().cpu().numpy() - ref[1]).max() <= 1e-3


@pytest.mark.parametrize("B,Hq,Hkv,d,L", [(1, 3, 1, 128, 1), (1, 3, 1, 128, 64), (1, 24, 8, 128, 65), (1, 24, 8, 128, 1023),
                                          (2, 24, 8, 128, 2113), (1, 14, 2, 64, 129), (1, 14, 2, 64, 1000), (1, 8, 1, 64, 20000),
                                          (1, 7, 1, 128, 9000), (40, 8, 8, 64, 300)])
def test_splits_against_oracle(B, Hq, Hkv, d, L):
    import paper_2608_02947_b200 as atf
    q, K, V, W = _case(B, Hq, Hkv, d, L, 800 + L)
    ref = orc.decode(gen.to_f64(q), gen.to_f64(K), gen.to_f64(V), W)
    q, K, V = q.cuda(), K.cuda(), V.cuda()
    for cache in (K, atf.atf_kcache_pack(K)):
        _check(*atf.atf_decode(q, cache, V, table=W, return_lse=True), ref)


def test_scratch_for_one_split():
    import paper_2608_02947_b200 as atf
    lib = atf.lib()
    B, Hq, Hkv, d, L = 1, 24, 8, 128, 1000
    q, K, V, W = _case(B, Hq, Hkv, d, L, 77)
    ref = orc.decode(gen.to_f64(q), gen.to_f64(K), gen.to_f64(V), W)
    q, K, V = q.cuda(), K.cuda(), V.cuda()
    one = HEADER + (Hq * (d + 2) * 4 + 255) // 256 * 256
    assert lib.atf_workspace_bytes(1, B, Hq, Hkv, L, d) > one
    ws = torch.zeros(one, dtype=torch.uint8, device="cuda")
    O = torch.empty_like(q)
    tab = (C.c_int64 * (d // 2))(*[int(x) for x in W])
    opts = atf.binding._Opts()
    for nbytes, code in ((one, 0), (one - 256, 4)):
        opts.workspace, opts.workspace_bytes = ws.data_ptr(), nbytes
        p = [C.c_void_p(t.data_ptr()) for t in (q, K, V, O)]
        assert lib.atf_decode_ex(*p, B, Hq, Hkv, L, d, tab, C.byref(opts), C.c_void_p(torch.cuda.current_stream().cuda_stream)) == code
    torch.cuda.synchronize()
    _check(O, None, ref)


@pytest.mark.parametrize("L", [700, 1000, 2100])
def test_infinite_value_stays_in_its_column(L):
    """An infinite element of V makes its output column infinite and no other (11, 16 and more splits, in the last one too)."""
    import paper_2608_02947_b200 as atf
    q, K, V, W = _case(1, 6, 2, 128, L, 41)
    q, K, V = q.cuda(), K.cuda(), V.cuda()
    for cache in (K, atf.atf_kcache_pack(K)):
        plain = atf.atf_decode(q, cache, V, table=W)
        for key in (3, L // 2, L - 1):
            v = V.clone()
            v[0, 0, key, 5] = float("inf")
            v[0, 0, key, 77] = -float("inf")
            want = plain.clone()
            want[0, :3, 5] = float("inf")
            want[0, :3, 77] = -float("inf")
            assert torch.equal(atf.atf_decode(q, cache, v, table=W), want), key


@pytest.mark.parametrize("B,Hq,Hkv,d,L,least,most", [
    (40, 24, 8, 128, 4096, 3, 8),    # 320 groups: one split each would leave 24 CTAs to walk 64 tiles on an idle GPU (181 us, 136 with 5)
    (75, 28, 4, 128, 8192, 4, 12),   # 300 groups (330 us with one split, 233 with 7)
    (51, 28, 4, 128, 65536, 3, 17),  # 204 groups, long contexts
    (1, 24, 8, 128, 512, 8, 8)])
def test_split_count(B, Hq, Hkv, d, L, least, most):
    """Splits that a call takes: as many slots of its scratch are written, and its size does not fall as L grows."""
    import paper_2608_02947_b200 as atf
    size = [atf.atf_workspace_bytes(1, B, Hq, Hkv, n, d) for n in (1, L // 2, L, 2 * L, (2 ** 31 - 1) // d)]
    assert size == sorted(size)
    ws = torch.zeros(size[2], dtype=torch.uint8, device="cuda")
    q = torch.randn((B, Hq, d), device="cuda").to(torch.bfloat16)
    K = torch.randn((1, 1, L, d), device="cuda").to(torch.bfloat16).expand(B, Hkv, L, d).contiguous()
    opts = atf.binding._Opts()
    opts.workspace, opts.workspace_bytes = ws.data_ptr(), size[2]
    O = torch.empty_like(q)
    p = [C.c_void_p(t.data_ptr()) for t in (q, K, K, O)]
    assert atf.lib().atf_decode_ex(*p, B, Hq, Hkv, L, d, None, C.byref(opts), C.c_void_p(torch.cuda.current_stream().cuda_stream)) == 0
    part = ws[HEADER:].view(torch.float32)
    written = int(part.nonzero().max()) + 1
    splits = -(-written // (B * Hq * (d + 2)))
    assert least <= splits <= most


def test_one_scratch_for_a_generation():
    """The binding's workspace does not change while a context grows token by token or by leaps."""
    import paper_2608_02947_b200 as atf
    torch.cuda.synchronize()
    atf.binding._ws = None  # the next call binds a new one
    B, Hq, Hkv, d = 1, 24, 8, 128
    K = torch.randn((B, Hkv, 20000, d), device="cuda").to(torch.bfloat16)
    q = torch.randn((B, Hq, d), device="cuda").to(torch.bfloat16)
    seen = set()
    for L in (60, 61, 65, 700, 5000, 20000, 300):
        k = K[:, :, :L].contiguous()
        atf.atf_decode(q, k, k)
        seen.add((atf.binding._ws.data_ptr(), atf.binding._ws.numel()))
    torch.cuda.synchronize()
    assert len(seen) == 1


def test_workspace_sized_by_the_caller_stays():
    """A workspace of the size asked for one length is kept for calls of that length (and replaced for a longer one)."""
    import paper_2608_02947_b200 as atf
    B, Hq, Hkv, d, L = 1, 14, 2, 64, 1000
    torch.cuda.synchronize()
    atf.binding._ws = None
    ws = atf.ensure_workspace(atf.atf_workspace_bytes(1, B, Hq, Hkv, L, d), "cuda:0")
    K = torch.randn((B, Hkv, 8 * L, d), device="cuda").to(torch.bfloat16)
    q = torch.randn((B, Hq, d), device="cuda").to(torch.bfloat16)
    for n in (L, L - 1, 1):
        k = K[:, :, :n].contiguous()
        atf.atf_decode(q, k, k)
        assert atf.binding._ws is ws
    atf.atf_decode(q, K, K)
    assert atf.binding._ws.numel() > ws.numel()
    torch.cuda.synchronize()
