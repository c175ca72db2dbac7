"""How a prefill's tiles are dealt to blocks: groups of heads (a whole one, a ragged last one), and tiles that two blocks share."""
import pytest
import torch

pytestmark = pytest.mark.gpu
SMS = 148  # tiles that are cut, if any


def _cut_flags(ws, B, Hq, Hkv, N, Nq, d, split=False):
    """The flags of the cut tiles, in the workspace behind schedule, operands and state."""
    part = lambda heads, rows: (B * heads * rows * d * 2 + 255) // 256 * 256
    at = 256 + 4 * 16384 + (((N + 127) // 128 + 1) * 32 + 255) // 256 * 256
    at += 2 * (part(Hq, Nq) + part(Hkv, N)) if split else part(Hkv, N)
    at += SMS * 128 * (d + 3) * 4
    return ws[at:at + 4 * SMS].view(torch.int32)


def _group(B, Hq, Hkv, N, Nq, d, split, W):
    """Heads whose tiles are dealt out together, longest rows first, by the rule beside the launch; 1: head by head."""
    tiles = (N + 127) // 128 - (N - Nq) // 128
    reach = (int(W.max()) + 127) // 128 + 1
    longest, shortest = min((N + 127) // 128, reach), min((N - Nq) // 128 + 1, reach)
    if 2 * shortest > longest or (tiles >= 64 and 8 * (-tiles * B * Hq % SMS) * shortest > SMS * (longest + shortest)):
        return 1
    per_kv = Hq // Hkv
    fit = (64 << 20) // (N * d * 2 * (3 if split else 2)) * per_kv
    if fit == 0:
        return 1
    groups = -(-B * Hq // fit)
    return min(-(-(-(-B * Hq // groups)) // per_kv) * per_kv, B * Hq)


# rows of different lengths; keys and values of a KV head: 36 MB (one a group), 13 MB (two groups, the last one short); split
# mode: 27 MB (two groups, the last one short); rows of about the same length: head by head; so, too, where a head has many tiles
# and the last wave is not full, the first two against the next two; the next two lie on either side of 64 tiles,
# the last two of 64 MB
@pytest.mark.parametrize("B,Hq,Hkv,N,Nq,d,split,group", [
    (3, 6, 2, 70000, 36000, 128, False, 1), (7, 2, 1, 50000, 26000, 64, False, 1),
    (3, 6, 2, 70000, 35696, 128, False, 3), (7, 2, 1, 50000, 26960, 64, False, 8),
    (3, 3, 1, 35000, 18000, 128, True, 6), (2, 6, 2, 9000, 300, 128, False, 1),
    (1, 14, 2, 13607, 8000, 64, False, 1), (1, 14, 2, 13600, 7900, 64, False, 14),
    (1, 2, 1, 131072, 131072, 128, False, 2), (1, 2, 1, 131073, 131073, 128, False, 1)])
def test_heads_in_groups(B, Hq, Hkv, N, Nq, d, split, group):
    import paper_2608_02947_b200 as atf
    g = torch.Generator(device="cuda").manual_seed(N)
    kind = torch.float32 if split else torch.bfloat16
    Q, K, V = [torch.randn((B, h, n, d), generator=g, device="cuda").to(t) for h, n, t in ((Hq, Nq, kind), (Hkv, N, kind), (Hkv, N, torch.bfloat16))]
    W, _ = atf.atf_window_table(5e5, d, 2.0, N)
    assert _group(B, Hq, Hkv, N, Nq, d, split, W) == group
    call = atf.atf_prefill_split if split else atf.atf_prefill
    O, lse = call(Q, K, V, table=W)
    for b in range(B):
        for k in range(Hkv):
            h = slice(k * Hq // Hkv, (k + 1) * Hq // Hkv)
            o, l = call(Q[b:b + 1, h].contiguous(), K[b:b + 1, k:k + 1].contiguous(), V[b:b + 1, k:k + 1].contiguous(), table=W)
            assert torch.equal(O[b:b + 1, h], o) and torch.equal(lse[b:b + 1, h], l)
    atf.binding.check_status()


def _cut_case(B, Hq, Hkv, N, Nq, d, far, split):
    import paper_2608_02947_b200 as atf
    g = torch.Generator(device="cuda").manual_seed(N + far)
    kind = torch.float32 if split else torch.bfloat16
    Q, K, V = [torch.randn((B, h, n, d), generator=g, device="cuda") for h, n in ((Hq, Nq), (Hkv, N), (Hkv, N))]
    W, _ = atf.atf_window_table(5e5, d, 2.0, N)
    if far == 3:  # no pair reaches further: every tile has the same few steps
        W = W.clamp(max=7000)
    elif far == 4:  # every pair reaches every key
        W = None
    elif far:     # logits that the reference of the diagonal tile cannot hold, in near (1) or far (2) keys
        K[:, :, slice(N - 2000, N - 1500) if far == 1 else slice(0, 500)] *= 30
        Q *= 4
    return Q.to(kind), K.to(kind), V.to(torch.bfloat16), W


# Bit for bit what one block gives (a call that counts terms never cuts): just above one wave of blocks, an odd number of waves,
# ragged rows, windows that end (equal short tiles), the safe second pass seen in front of the cut and behind it; every form of the
# kernel goes on from a state.  The third case lies just below the idle share from which tiles are cut.
@pytest.mark.parametrize("B,Hq,Hkv,N,Nq,d,mode,far,split", [
    (1, 24, 8, 9000, 850, 128, 0, 0, False), (2, 14, 2, 12345, 700, 64, 0, 0, False), (1, 24, 8, 30000, 1111, 128, 1, 0, False),
    (1, 40, 8, 9000, 512, 128, 0, 1, False), (1, 40, 8, 9000, 512, 64, 0, 2, False), (1, 40, 8, 9000, 512, 128, 1, 2, False),
    (3, 14, 2, 20000, 500, 64, 1, 3, False), (1, 24, 8, 9000, 850, 128, 0, 0, True), (1, 40, 8, 9000, 512, 128, 0, 2, True),
    (1, 24, 8, 9000, 850, 128, 1, 0, False), (1, 24, 8, 9000, 850, 128, 0, 4, False), (2, 14, 2, 12345, 700, 64, 0, 4, False),
    (1, 40, 8, 9000, 512, 128, 1, 1, False), (1, 24, 8, 9000, 850, 128, 1, 0, True), (2, 14, 2, 12345, 700, 64, 0, 0, True),
    (2, 14, 2, 12345, 700, 64, 1, 1, True)])
def test_cut_tiles(B, Hq, Hkv, N, Nq, d, mode, far, split):
    import paper_2608_02947_b200 as atf
    Q, K, V, W = _cut_case(B, Hq, Hkv, N, Nq, d, far, split)
    call = atf.atf_prefill_split if split else atf.atf_prefill
    # room for the state of the cut tiles beside what the call asks for
    ws = atf.ensure_workspace(3 * atf.atf_workspace_bytes(atf.binding.ATF_OP_PREFILL_SPLIT, B, Hq, Hkv, N, d), "cuda:0")
    flags = _cut_flags(ws, B, Hq, Hkv, N, Nq, d, split)
    whole = call(Q, K, V, table=W, mode=mode, kept_terms=torch.zeros(B * Hq, dtype=torch.int64, device="cuda"))
    for _ in range(3):
        flags.fill_(-1)
        O, lse = call(Q, K, V, table=W, mode=mode)
        assert torch.equal(O, whole[0]) and torch.equal(lse, whole[1])
        seen = flags.tolist()
        if N == 30000:
            assert set(seen) == {-1}
        else:  # 3: went on from the state; 7: overflow in the first part, all of it again; 0: no first part
            assert set(seen) <= ({0, 3, 7} if far in (1, 2) else {0, 3})
            assert seen.count(3) > (10 if far == 1 else 100) and (far != 1 or seen.count(7) > 50)
    atf.binding.check_status()


@pytest.mark.parametrize("d,mode,far", [(128, 0, 0), (128, 1, 1), (64, 0, 1), (64, 1, 0)])
def test_cut_output_over_its_queries(d, mode, far):
    import paper_2608_02947_b200 as atf
    B, Hq, Hkv, N, Nq = 1, 40, 8, 9000, 512
    Q, K, V, W = _cut_case(B, Hq, Hkv, N, Nq, d, far, False)
    ws = atf.ensure_workspace(3 * atf.atf_workspace_bytes(atf.binding.ATF_OP_PREFILL, B, Hq, Hkv, N, d), "cuda:0")
    flags = _cut_flags(ws, B, Hq, Hkv, N, Nq, d)
    O, lse = atf.atf_prefill(Q, K, V, table=W, mode=mode)
    flags.fill_(-1)
    got, lse2 = atf.atf_prefill(Q, K, V, table=W, mode=mode, O=Q)
    assert got.data_ptr() == Q.data_ptr() and torch.equal(got, O) and torch.equal(lse2, lse)
    assert 3 in flags.tolist()


# CUDA promises no order in which blocks start: the second block of a cut tile waits only for a first one that runs.  Every first
# block with a part has said so (1) and that its state is there (2).
@pytest.mark.parametrize("B,Hq,Hkv,N,Nq,d,mode,split", [(1, 24, 8, 9000, 850, 128, 0, False), (2, 14, 2, 12345, 700, 64, 1, False),
                                                        (1, 24, 8, 9000, 850, 128, 0, True)])
def test_first_blocks_of_cut_tiles_say_that_they_run(B, Hq, Hkv, N, Nq, d, mode, split):
    import paper_2608_02947_b200 as atf
    kind = torch.float32 if split else torch.bfloat16
    Q, K, V = [torch.randn((B, h, n, d), device="cuda").to(t) for h, n, t in ((Hq, Nq, kind), (Hkv, N, kind), (Hkv, N, torch.bfloat16))]
    W, _ = atf.atf_window_table(5e5, d, 2.0, N)
    ws = atf.ensure_workspace(3 * atf.atf_workspace_bytes(atf.binding.ATF_OP_PREFILL_SPLIT, B, Hq, Hkv, N, d), "cuda:0")
    flags = _cut_flags(ws, B, Hq, Hkv, N, Nq, d, split)
    for _ in range(2):  # the second call finds what the first one left
        flags.fill_(-1)
        (atf.atf_prefill_split if split else atf.atf_prefill)(Q, K, V, table=W, mode=mode)
        torch.cuda.synchronize()
        got = flags.tolist()
        steps = [min((N - 1) // 128 - j // (B * Hq) + 1, (int(W.max()) + 127) // 128 + 1) for j in range(SMS)]
        assert got == [3 if n * (2 * j + 1) // (2 * SMS) else 0 for j, n in enumerate(steps)]
    atf.binding.check_status()
