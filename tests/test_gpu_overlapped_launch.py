"""Kernels launched to overlap the one before them in the stream: chains in which every call reads what the call before wrote give
what they give with a synchronisation between any two."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,L", [(128, 3000), (64, 200)])
def test_chain_of_dependent_calls(d, L):
    import paper_2608_02947_b200 as atf
    B, Hq, Hkv = 2, 6, 2
    g = torch.Generator(device="cuda").manual_seed(L)
    W, theta = atf.atf_window_table(5e5, d, 2.0, L)
    table = atf.WindowTable(W)
    K, V = [torch.randn((B, Hkv, L, d), generator=g, device="cuda").to(torch.bfloat16) for _ in range(2)]
    q0 = torch.randn((B, Hq, d), generator=g, device="cuda").to(torch.bfloat16)
    Kg = atf.new_kcache_groups(B, Hkv, L, d, "cuda")
    q, k, Qn = torch.empty_like(q0), torch.empty_like(K), torch.empty((B, Hq, L, d), dtype=torch.bfloat16, device="cuda")
    O = torch.empty_like(Qn)

    def chain(sync):
        out = []
        wait = torch.cuda.synchronize if sync else (lambda: None)
        q.copy_(q0)
        for i in range(6):
            k.copy_(K)
            for X, pos in ((q[:, :, None], L - 1 + i), (k, i)):
                wait()
                atf.atf_rope(X, theta, pos0=pos)  # in place, read by the next call
            wait()
            a = atf.atf_decode(q, k, V, table=table, O=torch.empty_like(q))
            wait()
            atf.atf_decode(a, k, V, table=table, O=q)  # the query of the next calls
            wait()
            Qn.copy_(q[:, :, None].expand_as(Qn))
            atf.atf_rope(Qn, theta)
            wait()
            _, lse = atf.atf_prefill(Qn, k, V, table=table, O=O, kcache_groups=Kg)
            wait()
            b = atf.atf_decode(O[:, :, -1].contiguous(), Kg, V, table=table)
            wait()
            atf.atf_decode(b, Kg, V, table=table, O=q)
            out += [a, b, lse, q.clone()]
        torch.cuda.synchronize()
        return out

    want = chain(True)
    for _ in range(10):
        for x, y in zip(want, chain(False)):
            assert torch.equal(x, y)


def test_captured_chain():
    import paper_2608_02947_b200 as atf
    B, Hq, Hkv, d, L = 1, 6, 2, 128, 700
    g = torch.Generator(device="cuda").manual_seed(L)
    W, theta = atf.atf_window_table(5e5, d, 2.0, L)
    table = atf.WindowTable(W)
    K, V = [torch.randn((B, Hkv, L, d), generator=g, device="cuda").to(torch.bfloat16) for _ in range(2)]
    q0 = torch.randn((B, Hq, d), generator=g, device="cuda").to(torch.bfloat16)
    q = q0.clone()

    def steps(wait):
        got = []
        for i in range(4):
            atf.atf_rope(q[:, :, None], theta, pos0=L + i)
            wait()
            got.append(atf.atf_decode(q, K, V, table=table))
            wait()
            atf.atf_decode(got[-1], K, V, table=table, O=q)
            wait()
        return got

    want = steps(torch.cuda.synchronize)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        got = steps(lambda: None)
    for _ in range(3):
        q.copy_(q0)
        graph.replay()
        torch.cuda.synchronize()
        for a, b in zip(want, got):
            assert torch.equal(a, b)


def _queued(steps, rounds):
    """steps(i) for every round: with a synchronisation behind each call, queued behind a kernel that keeps the GPU busy (the
    host is ahead, so the kernels follow one another as closely as they can), and captured in a graph."""
    want = [steps(i, torch.cuda.synchronize) for i in range(rounds)]
    torch.cuda.synchronize()
    for _ in range(5):
        torch.cuda._sleep(20_000_000)
        got = [steps(i, lambda: None) for i in range(rounds)]
        torch.cuda.synchronize()
        for a, b in zip(want, got):
            assert all(torch.equal(x, y) for x, y in zip(a, b))
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        got = [steps(i, lambda: None) for i in range(rounds)]
    for _ in range(3):
        graph.replay()
        torch.cuda.synchronize()
        for a, b in zip(want, got):
            assert all(torch.equal(x, y) for x, y in zip(a, b))


# Q and K rotated right before the call that reads them, other values in the same buffers each time: a read in front of the wait,
# or one that the read-only path kept from the round before, would give other bits
@pytest.mark.parametrize("d,Hkv,N,Nq,mode", [(128, 8, 3000, 3000, 0), (128, 8, 3000, 400, 1), (64, 2, 12000, 12000, 1), (64, 3, 700, 700, 0)])
def test_rotation_then_prefill(d, Hkv, N, Nq, mode):
    import paper_2608_02947_b200 as atf
    g = torch.Generator(device="cuda").manual_seed(N + Nq)
    W, theta = atf.atf_window_table(5e5, d, 2.0, N)
    table = atf.WindowTable(W)
    Qs, Ks, Vs = [[torch.randn((1, h, n, d), generator=g, device="cuda").to(torch.bfloat16) for _ in range(3)]
                  for h, n in ((2 * Hkv, Nq), (Hkv, N), (Hkv, N))]
    Q, K, V = Qs[0].clone(), Ks[0].clone(), Vs[0].clone()
    cache = atf.new_kcache_groups(1, Hkv, N, d, "cuda")

    def steps(i, wait):
        for x, src in ((Q, Qs), (K, Ks), (V, Vs)):
            x.copy_(src[i])
        wait()
        atf.atf_rope(Q, theta, pos0=N - Nq)
        wait()
        atf.atf_rope(K, theta)
        wait()
        O, lse = atf.atf_prefill(Q, K, V, table=table, mode=mode, kcache_groups=cache)
        wait()
        return O, lse, cache.clone()

    _queued(steps, 3)


@pytest.mark.parametrize("d,Hkv,N,Nq,mode", [(128, 4, 3000, 3000, 0), (64, 2, 9000, 500, 1)])
def test_rotation_then_split_prefill(d, Hkv, N, Nq, mode):
    import paper_2608_02947_b200 as atf
    g = torch.Generator(device="cuda").manual_seed(N + Nq)
    W, theta = atf.atf_window_table(5e5, d, 2.0, N)
    table = atf.WindowTable(W)
    Qs, Ks = [[torch.randn((1, h, n, d), generator=g, device="cuda") for _ in range(3)] for h, n in ((2 * Hkv, Nq), (Hkv, N))]
    Vs = [torch.randn((1, Hkv, N, d), generator=g, device="cuda").to(torch.bfloat16) for _ in range(3)]
    Q, K, V = Qs[0].clone(), Ks[0].clone(), Vs[0].clone()

    def steps(i, wait):
        for x, src in ((Q, Qs), (K, Ks), (V, Vs)):
            x.copy_(src[i])
        for x, pos in ((K, 0), (Q, N - Nq)) if i == 1 else ((Q, N - Nq), (K, 0)):
            wait()
            atf.atf_rope_f32(x, theta, pos0=pos)
        wait()
        out = atf.atf_prefill_split(Q, K, V, table=table, mode=mode)
        wait()
        return out

    _queued(steps, 3)


@pytest.mark.parametrize("d,G,L", [(128, 3, 5000), (64, 7, 300)])
def test_tables_then_decode(d, G, L):
    """Rotation tables of another base in the same buffer, built right before the decode that reads them."""
    import ctypes as C

    import paper_2608_02947_b200 as atf
    g = torch.Generator(device="cuda").manual_seed(L)
    K, V = [torch.randn((2, 2, L, d), generator=g, device="cuda").to(torch.bfloat16) for _ in range(2)]
    q = torch.randn((2, 2 * G, d), generator=g, device="cuda").to(torch.bfloat16)
    cache = atf.atf_kcache_pack(K)
    W, _ = atf.atf_window_table(5e5, d, 2.0, L)
    table = atf.WindowTable(W)
    thetas = [atf.atf_window_table(base, d, 2.0, L)[1] for base in (1e4, 5e5, 1e7)]
    tables = atf.atf_rope_tables(thetas[0], d, L)

    def steps(i, wait):
        arr = (C.c_double * (d // 2))(*thetas[i].tolist())
        atf.binding._check(atf.lib().atf_rope_tables(arr, d, 7 * i, L, C.c_void_p(tables.buf.data_ptr()), tables.buf.numel(),
                                                     C.c_void_p(torch.cuda.current_stream().cuda_stream)))
        wait()
        x = q.clone()
        atf.atf_rope(x[:, :, None], thetas[i], pos0=7 * i + L - 1)
        wait()
        out = atf.atf_decode(x, cache, V, table=table, return_lse=True, rope_tables=tables)
        wait()
        atf.binding._check(atf.lib().atf_rope_tables(arr, d, 7 * i + 1, L, C.c_void_p(tables.buf.data_ptr()), tables.buf.numel(),
                                                     C.c_void_p(torch.cuda.current_stream().cuda_stream)))
        wait()
        return out + atf.atf_decode(x, cache, V, table=table, return_lse=True, rope_tables=tables)

    _queued(steps, 3)


@pytest.mark.parametrize("f32", [False, True])
@pytest.mark.parametrize("d,H,N", [(128, 8, 9000), (64, 24, 1), (128, 32, 130)])
def test_rotations_in_a_row(d, H, N, f32):
    """In place, each on what the one before it wrote."""
    import paper_2608_02947_b200 as atf
    g = torch.Generator(device="cuda").manual_seed(N)
    _, theta = atf.atf_window_table(5e5, d, 2.0, N)
    src = torch.randn((3, H, N, d), generator=g, device="cuda")
    src = src if f32 else src.to(torch.bfloat16)
    X = src[:1].clone()

    def steps(i, wait):
        X.copy_(src[i:i + 1])
        for pos in (0, 3, 1000, 77):
            wait()
            (atf.atf_rope_f32 if f32 else atf.atf_rope)(X, theta, pos0=pos + i)
        wait()
        return X.clone(),

    _queued(steps, 3)
