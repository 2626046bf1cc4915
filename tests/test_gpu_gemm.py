"""The standalone linear and lm_head at the edges of their kernels' tiles and dispatch: one row to
several token tiles, K of one 64-wide atom to many slices, every kind of adapter rank, operands that
no tensor map can describe, ties and infinities in the read-out.  References in float64."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2607_12422_gb300 import pbd
    pbd.load()
    return torch


def _rand(torch, g, shape, std):
    return (torch.randn(shape, generator=g, device="cuda") * std).to(torch.bfloat16)


def _linear_ref(x, W, A, B, scale):
    """(y in float64, bound): one bf16 rounding of y, fp32 sums of K products, and a rounding of each
    u to bf16 that may fall the other way."""
    y = x.double() @ W.double().T
    tol = 2e-6 * (x.double().abs() @ W.double().abs().T)
    if A is not None:
        u = (x.double() @ A.double().T).bfloat16().double()
        y = y + scale * (u @ B.double().T)
        tol = tol + abs(scale) * 2.0 ** -8 * (u.abs() @ B.double().abs().T)
    return y, tol + 2.0 ** -8 * y.abs() + 1e-7


LINEARS = [(1, 64, 128, 0), (2, 64, 128, 1), (31, 320, 256, 3), (32, 256, 128, 32), (33, 3072, 1024, 16),
           (64, 256, 128, 32), (65, 64, 128, 0), (65, 192, 256, 5), (129, 1024, 384, 8), (257, 512, 6272, 3),
           (300, 2048, 1024, 24), (1000, 320, 128, 16), (4096, 64, 128, 16), (3, 4096, 128, 16), (3, 4352, 128, 16),
           # more slices than a cluster has CTAs, one slice of many atoms, blocks of 64 rows
           (64, 8192, 256, 32), (33, 12544, 128, 16), (1, 4160, 128, 1), (5, 65536, 128, 8), (65, 8192, 128, 16),
           (200, 16384, 256, 3), (129, 3072, 128, 16), (128, 4352, 256, 0), (1000, 6144, 128, 32), (64, 4096, 6144, 16),
           (17, 3328, 8192, 16)]


@pytest.mark.parametrize("M,K,N,r", LINEARS)
def test_linear_tile_edges(torch, M, K, N, r):
    from paper_2607_12422_gb300 import pbd
    g = torch.Generator(device="cuda").manual_seed(M + K + N + r)
    x, W = _rand(torch, g, (M, K), 1.0), _rand(torch, g, (N, K), 0.02)
    A, B = (_rand(torch, g, (r, K), 0.02), _rand(torch, g, (N, r), 0.02)) if r else (None, None)
    ref, tol = _linear_ref(x, W, A, B, 2.0)
    y = pbd.pbd_op_linear(x, W, A, B, 2.0)
    assert ((y.double() - ref).abs() <= tol).all()
    slices = K // 256 if K % 256 == 0 else 1
    if 2048 + (N // 128 + (r > 0)) * (K // 64) * 16384 + 4 * slices * M * (N + r) <= 16 << 20:  # the static scratch holds it
        assert torch.equal(pbd.pbd_op_linear_static(x, W, A, B, 2.0), y)


@pytest.mark.parametrize("M,N", [(17, 256), (200, 256), (300, 6144)])
def test_linear_unaligned_adapter_and_output(torch, M, N):
    """B and y start on odd element offsets: B has no tensor map, y takes no 32-bit stores."""
    from paper_2607_12422_gb300 import pbd
    g = torch.Generator(device="cuda").manual_seed(M)
    K, r = 256, 16
    x, W, A = _rand(torch, g, (M, K), 1.0), _rand(torch, g, (N, K), 0.02), _rand(torch, g, (r, K), 0.02)
    B = _rand(torch, g, (N * r + 1,), 0.02)[1:].view(N, r)
    y = torch.zeros(M * N + 1, dtype=torch.bfloat16, device="cuda")
    got = pbd.pbd_op_linear_static(x, W, A, B, 2.0, y=y[1:].view(M, N))
    ref, tol = _linear_ref(x, W, A, B, 2.0)
    assert ((got.double() - ref).abs() <= tol).all() and float(y[0]) == 0.0


@pytest.mark.parametrize("M,K,N,r", [(1, 4352, 128, 1), (1, 4352, 128, 7), (2, 4608, 128, 3), (64, 4352, 256, 5),
                                     (65, 64, 128, 1), (70, 320, 128, 31), (17, 1024, 128, 3), (4096, 64, 128, 9)])
def test_linear_stays_inside_its_workspace(torch, M, K, N, r):
    """A workspace of exactly the reported size, bytes of a known value right behind it: they keep it.
    Ranks whose B rows are padded to 32 columns, with few and with many slices of K."""
    from paper_2607_12422_gb300 import pbd
    lib = pbd.load()
    g = torch.Generator(device="cuda").manual_seed(M + K + r)
    x, W = _rand(torch, g, (M, K), 1.0), _rand(torch, g, (N, K), 0.02)
    A, B = _rand(torch, g, (r, K), 0.02), _rand(torch, g, (N, r), 0.02)
    need, guard = lib.pbd_op_linear_workspace_bytes(M, K, N, r), 1 << 16
    buf = torch.full((need + guard + 1024,), 0xA5, dtype=torch.uint8, device="cuda")
    off = -buf.data_ptr() % 1024
    y = torch.empty(M, N, dtype=torch.bfloat16, device="cuda")
    st = torch.cuda.current_stream().cuda_stream
    args = [t.data_ptr() for t in (x, W, A, B, y)]
    assert lib.pbd_op_linear(M, K, N, r, 2.0, *args, buf.data_ptr() + off, need, st) == 0
    assert lib.pbd_op_status(buf.data_ptr() + off, st, None) == 0
    assert (buf[off + need:] == 0xA5).all()
    ref, tol = _linear_ref(x, W, A, B, 2.0)
    assert ((y.double() - ref).abs() <= tol).all()


@pytest.mark.parametrize("M,K,N,r", [(17, 256, 256, 1), (65, 256, 256, 1), (70, 320, 6144, 3), (200, 256, 4096, 16),
                                     (65, 256, 256, 32), (3, 4352, 256, 5), (4096, 1024, 256, 3), (100, 2048, 4096, 5)])
def test_linear_infinite_operand(torch, M, K, N, r):
    """An infinite x among positive operands: its row is infinite, whatever the rank, and no other row is."""
    from paper_2607_12422_gb300 import pbd
    g = torch.Generator(device="cuda").manual_seed(M + N + r)
    x, W = _rand(torch, g, (M, K), 1.0).abs(), _rand(torch, g, (N, K), 0.02).abs() + 0.01
    A, B = _rand(torch, g, (r, K), 0.02).abs() + 0.01, _rand(torch, g, (N, r), 0.02).abs() + 0.01
    ref, tol = _linear_ref(x, W, A, B, 2.0)
    x[M // 2, 5] = float("inf")
    y = pbd.pbd_op_linear(x, W, A, B, 2.0)
    assert torch.isposinf(y[M // 2]).all()
    rest = torch.arange(M, device="cuda") != M // 2
    assert ((y.double() - ref).abs() <= tol)[rest].all()


OVER = [(17, 256, 256, 0), (64, 4096, 4096, 0), (64, 2048, 2048, 16), (4096, 2048, 2048, 0), (300, 512, 512, 5),
        (1, 64, 128, 1), (65, 64, 128, 1)]


@pytest.mark.parametrize("M,K,N,r,over", [(*c, o) for c in OVER for o in ("xWAB" if c[3] else "xW")])
def test_linear_output_over_an_operand(torch, M, K, N, r, over):
    """y may lie over an operand: the result is that of a y of its own, and nothing behind the workspace's or
    y's end is written."""
    from paper_2607_12422_gb300 import pbd
    lib = pbd.load()
    g = torch.Generator(device="cuda").manual_seed(M + K + r)
    ops = dict(x=_rand(torch, g, (M, K), 1.0), W=_rand(torch, g, (N, K), 0.02), A=_rand(torch, g, (max(r, 1), K), 0.02),
               B=_rand(torch, g, (N, max(r, 1)), 0.02))
    want = pbd.pbd_op_linear(ops["x"], ops["W"], *((ops["A"], ops["B"]) if r else ()), scale=2.0)
    need, st = lib.pbd_op_linear_workspace_bytes(M, K, N, r), torch.cuda.current_stream().cuda_stream
    ws = torch.full((need + 2048,), 0xA5, dtype=torch.uint8, device="cuda")
    off = -ws.data_ptr() % 1024
    size = max(M * N, ops[over].numel())
    room = torch.full((size + 64,), 7.0, dtype=torch.bfloat16, device="cuda")  # the operand, and y over its start
    room[:ops[over].numel()] = ops[over].flatten()
    ptr = {k: (room if k == over else v).data_ptr() for k, v in ops.items()}
    assert lib.pbd_op_linear(M, K, N, r, 2.0, ptr["x"], ptr["W"], ptr["A"] if r else None, ptr["B"] if r else None,
                             room.data_ptr(), ws.data_ptr() + off, need, st) == 0
    assert lib.pbd_op_status(ws.data_ptr() + off, st, None) == 0
    assert torch.equal(room[:M * N].view(M, N), want)
    assert (room[size:] == 7.0).all() and (ws[off + need:] == 0xA5).all()


def test_linear_rows_do_not_depend_on_the_row_count(torch):
    from paper_2607_12422_gb300 import pbd
    g = torch.Generator(device="cuda").manual_seed(9)
    for K in (1024, 3072, 320, 8192):  # (one kernel or the other, by M and K)
        x, W = _rand(torch, g, (700, K), 1.0), _rand(torch, g, (512, K), 0.02)
        y = pbd.pbd_op_linear(x, W)
        for M in (1, 17, 64, 65, 300):
            assert torch.equal(pbd.pbd_op_linear(x[:M].contiguous(), W), y[:M]), (K, M)


@pytest.mark.parametrize("M,H,V", [(1, 64, 128), (32, 1024, 128 * 155), (33, 256, 128 * 153), (64, 1024, 2048),
                                   (65, 1024, 128 * 160), (144, 512, 4096), (256, 256, 128 * 3), (7, 2048, 1024)])
def test_lm_head_edges(torch, M, H, V):
    from paper_2607_12422_gb300 import pbd
    g = torch.Generator(device="cuda").manual_seed(M + H + V)
    x, E = _rand(torch, g, (M, H), 1.0), _rand(torch, g, (V, H), 0.02)
    # every row of E again at the far end: each maximum occurs twice, the lower id wins
    E[V // 2:] = E[:V - V // 2]
    x[0, 3] = float("inf")  # infinite logits of both signs in one row
    ids, lg = pbd.pbd_op_lm_head_argmax(x, E, want_logits=True)
    ref = x[1:].double() @ E.double().T
    assert ((lg[1:].double() - ref).abs() <= 2e-6 * (x[1:].double().abs() @ E.double().abs().T)).all()
    want = np.argmax(lg.cpu().numpy(), axis=1)  # lowest index among equal maxima
    assert not torch.isnan(lg).any() and np.array_equal(ids.cpu().numpy(), want)
    assert (want < max(V // 2, 1)).all()
    plain, none = pbd.pbd_op_lm_head_argmax(x, E)
    assert none is None and torch.equal(plain, ids)


@pytest.mark.parametrize("M,H,V", [(17, 256, 128 * 400), (136, 512, 128 * 320)])
def test_lm_head_logits_over_the_table(torch, M, H, V):
    from paper_2607_12422_gb300 import pbd
    lib = pbd.load()
    g = torch.Generator(device="cuda").manual_seed(M)
    x, E = _rand(torch, g, (M, H), 1.0), _rand(torch, g, (V, H), 0.02)
    ids, lg = pbd.pbd_op_lm_head_argmax(x, E, want_logits=True)
    room = torch.empty(max(V * H, 2 * M * V), dtype=torch.bfloat16, device="cuda")
    room[:V * H] = E.flatten()
    need, st = lib.pbd_op_lm_head_workspace_bytes(M, H, V), torch.cuda.current_stream().cuda_stream
    ws = torch.empty(need + 1024, dtype=torch.uint8, device="cuda")
    off = -ws.data_ptr() % 1024
    got = torch.empty(M, dtype=torch.int32, device="cuda")
    assert lib.pbd_op_lm_head_argmax(M, H, V, x.data_ptr(), room.data_ptr(), got.data_ptr(), room.data_ptr(),
                                     ws.data_ptr() + off, need, st) == 0
    assert lib.pbd_op_status(ws.data_ptr() + off, st, None) == 0
    assert torch.equal(room[:2 * M * V].view(torch.float32).view(M, V), lg) and torch.equal(got, ids)


@pytest.mark.parametrize("shape,max_seq,start,rounds,ctas", [("tiny", 256, 1, 9, 0), ("qwen2", 420, 40, 21, 0),
                                                            ("qwen2", 4096, 301, 30, 0), ("grp4", 420, 17, 10, 0),
                                                            ("qwen2", 420, 130, 14, 20), ("tiny", 600, 130, 25, 4)])
def test_prefill_equals_decoded_rows_bitwise(torch, shape, max_seq, start, rounds, ctas):
    """The many-row kernels of the prefill against the pass kernel: K/V of every layer, written by
    verify rounds that commit 17 random tokens each, equal a prefill of the same tokens, and so do the
    logits that follow.  Both partitions of an attention split (two halves; whole, at max_seq 4096),
    heads of 64 and 128, one to four query heads per KV head, last tiles of 1 to 128 rows, few CTAs."""
    import dataclasses
    from paper_2607_12422_gb300 import pbd, synth
    S = synth.TINY if shape == "tiny" else dataclasses.replace(synth.QWEN3_0_6B, n_layers=2, vocab=4096)
    if shape == "grp4":
        S = dataclasses.replace(S, n_kv_heads=4, hidden=1280, intermediate=1792)
    D = 16
    base, ad = synth.with_random_norm_gains(synth.gen_base_weights(S)), synth.gen_adapter(S)
    eng = pbd.Engine(S, base, ad, block_D=D, max_batch=1, max_seq_len=max_seq, max_ctas=ctas)
    rng = np.random.default_rng(start)
    prompt = rng.integers(0, S.vocab, start).astype(np.int32)
    eng.pbd_prefill([prompt], max_new=(D + 1) * rounds + 2)
    for _ in range(rounds):
        eng.pbd_verify_block(drafts=rng.integers(0, S.vocab, (1, D)).astype(np.int32))
        eng.pbd_accept_commit(forced_n=[D])
    L, pend, n_out = (int(z[0]) for z in eng.pbd_get_state())
    toks = eng.pbd_get_tokens()[0].cpu().numpy()[:n_out]
    kv = [eng.pbd_read_kv(l, 0, L) for l in range(S.n_layers)]
    _, lg = eng.pbd_decode_step(want_logits=True)
    seq = np.concatenate([prompt, toks[:-1]]).astype(np.int32)
    assert len(seq) == L
    first = eng.pbd_prefill([seq], max_new=2)
    assert int(first[0]) == pend
    for l in range(S.n_layers):
        k, v = eng.pbd_read_kv(l, 0, L)
        assert torch.equal(kv[l][0], k) and torch.equal(kv[l][1], v), l
    _, lg2 = eng.pbd_decode_step(want_logits=True)
    assert torch.equal(lg, lg2)
    eng.close()


def test_prefill_batch_and_passes_match_single_prompts(torch):
    """Ragged prompts share passes and a long one spans two (4096 rows each): first tokens and last-layer
    K/V equal those of each prompt alone."""
    import dataclasses
    from paper_2607_12422_gb300 import pbd, synth
    S = dataclasses.replace(synth.TINY, vocab=1024)
    base, ad = synth.gen_base_weights(S), synth.gen_adapter(S)
    rng = np.random.default_rng(4)
    prompts = [rng.integers(0, S.vocab, n).astype(np.int32) for n in (1, 65, 4100, 300, 17)]
    eng = pbd.Engine(S, base, ad, block_D=4, max_batch=5, max_seq_len=4200)
    first = eng.pbd_prefill(prompts, max_new=4).cpu().numpy()
    kv = [eng.pbd_read_kv(S.n_layers - 1, b, len(p)) for b, p in enumerate(prompts)]
    for b, p in enumerate(prompts):
        assert int(eng.pbd_prefill([p], max_new=4)[0]) == first[b], b
        k, v = eng.pbd_read_kv(S.n_layers - 1, 0, len(p))
        assert torch.equal(k, kv[b][0]) and torch.equal(v, kv[b][1]), b
    eng.close()


@pytest.mark.parametrize("shape", ["tiny", "qwen2"])
def test_prompt_over_pages_that_hold_nan(torch, shape):
    """Pages keep what an earlier generation left there.  After a prompt whose every K and V is NaN (an
    infinite embedding row), shorter prompts give the first token and K/V of a context without that past:
    keys beyond the prompt's end take no part, whatever their page holds."""
    import dataclasses
    from paper_2607_12422_gb300 import pbd, synth
    S = synth.TINY if shape == "tiny" else dataclasses.replace(synth.QWEN3_0_6B, n_layers=2, vocab=4096)
    base, ad = synth.gen_base_weights(S), synth.gen_adapter(S)
    base["embed"] = base["embed"].copy()
    base["embed"][7] = 0x7F80
    rng = np.random.default_rng(11)
    used, fresh = (pbd.Engine(S, base, ad, block_D=4, max_batch=1, max_seq_len=300) for _ in range(2))
    for P in (129, 143, 190):
        used.pbd_prefill([np.full(250, 7, np.int32)], max_new=4)
        assert torch.isnan(used.pbd_read_kv(1, 0, 250)[1].float()).all()
        p = rng.integers(8, S.vocab, P).astype(np.int32)
        assert int(used.pbd_prefill([p], max_new=4)[0]) == int(fresh.pbd_prefill([p], max_new=4)[0])
        for l in range(S.n_layers):
            for x, y in zip(used.pbd_read_kv(l, 0, P), fresh.pbd_read_kv(l, 0, P)):
                assert torch.equal(x, y) and not torch.isnan(x.float()).any(), (P, l)
    used.close()
    fresh.close()
