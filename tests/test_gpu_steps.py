"""Decoding passes as kernel chains against the persistent pass kernel (which max_ctas selects), bit for
bit: draft, verify and plain-decoding logits, accepted lengths and cached K/V, over block sizes, batch
sizes, head layouts, context lengths (one cluster per group; partial results in memory), draft variants
and adapter ranks."""
import dataclasses

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    return torch


def _shape(name):
    from paper_2607_12422_gb300 import synth
    two = dataclasses.replace(synth.QWEN3_0_6B, n_layers=2, vocab=2048)
    return {
        "tiny": synth.TINY,
        "qwen2": two,
        "grp4": dataclasses.replace(two, n_kv_heads=4, hidden=768, intermediate=1280),
        "grp1-d64": dataclasses.replace(synth.TINY, n_q_heads=8, n_kv_heads=8, hidden=512, intermediate=512, vocab=1024),
        # 13 and 16 K slices: clusters beyond the portable size
        "h3328": dataclasses.replace(two, n_layers=1, hidden=3328, vocab=512),
        "h4096": dataclasses.replace(two, n_layers=1, hidden=4096, n_q_heads=32, n_kv_heads=16, intermediate=4096, vocab=512),
        "r8": dataclasses.replace(two, lora_rank=8, lora_alpha=16.0),
    }[name]


CASES = [
    # shape, D, prompt lengths, max_seq, engine options
    ("tiny", 16, (64,), 256, {}),
    ("tiny", 1, (1,), 64, {}),
    ("qwen2", 16, (512,), 640, {}),
    ("qwen2", 32, (200,), 320, {}),
    ("qwen2", 64, (30,), 256, {}),
    ("qwen2", 4, (1100,), 1400, {}),
    ("qwen2", 16, (128, 127, 129), 400, {}),
    ("qwen2", 16, (700, 40, 333, 512, 90, 1, 600, 257), 900, {}),
    ("qwen2", 31, (50, 60, 70, 80, 90, 100, 110, 120), 320, {}),  # 256 rows
    ("qwen2", 16, (300,), 400, dict(draft_layers=1)),
    ("qwen2", 16, (300, 20), 400, dict(draft_skip=1, denoise_steps=2, anchored=False)),
    ("grp4", 16, (333, 40), 500, {}),
    ("grp1-d64", 8, (150, 33), 300, {}),
    ("r8", 16, (140,), 300, {}),
    ("h3328", 16, (140,), 300, {}),
    ("h4096", 16, (40, 200), 300, {}),
]


@pytest.mark.parametrize("shape,D,lens,max_seq,opt", CASES, ids=lambda v: str(v).replace(" ", "")[:40])
def test_kernel_chain_equals_persistent_kernel(torch, shape, D, lens, max_seq, opt):
    from paper_2607_12422_gb300 import pbd, synth
    S = _shape(shape)
    base, ad = synth.with_random_norm_gains(synth.gen_base_weights(S)), synth.gen_adapter(S)
    rng = np.random.default_rng(D + sum(lens))
    prompts = [rng.integers(0, S.vocab, n).astype(np.int32) for n in lens]
    rounds = 3
    drafts = rng.integers(0, S.vocab, (rounds, len(lens), D)).astype(np.int32)
    forced = rng.integers(0, D + 1, (rounds, len(lens))).astype(np.int32)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    got = []
    for ctas in (0, sms):
        eng = pbd.Engine(S, base, ad, block_D=D, max_batch=len(lens), max_seq_len=max_seq, max_ctas=ctas, **opt)
        out = [eng.pbd_prefill(prompts, max_new=rounds * (D + 1) + 4)]
        for r in range(rounds):  # (the third round replays the chains as graphs)
            d_ids, d_lg = eng.pbd_draft_block(want_logits=True)
            v_ids, v_lg = eng.pbd_verify_block(drafts=drafts[r], want_logits=True)
            out += [d_ids, d_lg, v_ids, v_lg, eng.pbd_accept_commit(forced_n=forced[r])]
        for _ in range(3):
            out += list(eng.pbd_decode_step(want_logits=True))
        L = [int(x) for x in eng.pbd_get_state()[0]]
        for b in range(len(lens)):
            for l in range(S.n_layers):
                out += list(eng.pbd_read_kv(l, b, L[b]))
        got.append((L, [t.clone() for t in out]))
        eng.close()
    assert got[0][0] == got[1][0]
    for i, (x, y) in enumerate(zip(got[0][1], got[1][1])):
        assert torch.equal(x, y), i


def test_graphs_follow_the_generation(torch):
    """One engine, generations of other batch and prompt sizes in turn: chains and their graphs are those of the
    current generation, not of the one before."""
    from paper_2607_12422_gb300 import pbd, synth
    S = _shape("qwen2")
    base, ad = synth.gen_base_weights(S), synth.gen_adapter(S)
    rng = np.random.default_rng(2)
    eng = pbd.Engine(S, base, ad, block_D=8, max_batch=3, max_seq_len=900)
    for lens in ((40,), (700, 30, 300), (40,), (300, 30), (820,)):
        prompts = [rng.integers(0, S.vocab, n).astype(np.int32) for n in lens]
        spec, _ = eng.pbd_generate(prompts, 24, mode=0)
        eng.pbd_prefill(prompts, max_new=24)
        toks = [eng.pbd_decode_step()[0].clone() for _ in range(23)]
        assert torch.equal(spec[:, 1:], torch.stack(toks, 1)), lens
    eng.close()


def test_refused_prefill_leaves_no_generation(torch):
    """A prefill that the device refuses (a token id beyond the vocabulary) after a good one of another batch
    size: what needs a generation is refused until a prefill succeeds, which then gives what a new context
    gives.  Arguments refused on the host leave the generation as it was."""
    from paper_2607_12422_gb300 import pbd, synth
    S = _shape("tiny")
    base, ad = synth.gen_base_weights(S), synth.gen_adapter(S)
    rng = np.random.default_rng(5)
    one, three = ([rng.integers(0, S.vocab, n).astype(np.int32) for n in lens] for lens in ((40,), (200, 20, 64)))
    bad = [p.copy() for p in three]
    bad[1][7] = S.vocab
    used, fresh = (pbd.Engine(S, base, ad, block_D=4, max_batch=3, max_seq_len=256) for _ in range(2))
    used.pbd_prefill(one, max_new=16)
    with pytest.raises(pbd.PbdError) as ei:
        used.pbd_prefill(three + one, max_new=16)
    assert ei.value.status == 3
    for _ in range(3):
        used.pbd_draft_block()
        used.pbd_verify_block()
        used.pbd_accept_commit()
    with pytest.raises(pbd.PbdError) as ei:
        used.pbd_prefill(bad, max_new=16)
    assert ei.value.status == 6
    drafts = np.zeros((1, 4), np.int32)
    for call in (used.pbd_draft_block, lambda: used.pbd_verify_block(drafts=drafts), used.pbd_accept_commit,
                 used.pbd_decode_step, used.pbd_get_tokens, lambda: used.pbd_time_pass(1, 1),
                 lambda: used.pbd_bench_rounds(0, 0, 1), lambda: used.pbd_trace_pass(1)):
        with pytest.raises(pbd.PbdError) as ei:
            call()
        assert ei.value.status == 4
    got, want = used.pbd_generate(three, 16)[0], fresh.pbd_generate(three, 16)[0]
    assert torch.equal(got, want)
    used.close()
    fresh.close()


def test_pass_before_the_first_draft(torch):
    """A verify pass that is timed before anything was drafted verifies zeros, not what the workspace held."""
    import ctypes as C
    from paper_2607_12422_gb300 import pbd, synth
    S = _shape("tiny")
    cfg = pbd.make_config(S, 16, 1, 256)
    need = pbd.load().pbd_workspace_bytes(C.byref(cfg))
    torch.full((need + 256,), 0x7F, dtype=torch.uint8, device="cuda")  # (the engine's workspace takes this place)
    eng = pbd.Engine(S, synth.gen_base_weights(S), synth.gen_adapter(S), block_D=16, max_batch=1, max_seq_len=256)
    eng.pbd_prefill([np.arange(50, dtype=np.int32)], max_new=8)
    assert eng.pbd_time_pass(1, 2)[0] > 0
    eng.close()


@pytest.mark.parametrize("P,max_seq,ctas", [(40, 256, 0), (1100, 1400, 0), (40, 256, 4)])
def test_waits_that_run_out_are_reported(torch, P, max_seq, ctas):
    """Every kind of pass that a context runs is made to wait in vain (kernel chain, with the attention merged in a
    cluster or through memory; persistent kernel; prompt kernels): the codes are reported, the committed K/V and
    the state are what they were, and the same context then decodes what a new one decodes."""
    from paper_2607_12422_gb300 import pbd, synth
    S = _shape("tiny")
    base, ad = synth.gen_base_weights(S), synth.gen_adapter(S)
    p = np.random.default_rng(P).integers(0, S.vocab, P).astype(np.int32)
    eng = pbd.Engine(S, base, ad, block_D=16, max_batch=1, max_seq_len=max_seq, max_ctas=ctas)
    want = eng.pbd_generate([p], 40)[0].clone()
    eng.pbd_prefill([p], max_new=40)
    kv, state = [eng.pbd_read_kv(l, 0, P) for l in range(S.n_layers)], eng.pbd_get_state()
    status, code = eng.pbd_check_stalled_pass()
    assert status == 6 and code in (1, 2, 3, 6)  # PBD_ERR_DEVICE, DEV_TIMEOUT_*
    for l in range(S.n_layers):
        assert all(torch.equal(x, y) for x, y in zip(kv[l], eng.pbd_read_kv(l, 0, P)))
    assert all(np.array_equal(x, y) for x, y in zip(state, eng.pbd_get_state()))
    got = [state[1][0]] + [int(eng.pbd_decode_step()[0][0]) for _ in range(39)]
    assert got == [int(t) for t in want[0].cpu()]
    assert torch.equal(eng.pbd_generate([p], 40)[0], want)
    eng.close()


@pytest.mark.parametrize("shape,P", [("qwen2", 33), ("qwen2", 127), ("qwen2", 128), ("qwen2", 129), ("tiny", 100)])
def test_prompt_of_few_tokens_equals_the_many_row_kernels(torch, shape, P):
    """A lone prompt up to the chain's limit is one decoding pass; in a batch it goes through the many-row
    kernels: the same first token and K/V, bit for bit."""
    from paper_2607_12422_gb300 import pbd, synth
    S = _shape(shape)
    base, ad = synth.with_random_norm_gains(synth.gen_base_weights(S)), synth.gen_adapter(S)
    eng = pbd.Engine(S, base, ad, block_D=8, max_batch=2, max_seq_len=256)
    p = np.random.default_rng(P).integers(0, S.vocab, P).astype(np.int32)
    first = int(eng.pbd_prefill([p], max_new=4)[0])
    kv = [eng.pbd_read_kv(l, 0, P) for l in range(S.n_layers)]
    both = eng.pbd_prefill([p, p], max_new=4)
    assert first == int(both[0]) == int(both[1])
    for l in range(S.n_layers):
        for b in (0, 1):
            k, v = eng.pbd_read_kv(l, b, P)
            assert torch.equal(kv[l][0], k) and torch.equal(kv[l][1], v), (l, b)
    eng.close()
