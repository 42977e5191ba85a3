"""GPU tests of single kernels and dispatch branches at the sizes where they can go wrong, against the oracle's functions or a
plain fp64 computation."""
import dataclasses

import numpy as np
import pytest

from oracle import bild as obild
from workloads import MODEL_SHAPES, WORKLOADS, gen_model

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch_cuda():
    import torch
    assert torch.cuda.is_available()
    return torch


@pytest.mark.parametrize("vocab,scale,equal", [(30, 5.0, 1), (33, 0.5, 1), (1000, 1.0, 7), (8192, 20.0, 1), (40003, 1.0, 1),
                                               (40003, 4.0, 9000), (270001, 0.5, 1)])
def test_drawn_token_over_vocabulary_sizes(torch_cuda, vocab, scale, equal):
    """The token-drawing kernel (few candidates / radix search; probabilities kept in registers or not; runs of `equal`
    tokens with the same logit) against nucleus_sample on the same logits."""
    from paper_2302_07863_b200 import MODE_SMALL_ONLY
    from paper_2302_07863_b200.binding import FP32, Config, Context, model_cfg, upload_model
    torch = torch_cuda
    s = dataclasses.replace(MODEL_SHAPES["tiny_s"], vocab=vocab)
    w = gen_model(s, 3, "fp32")
    w["lm_head"] = w["lm_head"][np.arange(vocab) // equal * equal]
    dev = upload_model(w, "cuda:0")
    ctx = Context(Config(model_cfg(s, scale), model_cfg(s, scale), FP32, 8, 8, 4, 0, -1, 0), s, dev, s, dev)
    ctx.encode(np.arange(2, 8, dtype=np.int32))
    buf = torch.empty((1, vocab), dtype=torch.float32, device="cuda")
    ctx.small_step(0, 0.4, buf)
    z = buf[0].cpu().numpy().astype(np.float64)
    order = np.argsort(-z, kind="stable")
    c = np.concatenate([[0.0], np.cumsum(np.exp(z[order] - z.max()) / np.exp(z - z.max()).sum())])
    rng = np.random.default_rng(vocab)
    checked = 0
    for top_p in (1e-9, 0.05, 0.5, 0.8, 0.95, 1.0):
        for u in (0.0, float(rng.random()), float(rng.random()), 0.999999):
            uu = np.full(3, u, np.float32)
            want, n, margin = obild.nucleus_sample(z, float(np.float32(top_p)), float(uu[1]))
            got = ctx.generate_sampled(MODE_SMALL_ONLY, 0.0, 10.0, 1, top_p, uu, uu)["tokens"][0]
            if margin > 3e-6:
                assert got == want, (top_p, u, margin)
                checked += 1
            at = int(np.nonzero(order == got)[0][0])   # in any case: the running mass at the drawn token is the one asked for
            assert c[at] <= uu[1] * c[n] + 1e-5 and c[at + 1] >= uu[1] * c[n] - 1e-5, (top_p, u, margin)
    assert checked >= 2
    ctx.close()


@pytest.mark.parametrize("name,n_layers,d,H,dkv,F,ffn", [("a", 3, 64, 3, 16, 136, "gated_gelu"), ("b", 2, 128, 10, 16, 40, "relu"),
                                                         ("c", 2, 256, 2, 64, 64, "gated_gelu"), ("d", 1, 72, 1, 128, 520, "relu")])
def test_small_fp32_passes_match_oracle(torch_cuda, name, n_layers, d, H, dkv, F, ffn):
    """Passes of small fp32 models in one cluster kernel: fewer and more heads than blocks, slices of unequal size and empty ones,
    1 to 16 rows, caches around the count of staged keys."""
    from oracle.t5 import Model
    from paper_2302_07863_b200.binding import FP32, Config, Context, model_cfg, upload_model
    torch = torch_cuda
    s = dataclasses.replace(MODEL_SHAPES["tiny_s"], name=name, n_layers=n_layers, d_model=d, n_heads=H, d_kv=dkv, d_ff=F, ffn=ffn, vocab=97)
    w = gen_model(s, 5, "fp32")
    dev = upload_model(w, "cuda:0")
    ctx = Context(Config(model_cfg(s, 3.0), model_cfg(s, 3.0), FP32, 150, 150, 15, 0, -1, 0), s, dev, s, dev)
    rng = np.random.default_rng(d)
    ids = rng.integers(2, 97, size=140).astype(np.int32)
    ctx.encode(ids)
    m = Model(s, w, 3.0)
    st, st1 = m.start(ids, 150), m.start(ids, 150)
    buf = torch.empty((16, 97), dtype=torch.float32, device="cuda")
    toks = [int(t) for t in rng.integers(2, 97, size=150)]
    at = 0
    for k in (1, 2, 3, 5, 8, 9, 16, 16, 16, 16, 16, 16, 4, 1, 7, 13):   # the cache grows past 128 rows
        ctx.large_verify(toks[at:at + k], 10.0, buf)
        z = m.forward_block(st, toks[at:at + k])
        assert np.max(np.abs(buf[:k].cpu().numpy() - z)) <= 1e-4 * max(1.0, np.max(np.abs(z))), (k, at)
        at += k
    for t in toks[:5]:
        ctx.small_step(t, 0.5, buf)
        z = m.forward_one(st1, t)
        assert np.max(np.abs(buf[0].cpu().numpy() - z)) <= 1e-4 * max(1.0, np.max(np.abs(z)))
    ctx.close()


@pytest.mark.parametrize("E", [1, 17, 63, 64, 65, 127, 128, 129, 200, 257, 300])
@pytest.mark.parametrize("ffn,d,H,F", [("relu", 512, 8, 1024), ("gated_gelu", 512, 6, 1024)])
def test_encoder_lengths_match_oracle(torch_cuda, E, ffn, d, H, F):
    """Cross keys and values of every layer against the oracle around the tile sizes of the encoder's kernels (64 and 128 tokens a GEMM
    tile, K split over a cluster or not, 64 keys and 128 queries an attention tile, one or two blocks per query tile)."""
    from oracle.t5 import Model
    from paper_2302_07863_b200.binding import BF16, Config, Context, model_cfg, upload_model
    s = dataclasses.replace(MODEL_SHAPES["wide_s"], name="len_" + ffn, n_layers=2, d_model=d, n_heads=H, d_kv=64, d_ff=F, ffn=ffn, vocab=300)
    key = (ffn, d)
    if key not in _len_cache:
        w = gen_model(s, 5, "bf16")
        dev = upload_model(w, "cuda:0")
        _len_cache.clear()
        _len_cache[key] = (Context(Config(model_cfg(s, 3.0), model_cfg(s, 3.0), BF16, 320, 20, 8, 0, -1, 0), s, dev, s, dev), Model(s, w, 3.0))
    ctx, m = _len_cache[key]
    ids = np.random.default_rng(E).integers(2, 300, size=E).astype(np.int32)
    ctx.encode(ids)
    st = m.start(ids, 4)
    for which in (0, 1):
        for layer in range(2):
            for what, ref in ((0, st.ck[layer]), (1, st.cv[layer])):
                got = ctx.read_cache(which, what, layer, H, 320, 64)[:, :E]
                want = ref.reshape(E, H, 64).transpose(1, 0, 2)
                assert float(np.max(np.abs(got - want))) <= 2e-3 * max(1.0, float(np.max(np.abs(want)))), (which, layer, what)



@pytest.mark.parametrize("F", [1024, 5120])
@pytest.mark.parametrize("ffn,H", [("relu", 8), ("gated_gelu", 6)])
def test_encoder_columns_of_short_inputs(torch_cuda, ffn, H, F):
    """Inputs of up to 64 ids, whose GEMMs exchange the columns of tokens that exist, in units of 4, 8 and 16, between the two (d_ff = 5120) or four
    blocks of a cluster: cross keys and values against the oracle, each behind an input whose keys and values are not numbers."""
    from oracle.t5 import Model
    from paper_2302_07863_b200.binding import BF16, Config, Context, model_cfg, upload_model
    s = dataclasses.replace(MODEL_SHAPES["wide_s"], name="cols_" + ffn, n_layers=2, d_model=512, n_heads=H, d_kv=64, d_ff=F, ffn=ffn, vocab=300)
    w = gen_model(s, 5, "bf16")
    dev = upload_model(w, "cuda:0")
    dev["emb"][299] = float("nan")
    ctx, m = Context(Config(model_cfg(s, 3.0), model_cfg(s, 3.0), BF16, 64, 20, 8, 0, -1, 0), s, dev, s, dev), Model(s, w, 3.0)
    for E in (64, 48, 33, 32, 31, 16, 9, 8, 5, 4, 2):
        ctx.encode(np.full(64, 299, dtype=np.int32))
        ids = np.random.default_rng(E).integers(2, 299, size=E).astype(np.int32)
        ctx.encode(ids)
        st = m.start(ids, 4)
        for layer in range(2):
            for what, ref in ((0, st.ck[layer]), (1, st.cv[layer])):
                got = ctx.read_cache(1, what, layer, H, 64, 64)[:, :E]
                want = ref.reshape(E, H, 64).transpose(1, 0, 2)
                # (bound: 16 mantissa bits of the activations, as above)
                assert float(np.max(np.abs(got - want))) <= 2e-3 * max(1.0, float(np.max(np.abs(want)))), (E, layer, what)
    ctx.close()


@pytest.mark.parametrize("cap", [128, 160])
@pytest.mark.parametrize("name,F", [("tiny_l", 512), ("odd_l", 328), ("odd_l", 1096)])
def test_fp32_encoder_lengths_match_oracle(torch_cuda, name, F, cap):
    """The encoder's kernels of fp32 weights: 16 token rows a block, K of one chunk in registers, of several and past what is staged at once; keys
    staged (contexts of up to 128 ids, one to 128 threads a key) and read where they lie."""
    from oracle.t5 import Model
    from paper_2302_07863_b200.binding import FP32, Config, Context, model_cfg, upload_model
    s = dataclasses.replace(MODEL_SHAPES[name], n_layers=2, d_ff=F)
    w = gen_model(s, 5, "fp32")
    dev = upload_model(w, "cuda:0")
    ctx, m = Context(Config(model_cfg(s, 3.0), model_cfg(s, 3.0), FP32, cap, 20, 8, 0, -1, 0), s, dev, s, dev), Model(s, w, 3.0)
    for E in (1, 2, 16, 17, 32, 33, 63, 64, 65, 127, 128):
        ids = np.random.default_rng(E).integers(2, s.vocab, size=E).astype(np.int32)
        ctx.encode(ids)
        st = m.start(ids, 4)
        for layer in range(2):
            for what, ref in ((0, st.ck[layer]), (1, st.cv[layer])):
                got = ctx.read_cache(1, what, layer, s.n_heads, cap, s.d_kv)[:, :E]
                want = ref.reshape(E, s.n_heads, s.d_kv).transpose(1, 0, 2)
                # fp32 sums of up to 1096 terms in six matrices one after the other, 1e-7 each
                assert float(np.max(np.abs(got - want))) <= 3e-5 * max(1.0, float(np.max(np.abs(want)))), (E, layer, what)
    ctx.close()


@pytest.mark.parametrize("E", [300, 700])
def test_encoder_attention_with_maxima_far_apart(torch_cuda, E):
    """Relative-position biases of N(0, 20): the maximum of a row's scores grows by far more than 2^8 from one tile of keys to a later one, so that
    the sums kept so far are rescaled (the bias is added in fp32: bounds as above)."""
    from oracle.t5 import Model
    from paper_2302_07863_b200.binding import BF16, Config, Context, model_cfg, upload_model
    s = dataclasses.replace(MODEL_SHAPES["wide_s"], name="far", n_layers=1, d_model=512, n_heads=8, d_kv=64, d_ff=512, ffn="relu", vocab=300)
    w = gen_model(s, 5, "bf16")
    w["enc.rel_bias"] = w["enc.rel_bias"] * np.float32(20)
    dev = upload_model(w, "cuda:0")
    ctx, m = Context(Config(model_cfg(s, 3.0), model_cfg(s, 3.0), BF16, 704, 20, 8, 0, -1, 0), s, dev, s, dev), Model(s, w, 3.0)
    ids = np.random.default_rng(E).integers(2, 300, size=E).astype(np.int32)
    ctx.encode(ids)
    st = m.start(ids, 4)
    for what, ref in ((0, st.ck[0]), (1, st.cv[0])):
        got = ctx.read_cache(1, what, 0, 8, 704, 64)[:, :E]
        want = ref.reshape(E, 8, 64).transpose(1, 0, 2)
        assert float(np.max(np.abs(got - want))) <= 2e-3 * max(1.0, float(np.max(np.abs(want)))), what
    ctx.close()


@pytest.mark.parametrize("spread", [1, 20])
def test_encoder_attention_of_one_block_over_several_tiles(torch_cuda, spread):
    """More (head, query tile) pairs than half of the SMs, so that one block takes all key tiles of a query tile: its two groups exchange their
    results where queries and keys were; biases of N(0, 1) and, so that sums are rescaled on the way, of N(0, 20).  Tiles of 128 keys and their halves."""
    from oracle.t5 import Model
    from paper_2302_07863_b200.binding import BF16, Config, Context, model_cfg, upload_model
    H, cap = 16, 1008
    sms = torch_cuda.cuda.get_device_properties(0).multi_processor_count
    s = dataclasses.replace(MODEL_SHAPES["wide_s"], name="one", n_layers=1, d_model=256, n_heads=H, d_kv=64, d_ff=512, ffn="relu", vocab=300)
    w = gen_model(s, 5, "bf16")
    w["enc.rel_bias"] = w["enc.rel_bias"] * np.float32(spread)
    dev = upload_model(w, "cuda:0")
    ctx, m = Context(Config(model_cfg(s, 3.0), model_cfg(s, 3.0), BF16, cap, 20, 8, 0, -1, 0), s, dev, s, dev), Model(s, w, 3.0)
    for E in (513, 576, 577, 640, 641, 1000):
        assert 2 * H * ((E + 127) // 128) > sms
        ids = np.random.default_rng(E).integers(2, 300, size=E).astype(np.int32)
        ctx.encode(ids)
        st = m.start(ids, 4)
        for what, ref in ((0, st.ck[0]), (1, st.cv[0])):
            got = ctx.read_cache(1, what, 0, H, cap, 64)[:, :E]
            want = ref.reshape(E, H, 64).transpose(1, 0, 2)
            # (bound: 16 mantissa bits of the activations, as above)
            assert float(np.max(np.abs(got - want))) <= 2e-3 * max(1.0, float(np.max(np.abs(want)))), (E, what)
    ctx.close()


@pytest.mark.parametrize("E", [17, 63, 64])
@pytest.mark.parametrize("ffn,H", [("relu", 8), ("gated_gelu", 6)])
def test_norms_without_epsilon(torch_cuda, E, ffn, H):
    """ln_eps = 0: rows that do not exist (the encoder's tiles past the last id, the places of a block pass past its last row) have no
    squares to divide by, and nothing of them may reach a row that does exist.  Cross keys and values, logits of 1, 5 and 9 rows."""
    from oracle.t5 import Model
    from paper_2302_07863_b200.binding import BF16, Config, Context, model_cfg, upload_model
    torch = torch_cuda
    s = dataclasses.replace(MODEL_SHAPES["wide_s"], name="eps_" + ffn, n_layers=2, d_model=512, n_heads=H, d_kv=64, d_ff=1024, ffn=ffn, vocab=300, eps=0.0)
    w = gen_model(s, 5, "bf16")
    dev = upload_model(w, "cuda:0")
    ctx, m = Context(Config(model_cfg(s, 3.0), model_cfg(s, 3.0), BF16, 96, 20, 8, 0, -1, 0), s, dev, s, dev), Model(s, w, 3.0)
    ids = np.random.default_rng(E).integers(2, 300, size=E).astype(np.int32)
    ctx.encode(ids)
    st = m.start(ids, 20)
    for layer in range(2):
        for what, ref in ((0, st.ck[layer]), (1, st.cv[layer])):
            got = ctx.read_cache(1, what, layer, H, 96, 64)[:, :E]
            want = ref.reshape(E, H, 64).transpose(1, 0, 2)
            assert float(np.max(np.abs(got - want))) <= 2e-3 * max(1.0, float(np.max(np.abs(want)))), (layer, what)
    buf = torch.empty((16, 300), dtype=torch.float32, device="cuda")
    toks = [int(t) for t in np.random.default_rng(1).integers(2, 300, size=15)]
    at = 0
    for k in (1, 5, 9):
        ctx.large_verify(toks[at:at + k], 10.0, buf)
        z = m.forward_block(st, toks[at:at + k])
        assert np.max(np.abs(buf[:k].cpu().numpy() - z)) <= 2e-3 * max(1.0, np.max(np.abs(z))), k
        at += k
    ctx.close()


_len_cache = {}


@pytest.mark.parametrize("name,tuning", [("tiny", None), ("tiny", dict(fused=0)), ("odd_bf16", None), ("tiny_bf16", None), ("wide_bf16", None),
                                         ("wide_bf16", dict(fused=1)), ("wide_bf16", dict(fused=2)), ("wide_bf16", dict(fused=0))])
def test_pass_starts_behind_its_set_up_kernel(torch_cuda, name, tuning):
    """No kernel of a single-step call's pass may start before the kernel that writes the call descriptor is complete, since the
    kernels read the descriptor ahead of their dependency wait.  The launches are recorded, nothing runs."""
    from paper_2302_07863_b200.synthetic import make_context
    ctx, _, _ = make_context(name, 9.0, 9.0, tuning=tuning)
    for which, k in ((0, 1), (1, 1), (1, 2), (1, 8), (1, 9), (1, 16)):
        assert ctx.setup_edges(which, k) == 0, (which, k)
    ctx.close()


@pytest.mark.parametrize("name,scS,scL", [("tiny", 9.0, 9.0), ("odd_bf16", 9.0, 9.0), ("wide_bf16", 9.0, 11.0)])
def test_single_step_calls_without_logits_match_oracle(torch_cuda, name, scS, scL):
    """Calls without a logits buffer, as a host program makes them: the first two of a kind (small step; large pass of one row, of 2 to 8
    and of 9 to 16) launch their kernels, the later ones replay a graph.  Results against the oracle for every call, on growing caches,
    after rewinds, after an input of another length, after a reset and after generations (which move the caches on the device)."""
    from oracle.t5 import Model
    from paper_2302_07863_b200 import MODE_LARGE_ONLY, MODE_SMALL_ONLY
    from paper_2302_07863_b200.synthetic import make_context
    wl = WORKLOADS[name]
    ctx, _, _ = make_context(name, scS, scL, max_enc_len=140, max_dec_len=130)
    S, L = (Model(MODEL_SHAPES[m], gen_model(MODEL_SHAPES[m], wl.seed, wl.dtype), sc) for m, sc in ((wl.small, scS), (wl.large, scL)))
    tol = 1e-4 if wl.dtype == "fp32" else 2e-3   # logit error e of the other tests; lse moves by at most e, gaps and distances by 2 e
    rng = np.random.default_rng(3)
    V, afb, arb = S.s.vocab, 0.4, 15.0

    def check(o, Z, toks):
        for i, z in enumerate(Z):
            top, pmax, lse, gap = obild.max_prob(z)
            if gap > 2 * tol:
                assert (o.argmax[i] if len(toks) else o.argmax) == top
            assert abs((o.lse[i] if len(toks) else o.lse) - lse) <= tol
        if not len(toks):
            assert abs(o.pmax - pmax) <= 2 * tol * pmax + 1e-6 and abs(o.max_logit - z[top]) <= tol
            assert o.fallback == int(pmax < afb) or abs(pmax - afb) <= 2 * tol
            return
        d = [obild.max_prob(z)[2] - z[t] for z, t in zip(Z, toks[1:])]
        assert all(abs(a - b) <= 2 * tol for a, b in zip(o.d, d))
        if all(abs(x - arb) > 2 * tol for x in d):
            assert o.first_violation == next((i for i, x in enumerate(d) if x > arb), -1)

    def step(st):
        t = int(rng.integers(2, V))
        check(ctx.small_step(t, afb), [S.forward_one(st, t)], [])

    def verify(st, k):
        toks = [int(t) for t in rng.integers(2, V, size=k)]
        check(ctx.large_verify(toks, arb), L.forward_block(st, toks), toks)

    KINDS = (1, 5, 12, 8, 9, 2)
    for E, again in ((23, 3), (131, 1)):
        ids = rng.integers(2, V, size=E).astype(np.int32)
        ctx.encode(ids)
        stS, stL = S.start(ids, 130), L.start(ids, 130)
        for _ in range(again):
            for k in KINDS[:3]:
                step(stS)
                verify(stL, k)
        for st, which in ((stS, 0), (stL, 1)):
            st.rewind(2)
            ctx.rewind(which, 2)
        for k in KINDS:
            step(stS)
            verify(stL, k)
        toks = ctx.generate(MODE_SMALL_ONLY, 0.0, 1.0, 7)["tokens"]
        stS = S.start(ids, 130)
        S.forward_block(stS, [0] + toks[:-1])
        step(stS)
        step(stS)
        toks = ctx.generate(MODE_LARGE_ONLY, 0.0, 1.0, 7)["tokens"]
        stL = L.start(ids, 130)
        L.forward_block(stL, [0] + toks[:-1])
        for k in KINDS:
            verify(stL, k)
        ctx.generate(MODE_SMALL_ONLY, 0.0, 1.0, 5)
        ctx.reset()
        stS, stL = S.start(ids, 130), L.start(ids, 130)
        for k in KINDS:
            step(stS)
            verify(stL, k)
    ctx.close()


@pytest.mark.parametrize("name,early_exit", [("tiny", 0), ("wide_bf16", 0), ("wide_bf16", 1)])
def test_encoder_time_out_reaches_the_caller(torch_cuda, name, early_exit):
    """A time-out noted while the encoder runs (bild_tuning.debug_skip_copies = 2 writes the code that an encoder kernel would): every call
    that decodes from that input must report it, also behind a reset or a generation, which start from a fresh decode state."""
    from paper_2302_07863_b200 import MODE_BILD, MODE_LARGE_ONLY, BildError
    from paper_2302_07863_b200.synthetic import make_context
    ctx, ids, wl = make_context(name, 9.0, 9.0, tuning=dict(debug_skip_copies=2), early_exit_layers=early_exit)

    def times_out(f):
        with pytest.raises(BildError) as e:
            f()
        assert e.value.code == -6
    u = np.full(4, 0.5, np.float32)
    for _ in range(2):
        ctx.encode(ids)
        times_out(lambda: ctx.small_step(0, 0.4))
        ctx.reset()
        times_out(lambda: ctx.large_verify([0, 5, 7], 10.0))
        times_out(lambda: ctx.generate(MODE_BILD, 0.4, 10.0, 3))
        times_out(lambda: ctx.generate(MODE_LARGE_ONLY, 0.4, 10.0, 2))
        times_out(lambda: ctx.generate_sampled(MODE_BILD, 0.4, 10.0, 3, 0.8, u, u))
    ctx.close()


def test_reciprocal_of_softmax_sums(torch_cuda):
    """The attention kernels' 1 / x against fp64 for every mantissa, at the exponents of a soft-max's sum (1 to 2048 keys and beyond).
    Bound: an approximation of relative error 2^-23, squared by the Newton step, and the step's two roundings of 2^-24 each."""
    from paper_2302_07863_b200 import binding
    torch = torch_cuda
    L = binding.lib()
    L.bild_debug_reciprocal.argtypes = [binding.C.c_void_p, binding.C.c_void_p, binding.C.c_int, binding.C.c_void_p]
    mant = torch.arange(1 << 23, device="cuda", dtype=torch.int32)
    y = torch.empty(1 << 23, device="cuda")
    for e in (-1, 0, 1, 5, 11, 12):
        x = (mant | ((127 + e) << 23)).view(torch.float32)
        assert L.bild_debug_reciprocal(x.data_ptr(), y.data_ptr(), x.numel(), torch.cuda.current_stream().cuda_stream) == 0
        err = (y.double() * x.double() - 1.0).abs().max().item()
        assert err <= 2.0 ** -23 + 2.0 ** -45, (e, err)
    assert (y > 0).all()


@pytest.mark.parametrize("name", ["tiny", "tiny_bf16"])
def test_new_context_takes_updated_weights(torch_cuda, name):
    """Some matrices are copied in another order when a context is created (W_fo; W_o and W_co of small fp32 models), so weights must not
    change under a context; one created after an update in place uses the new values of all of them."""
    from oracle.t5 import Model
    from paper_2302_07863_b200.binding import BF16, FP32, Config, Context, model_cfg, upload_model
    torch = torch_cuda
    wl = WORKLOADS[name]
    s = MODEL_SHAPES[wl.large]
    dev = upload_model(gen_model(s, 1, wl.dtype), "cuda:0")
    cfg = Config(model_cfg(s, 3.0), model_cfg(s, 3.0), BF16 if wl.dtype == "bf16" else FP32, 32, 20, 8, 0, -1, 0)
    ids = np.arange(2, 30, dtype=np.int32)
    old = Context(cfg, s, dev, s, dev)
    w = gen_model(s, 2, wl.dtype)
    for key, val in upload_model(w, "cuda:0").items():
        dev[key].copy_(val)
    new = Context(cfg, s, dev, s, dev)
    m = Model(s, w, 3.0)
    buf = torch.empty((16, s.vocab), dtype=torch.float32, device="cuda")
    for k in (1, 5):
        new.encode(ids)
        new.large_verify([0, 5, 9, 4, 7][:k], 10.0, buf)
        z = m.forward_block(m.start(ids, 20), [0, 5, 9, 4, 7][:k])
        assert np.max(np.abs(buf[:k].cpu().numpy() - z)) <= (1e-4 if wl.dtype == "fp32" else 2e-3) * max(1.0, np.max(np.abs(z)))
    old.close()
    new.close()


@pytest.mark.parametrize("name,noise", [("tiny", 0.0), ("tiny", 0.03), ("tiny", None), ("tiny_bf16", 0.0), ("tiny_bf16", 0.03), ("wide_bf16", None), ("wide_bf16", "exit")])
@pytest.mark.parametrize("top_p", [0.0, 0.8])
def test_drafting_ahead_is_the_serial_loop(torch_cuda, name, noise, top_p):
    """The loop in rounds against the serial one (draft_ahead = 0): tokens, trace and counts.  The small model is the large one
    (every large pass ends as proposed), the large one with `noise` on its weights (some do), another model (hardly any does) or the
    large one's first layer;
    fallbacks from none to all, blocks from 1 row to the most, ends by length at the first places and by token anywhere."""
    from paper_2302_07863_b200 import MODE_BILD, MODE_LARGE_ONLY, MODE_SMALL_ONLY
    from paper_2302_07863_b200.binding import BF16, FP32, Config, Context, model_cfg, upload_model
    wl = WORKLOADS[name]
    sL = MODEL_SHAPES[wl.large]
    wlarge = upload_model(gen_model(sL, wl.seed, wl.dtype), "cuda:0")
    if noise == "exit":
        sS, wsmall = dataclasses.replace(sL, n_layers=1), wlarge
    elif noise is None:
        sS = MODEL_SHAPES[wl.small]
        wsmall = upload_model(gen_model(sS, wl.seed, wl.dtype), "cuda:0")
    else:
        import torch
        torch.manual_seed(1)
        sS, wsmall = sL, {k: (v.float() * (1 + noise * torch.randn_like(v.float()))).to(v.dtype) for k, v in wlarge.items()}
    cap = 41
    ids = np.random.default_rng(5).integers(2, sL.vocab, size=min(wl.enc_len, 32)).astype(np.int32)
    u = np.random.default_rng(6).random((2, cap)).astype(np.float32)

    def contexts(max_draft, eos):
        cfg = Config(model_cfg(sS, 9.0), model_cfg(sL, 9.0), FP32 if wl.dtype == "fp32" else BF16, 32, cap, max_draft, 0, eos,
                     1 if noise == "exit" else 0)
        out = [Context(cfg, sS, wsmall, sL, wlarge, tuning=t) for t in (None, dict(draft_ahead=0))]
        for c in out:
            c.encode(ids)
        return out

    def run(c, afb, arb, n, mode=MODE_BILD):
        return c.generate_sampled(mode, afb, arb, n, top_p, u[0], u[1]) if top_p else c.generate(mode, afb, arb, n)

    eos = -1
    for max_draft in (10, 1, 4):
        both = contexts(max_draft, eos)
        r = run(both[1], 0.0, float("inf"), cap - 1)
        p = sorted(t[5] for t in r["trace"] if t[0] != 3)
        for q in (0.0, 0.2, 0.5, 1.1):   # share of the small model's steps that fall back (roughly: a run takes its own course)
            i = int(q * len(p))
            afb = 0.0 if i == 0 else 2.0 if i >= len(p) else (p[i - 1] + p[i]) / 2
            for arb in (1.0, 6.0):
                for n in (cap - 1,) if q != 0.5 else (1, 2, 3, 7, cap - 1):
                    want, got = run(both[1], afb, arb, n), run(both[0], afb, arb, n)
                    assert got["tokens"] == want["tokens"] and got["stats"] == want["stats"], (max_draft, q, arb, n)
                    assert [t[:5] for t in got["trace"]] == [t[:5] for t in want["trace"]]
                    # (fused sub-layers add partial sums in no fixed order: the last bits differ from run to run)
                    assert np.allclose([t[5] for t in got["trace"]], [t[5] for t in want["trace"]], rtol=1e-4, atol=1e-5)
        for mode in (MODE_SMALL_ONLY, MODE_LARGE_ONLY):
            assert run(both[0], 0.4, 1.0, cap - 1, mode)["tokens"] == run(both[1], 0.4, 1.0, cap - 1, mode)["tokens"]
        eos = want["tokens"][len(want["tokens"]) // 2] if max_draft == 10 else want["tokens"][-1]   # the next contexts end on it
        for c in both:
            c.close()


@pytest.mark.parametrize("dtype", ["bf16", "fp32"])
@pytest.mark.parametrize("later", [0.0, 0.3])
@pytest.mark.parametrize("top_p", [0.0, 0.8])
def test_several_blocks_of_drafts_in_a_large_pass(torch_cuda, dtype, later, top_p):
    """A small model much faster than the large one (its first layer of twelve; the others add `later` times what theirs would: nothing,
    or enough for a rollback or another token now and then), so that blocks of drafts pile up and a large pass takes several, to 16 rows:
    tokens, trace and counts against the serial loop."""
    from paper_2302_07863_b200 import MODE_BILD
    from paper_2302_07863_b200.binding import BF16, FP32, Config, Context, model_cfg, upload_model
    sL = dataclasses.replace(MODEL_SHAPES["wide_l"], n_layers=12)
    sS = dataclasses.replace(sL, n_layers=1)
    w = upload_model(gen_model(sL, 4, dtype), "cuda:0")
    for name in w:
        if name.startswith("dec.") and not name.startswith("dec.0.") and name.split(".")[-1] in ("wo", "wco", "wfo"):
            w[name] *= later
    cap = 120
    ids = np.random.default_rng(5).integers(2, sL.vocab, size=24).astype(np.int32)
    u = np.random.default_rng(6).random((2, cap)).astype(np.float32)
    for max_draft in (1, 4, 15):
        cfg = Config(model_cfg(sS, 9.0), model_cfg(sL, 9.0), FP32 if dtype == "fp32" else BF16, 32, cap, max_draft, 0, -1, 1)
        both = [Context(cfg, sS, w, sL, w, tuning=t) for t in (None, dict(draft_ahead=0))]

        def run(c, afb, arb):
            return c.generate_sampled(MODE_BILD, afb, arb, cap - 1, top_p, u[0], u[1]) if top_p else c.generate(MODE_BILD, afb, arb, cap - 1)

        for c in both:
            c.encode(ids)
        p = sorted(t[5] for t in run(both[1], 0.0, float("inf"))["trace"] if t[0] != 3)
        for q in (0.15, 0.5, 0.8):
            i = int(q * len(p))
            for arb in (4.0, float("inf")):
                want = run(both[1], (p[i - 1] + p[i]) / 2, arb)
                for _ in range(3):
                    got = run(both[0], (p[i - 1] + p[i]) / 2, arb)
                    assert got["tokens"] == want["tokens"] and got["stats"] == want["stats"], (max_draft, q, arb)
                    assert [t[:5] for t in got["trace"]] == [t[:5] for t in want["trace"]]
                    # (blocks of another size, partial sums in another order: a single row has its fp32 products, rows of a block 16 mantissa bits)
                    assert np.allclose([t[5] for t in got["trace"]], [t[5] for t in want["trace"]], rtol=1e-4 if dtype == "fp32" else 2e-3,
                                       atol=1e-5 if dtype == "fp32" else 2e-3)
        for c in both:
            c.close()


@pytest.mark.parametrize("dtype,tuning", [("bf16", {}), ("bf16", dict(fused=0, enc_split_k=0)), ("fp32", {}), ("small_fp32", {})])
@pytest.mark.parametrize("all_alone", [True, False])
def test_blocks_that_share_a_pass_are_computed_as_alone(torch_cuda, dtype, tuning, all_alone):
    """Drafts pile up in front of a slow large model (as below).  Blocks of one row (all of them, or some) keep the kernels of a single row, with 24
    mantissa bits of the activations: values of the trace and the large model's cached keys and values against the serial loop's, where every block has a pass
    of its own.  One kernel per operation and fp32: the same to the last bit, whatever the timing."""
    from paper_2302_07863_b200 import MODE_BILD
    from paper_2302_07863_b200.binding import BF16, FP32, Config, Context, model_cfg, upload_model
    sL = dataclasses.replace(MODEL_SHAPES["tiny_l" if dtype == "small_fp32" else "wide_l"], n_layers=12)
    sS = dataclasses.replace(sL, n_layers=1)
    w = upload_model(gen_model(sL, 4, "bf16" if dtype == "bf16" else "fp32"), "cuda:0")
    for name in w:
        if name.startswith("dec.") and not name.startswith("dec.0.") and name.split(".")[-1] in ("wo", "wco", "wfo"):
            w[name] *= 0.05   # (small enough that the small model's tokens stand, and what later layers compute still shows)
    cap, n = 61, 60
    cfg = Config(model_cfg(sS, 9.0), model_cfg(sL, 9.0), BF16 if dtype == "bf16" else FP32, 32, cap, 4, 0, -1, 1)
    both = [Context(cfg, sS, w, sL, w, tuning=dict(tuning, **t)) for t in ({}, dict(draft_ahead=0))]
    for c in both:
        c.encode(np.random.default_rng(5).integers(2, sL.vocab, size=24).astype(np.int32))
    afb = 2.0
    if not all_alone:
        p = sorted(t[5] for t in both[1].generate(MODE_BILD, 0.0, float("inf"), n)["trace"] if t[0] != 3)
        i = int(0.7 * len(p))
        afb = (p[i - 1] + p[i]) / 2
    want = both[1].generate(MODE_BILD, afb, float("inf"), n)
    keys = [both[1].read_cache(1, what, layer, sL.n_heads, cap, sL.d_kv)[:, :n - 8] for layer in range(12) for what in (2, 3)]
    exact = dtype != "bf16" or "fused" in tuning
    for _ in range(4):
        before = both[0].loop_counts()
        got = both[0].generate(MODE_BILD, afb, float("inf"), n)
        ran = {k: v - before[k] for k, v in both[0].loop_counts().items()}
        assert got["tokens"] == want["tokens"] and got["stats"] == want["stats"]
        alone = sum(1 for t in want["trace"] if t[0] == 3 and t[3] == 1)
        passes = ran["large1"] + ran["large8"] + ran["large_more"]
        assert ran["large1"] >= alone and (not all_alone or passes == ran["large1"])
        assert not exact or passes == want["stats"]["large_calls"]
        a, b = [t[5] for t in got["trace"]], [t[5] for t in want["trace"]]
        # (fused sub-layers add partial sums in no fixed order, 1e-7 each, through 12 layers: 6e-7 of the cached keys seen with single rows, 3e-6 with one
        # row in a block of 16 mantissa bits; two more rows a block: those 16 bits fall otherwise where the sums do)
        assert a == b if exact else np.allclose(a, b, rtol=1e-4, atol=1e-5)
        for i, k in enumerate(keys):
            g = both[0].read_cache(1, 2 + i % 2, i // 2, sL.n_heads, cap, sL.d_kv)[:, :n - 8]
            assert np.array_equal(g, k) if exact else np.max(np.abs(g - k)) <= (1.5e-6 if all_alone else 2e-5) * np.max(np.abs(k)), i
    for c in both:
        c.close()


@pytest.mark.parametrize("top_p", [0.0, 0.05, 0.2])
def test_large_passes_do_take_several_blocks(torch_cuda, top_p):
    """What the test above is about happens: over a sweep, fewer large passes than blocks, passes of more than 8 rows, rollbacks in a block behind
    another one of its pass, drawn tokens that stand behind others (top_p = 0.05: mostly of a nucleus of one); tokens, trace and counts against the serial loop."""
    from paper_2302_07863_b200 import MODE_BILD
    from paper_2302_07863_b200.binding import BF16, Config, Context, model_cfg, upload_model
    sL = dataclasses.replace(MODEL_SHAPES["wide_l"], n_layers=12)
    sS = dataclasses.replace(sL, n_layers=1)
    w = upload_model(gen_model(sL, 4, "bf16"), "cuda:0")
    for name in w:
        if name.startswith("dec.") and not name.startswith("dec.0.") and name.split(".")[-1] in ("wo", "wco", "wfo"):
            w[name] *= 0.0
    cap = 120
    u = np.random.default_rng(6).random((2, cap)).astype(np.float32)
    ran, blocks = {}, 0
    for max_draft in (3, 4):
        cfg = Config(model_cfg(sS, 9.0), model_cfg(sL, 9.0), BF16, 32, cap, max_draft, 0, -1, 1)
        both = [Context(cfg, sS, w, sL, w, tuning=t) for t in (None, dict(draft_ahead=0))]

        def run(c, afb, arb):
            return c.generate_sampled(MODE_BILD, afb, arb, cap - 1, top_p, u[0], u[1]) if top_p else c.generate(MODE_BILD, afb, arb, cap - 1)

        for c in both:
            c.encode(np.random.default_rng(5).integers(2, sL.vocab, size=24).astype(np.int32))
        p = sorted(t[5] for t in run(both[1], 0.0, float("inf"))["trace"] if t[0] != 3)
        for q in (0.0, 0.15, 0.3, 0.5):
            i = int(q * len(p))
            for arb in (1.0, 2.0, 4.0):
                afb = (p[i - 1] + p[i]) / 2 if i else 0.0
                want, got = run(both[1], afb, arb), run(both[0], afb, arb)
                assert got["tokens"] == want["tokens"] and got["stats"] == want["stats"], (max_draft, q, arb)
                assert [t[:5] for t in got["trace"]] == [t[:5] for t in want["trace"]]
                # (fused sub-layers add partial sums in no fixed order; every row is computed with the bits it has alone)
                assert np.allclose([t[5] for t in got["trace"]], [t[5] for t in want["trace"]], rtol=1e-4, atol=1e-5)
                blocks += want["stats"]["large_calls"]
        for k, n in both[0].loop_counts().items():
            ran[k] = ran.get(k, 0) + n
        for c in both:
            c.close()
    assert ran["large1"] + ran["large8"] + ran["large_more"] <= blocks - 40, (ran, blocks)
    assert ran["large_more"] >= 5, ran
    assert ran["later_rollbacks"] >= 1 or top_p == 0.2, ran


@pytest.mark.parametrize("n_layers,d,H,E", [(3, 128, 2, 5), (1, 64, 1, 64), (2, 128, 3, 65), (3, 192, 4, 130), (50, 64, 1, 40), (50, 64, 5, 200)])
def test_cross_kv_of_all_layers_in_one_launch(torch_cuda, n_layers, d, H, E):
    """Cross-attention keys and values of every decoder layer against the oracle: row tiles that do not fill a pair of blocks, more layers than a
    launch takes, fewer items than pairs and more than one a pair, token tiles of 64 and 128."""
    from oracle.t5 import Model
    from paper_2302_07863_b200.binding import BF16, Config, Context, model_cfg, upload_model
    s = dataclasses.replace(MODEL_SHAPES["wide_s"], n_layers=n_layers, d_model=d, n_heads=H, d_ff=128)
    w = gen_model(s, 11, "bf16")
    dev = upload_model(w, "cuda:0")
    cap = E + 3
    ctx = Context(Config(model_cfg(s, 1.0), model_cfg(s, 1.0), BF16, cap, 8, 4, 0, -1, 0), s, dev, s, dev)
    ids = np.random.default_rng(E).integers(2, s.vocab, size=E).astype(np.int32)
    ctx.encode(ids)
    st = Model(s, w, 1.0).start(ids, 8)
    for which in (0, 1):
        for l in sorted({0, n_layers // 2, n_layers - 1}):
            for what, ref in ((0, st.ck[l]), (1, st.cv[l])):
                got = ctx.read_cache(which, what, l, H, cap, 64)[:, :E]
                want = ref.reshape(E, H, 64).transpose(1, 0, 2)
                # 16 mantissa bits of the activations through n_layers encoder layers, fp32 sums
                assert np.max(np.abs(got - want)) <= 2e-3 * max(1.0, np.max(np.abs(want))), (which, l, what)
    ctx.close()


@pytest.mark.parametrize("d,H,vocab,n_layers", [(512, 6, 131099, 1), (512, 6, 150011, 3), (1024, 4, 66003, 2), (192, 3, 349600, 1)])
def test_single_rows_with_part_of_the_head_asked_for(torch_cuda, d, H, vocab, n_layers):
    """Single-row passes in front of a streaming head of more than 128 MB, for whose weights they ask: vocabularies that fill neither the last warp's
    range nor all ranges, fewer and more kernels than ask; logits of both models against the oracle."""
    from oracle.t5 import Model
    from paper_2302_07863_b200.binding import BF16, Config, Context, model_cfg, upload_model
    s = dataclasses.replace(MODEL_SHAPES["wide_s"], name="ahead", n_layers=n_layers, d_model=d, n_heads=H, d_kv=64, d_ff=256, vocab=vocab)
    w = gen_model(s, 3, "bf16")
    dev = upload_model(w, "cuda:0")
    ctx, m = Context(Config(model_cfg(s, 3.0), model_cfg(s, 3.0), BF16, 16, 8, 4, 0, -1, 0), s, dev, s, dev), Model(s, w, 3.0)
    ids = np.random.default_rng(1).integers(2, vocab, size=9).astype(np.int32)
    ctx.encode(ids)
    st = m.start(ids, 8)
    buf = torch_cuda.empty((1, vocab), dtype=torch_cuda.float32, device="cuda")
    for tok in (0, vocab - 1, 17):
        z = m.forward_one(st, tok)
        for call in (lambda: ctx.small_step(tok, 0.4, buf), lambda: ctx.large_verify([tok], 10.0, buf)):
            out = call()
            # 16 mantissa bits of the activations (encoder, cross keys), fp32 sums
            assert np.max(np.abs(buf[0].cpu().numpy() - z)) <= 2e-3 * max(1.0, float(np.max(np.abs(z)))), (d, vocab, tok)
            assert (out.argmax if hasattr(out, "pmax") else out.argmax[0]) == int(np.argmax(z))
    ctx.close()


@pytest.mark.parametrize("d,H,dkv,F,ffn", [(512, 6, 64, 1024, "gated_gelu"), (768, 12, 64, 2048, "relu"), (768, 12, 32, 1032, "gated_gelu"), (1024, 16, 64, 2816, "gated_gelu"),
                                           (640, 8, 64, 520, "relu"), (512, 8, 32, 4096, "relu"), (1024, 3, 64, 264, "relu")])
def test_single_rows_of_fixed_and_other_widths(torch_cuda, d, H, dkv, F, ffn):
    """The single-row kernels built for rows of 512, 768 and 1024 columns and heads of 64 channels, and those that take other shapes: logits of both
    models, steps one after the other, against the oracle."""
    from oracle.t5 import Model
    from paper_2302_07863_b200.binding import BF16, Config, Context, model_cfg, upload_model
    s = dataclasses.replace(MODEL_SHAPES["wide_s"], name="width", n_layers=2, d_model=d, n_heads=H, d_kv=dkv, d_ff=F, ffn=ffn, vocab=300)
    w = gen_model(s, 3, "bf16")
    dev = upload_model(w, "cuda:0")
    ctx, m = Context(Config(model_cfg(s, 3.0), model_cfg(s, 3.0), BF16, 96, 40, 4, 0, -1, 0), s, dev, s, dev), Model(s, w, 3.0)
    ctx.encode(np.random.default_rng(1).integers(2, 300, size=90).astype(np.int32))
    st = m.start(np.random.default_rng(1).integers(2, 300, size=90).astype(np.int32), 40)
    buf = torch_cuda.empty((1, 300), dtype=torch_cuda.float32, device="cuda")
    for tok in np.random.default_rng(2).integers(0, 300, size=35):
        z = m.forward_one(st, int(tok))
        for call in (lambda: ctx.small_step(int(tok), 0.4, buf), lambda: ctx.large_verify([int(tok)], 10.0, buf)):
            call()
            # 16 mantissa bits of the activations (encoder, cross keys), fp32 sums
            assert np.max(np.abs(buf[0].cpu().numpy() - z)) <= 2e-3 * max(1.0, float(np.max(np.abs(z)))), (d, H, tok)
    ctx.close()


@pytest.mark.parametrize("name", ["tiny", "wide_bf16"])
def test_rewinds_reach_the_device_by_every_way(torch_cuda, name):
    """A length that bild_rewind has set is the one the next step starts from, whatever comes between: nothing, a generation's results fetched
    again (which reads the state back), timed passes (which move the lengths), steps and rewinds of both models."""
    from paper_2302_07863_b200.synthetic import make_context
    ctx, ids, _ = make_context(name, 9.0, 11.0)
    ctx.encode(ids)

    def steps():
        ctx.small_step(8, 0.4)
        ctx.rewind(0, 1)
        ctx.large_verify([8, 2], 10.0)
        ctx.rewind(1, 1)

    def timed():
        ctx.time_pass(0, 1, 3, 1)
        ctx.time_pass(1, 2, 3, 1)
        ctx.rewind(0, 1)
        ctx.rewind(1, 1)

    between = [lambda: None, lambda: ctx.fetch_result(4), timed, steps]
    want = None
    for turn in range(2):   # (plain launches, then graphs)
        for i, f in enumerate(between):
            ctx.reset()
            for t in (0, 5, 9, 4):
                ctx.small_step(t, 0.4)
            ctx.large_verify([0, 5, 9, 4], 10.0)
            for n in (3, 1):
                ctx.rewind(0, n)
                ctx.rewind(1, n)
            f()
            s, v = ctx.small_step(7, 0.4), ctx.large_verify([7, 3, 6], 10.0)
            got = [s.max_logit, s.lse, s.pmax, *v.lse[:3], *v.d[:2]]
            want = want or got
            # (fused sub-layers add partial sums in no fixed order)
            assert np.allclose(got, want, rtol=1e-5, atol=1e-5), (turn, i)
    with pytest.raises(Exception):
        ctx.rewind(0, 3)   # the cache holds 2 rows
    ctx.close()


def _captured(ctx, call):
    """`call` while the context's stream is being captured into a graph that is dropped: nothing of it runs, and the wait at its end is an error."""
    from cuda.bindings import runtime as cudart
    from paper_2302_07863_b200 import BildError
    assert cudart.cudaStreamBeginCapture(ctx.stream.cuda_stream, cudart.cudaStreamCaptureMode.cudaStreamCaptureModeRelaxed)[0] == 0
    with pytest.raises(BildError):
        call()
    cudart.cudaStreamEndCapture(ctx.stream.cuda_stream)   # (reports that the capture was cut short)


def _context_on_a_stream(torch):
    from paper_2302_07863_b200.binding import BF16, Config, Context, model_cfg, upload_model
    s = MODEL_SHAPES["wide_s"]
    dev = upload_model(gen_model(s, 5, "bf16"), "cuda:0")
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()   # (the weights were written on another stream)
    ctx = Context(Config(model_cfg(s, 3.0), model_cfg(s, 3.0), BF16, 32, 20, 8, 0, -1, 0), s, dev, s, dev, stream=stream)
    ctx.encode(np.arange(2, 20, dtype=np.int32))
    return ctx


@pytest.mark.parametrize("call", ["step", "verify", "generate", "read"])
def test_an_error_is_reported_once(torch_cuda, call):
    """The call behind one that failed on the host checks its own launches, not that one's."""
    from paper_2302_07863_b200 import MODE_BILD
    ctx = _context_on_a_stream(torch_cuda)
    want = ctx.small_step(7, 0.4).lse
    ctx.reset()
    _captured(ctx, {"step": lambda: ctx.small_step(7, 0.4), "verify": lambda: ctx.large_verify([7], 10.0), "read": lambda: ctx.fetch_result(4),
                    "generate": lambda: ctx.generate(MODE_BILD, 0.4, 10.0, 3)}[call])
    ctx.reset()
    assert abs(ctx.small_step(7, 0.4).lse - want) <= 1e-5
    ctx.close()


@pytest.mark.parametrize("graphs", [False, True])
@pytest.mark.parametrize("call", ["step", "verify", "generate", "read"])
def test_rewinds_outlive_a_call_that_does_not_run(torch_cuda, call, graphs):
    """A length that bild_rewind has set holds although the call behind it fails before its kernels have run."""
    from paper_2302_07863_b200 import MODE_BILD

    def fill(ctx):
        for t in (0, 5, 9, 4) if graphs else (0,):   # (the first two calls of a kind are plain launches)
            ctx.small_step(t, 0.4)
            ctx.large_verify([t], 10.0)
        ctx.rewind(0, 2 if graphs else 0)
        ctx.rewind(1, 1 if graphs else 0)

    def results(ctx):
        a, b = ctx.small_step(7, 0.4), ctx.large_verify([7], 10.0)
        return [a.lse, a.pmax, a.max_logit, b.lse[0]]

    ctx = _context_on_a_stream(torch_cuda)
    fill(ctx)
    want = results(ctx)
    if graphs:
        ctx.reset()
    else:
        ctx.close()
        ctx = _context_on_a_stream(torch_cuda)
    fill(ctx)
    _captured(ctx, {"step": lambda: ctx.small_step(7, 0.4), "verify": lambda: ctx.large_verify([7], 10.0), "read": lambda: ctx.fetch_result(4),
                    "generate": lambda: ctx.generate(MODE_BILD, 0.4, 10.0, 3)}[call])
    # (fused sub-layers add partial sums in no fixed order; at another place of the caches the results are off by 1e-3)
    assert np.allclose(results(ctx), want, rtol=1e-5, atol=1e-5)
    ctx.close()


def test_steps_wait_as_the_device_flags_say(torch_cuda):
    """cudaDeviceScheduleBlockingSync: a step behind 15 ms of other work on its stream leaves the CPU alone while it waits.  (In a process of
    its own: the flags belong to the device's context.)"""
    import os
    import subprocess
    import sys
    code = """
import time
from cuda.bindings import runtime as r
assert r.cudaSetDeviceFlags(r.cudaDeviceScheduleBlockingSync)[0] == 0
import torch
from paper_2302_07863_b200.synthetic import make_context
ctx, ids, _ = make_context("wide_bf16", 9.0, 9.0)
ctx.encode(ids)
for t in range(4):
    ctx.small_step(t, 0.4)
share = []
for t in range(5):
    torch.cuda._sleep(30_000_000)   # clocks
    a, b = time.perf_counter(), time.thread_time()
    ctx.small_step(t, 0.4)
    a, b = time.perf_counter() - a, time.thread_time() - b
    assert a > 5e-3, a
    share.append(b / a)
ctx.close()
print("share", sorted(share)[2])
"""
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    out = subprocess.run([sys.executable, "-c", code], cwd=root, capture_output=True, text=True, timeout=300)
    assert out.returncode == 0, out.stderr
    # a blocked thread uses some tens of microseconds of 15 ms, a polling one all of them
    assert float(out.stdout.split("share")[1]) < 0.3, out.stdout


@pytest.mark.parametrize("M", [1, 5, 16])
def test_linear_on_weights_the_kernel_in_front_wrote(torch_cuda, M):
    """bild_op_linear whose matrix is the result of the call before, which lets the kernel behind it start early: the product of the two, with other
    numbers in the same memory each time."""
    from paper_2302_07863_b200 import op_linear
    torch = torch_cuda
    g = torch.Generator("cuda").manual_seed(1)
    for i in range(8):
        A, B, X = (torch.randn(size, device="cuda", generator=g) for size in ((1024, 2048), (16, 2048), (M, 1024)))
        W = op_linear(A, B, None, 0.0, 16, 1024, 2048)             # [16][1024] = B A^T
        Y = op_linear(W, X, None, 0.0, M, 16, 1024)                # [M][16] = X W^T
        want = X.double() @ (B.double() @ A.double().T).T
        # fp32 sums of 2048 and then 1024 terms in other orders: a few 1e-7 of the sums' magnitude
        assert (Y.double() - want).abs().max().item() <= 1e-5 * want.abs().max().item(), i
