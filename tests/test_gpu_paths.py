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
