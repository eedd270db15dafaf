"""Rounding of the tensor-core prefill attention against the mma.sync one's, which
serves the same prompts in smaller batches.

The layer is made exact everywhere else: embeddings of +-1 with epsilon 0, so that the
norm scale is 1; one-hot q, k, v and output matrices with 8-bit values in dimensions that
the rotation leaves alone (rotary base 1e38); no MLP; the LM head the identity. What
the logits then differ by from a 64-bit attention over the same q, k and v is the
rounding of the probabilities and that of the attention's output."""
import math

import numpy as np
import pytest

from helpers import create
from test_gpu_parity import _ax, run_prefill

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

H, G, d, D, V, S, N = 8, 2, 128, 1024, 1024, 384, 128
SHAPE = dict(L=1, D=D, H=H, G=G, d=d, F=64, V=V, tie=False, bias=False, theta=1e38, eps=0.0)
O_SCALE = 1024.0  # the attention's output dominates the residual stream


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2608_19889_gb300 import build
    build.build()


def _model(spread):
    """Weights, and (signs, q, k, v maps) to form the exact layer from: scores of a
    standard deviation of `spread` (natural units)."""
    r = np.random.default_rng(5)
    still = np.r_[d // 4:d // 2, 3 * d // 4:d]  # rotated by at most 1e-19 * position: not at all in 32 bits
    sign = r.choice([-1.0, 1.0], (V, D))
    c0 = math.sqrt(spread / math.sqrt(len(still) / d))  # std = c0^2 * sqrt(64 / 128)

    def bf16(v):
        return torch.tensor(v, dtype=torch.float32).to(torch.bfloat16)

    def one_hot(heads, dims, scale):
        col = np.stack([r.choice(D, d, replace=False) for _ in range(heads)])
        val = np.zeros((heads, d))
        val[:, dims] = bf16(scale * r.uniform(0.7, 1.3, (heads, len(dims)))).float().numpy()
        w = np.zeros((heads * d, D))
        w[np.arange(heads * d), col.ravel()] = val.ravel()
        return w

    wq, wk, wv = one_hot(H, still, c0), one_hot(G, still, c0), one_hot(G, np.arange(d), 1.0)
    p = "model.layers.0."
    one = torch.ones(D, dtype=torch.bfloat16, device="cuda")
    w = {"model.embed_tokens.weight": sign, "lm_head.weight": np.eye(D), p + "self_attn.q_proj.weight": wq,
         p + "self_attn.k_proj.weight": wk, p + "self_attn.v_proj.weight": wv,
         p + "self_attn.o_proj.weight": O_SCALE * np.eye(D), p + "mlp.gate_proj.weight": np.zeros((64, D)),
         p + "mlp.up_proj.weight": np.zeros((64, D)), p + "mlp.down_proj.weight": np.zeros((D, 64))}
    w = {n: bf16(v).cuda() for n, v in w.items()}
    for n in ("model.norm.weight", p + "input_layernorm.weight", p + "post_attention_layernorm.weight"):
        w[n] = one
    return w, [torch.tensor(x, device="cuda") for x in (sign, wq, wk, wv)]


def _exact(ids, sign, wq, wk, wv):
    """Logits of the last position of each prompt, float64."""
    x = sign[torch.from_numpy(ids).long().cuda()]  # [N, S, D]
    q = (x[:, -1] @ wq.T).view(-1, H, d)
    k, v = ((x @ m.T).view(-1, S, G, d).repeat_interleave(H // G, 2) for m in (wk, wv))
    o = torch.einsum("nhs,nshd->nhd", torch.softmax(torch.einsum("nhd,nshd->nhs", q, k) / math.sqrt(d), -1), v)
    y = x[:, -1] + O_SCALE * o.reshape(-1, D)
    return (y / y.square().mean(-1, keepdim=True).sqrt()).cpu().numpy()


def errors(spread, prec):
    """rms error of the last positions' logits in batches of 8 prompts (3,072 rows) and of 4 (1,536 rows)."""
    ax = _ax()
    w, parts = _model(spread)
    ids = np.random.default_rng(6).integers(0, V, (N, S)).astype(np.int32)
    ref = _exact(ids, *parts)
    m = create(SHAPE, w, max_batch=8, max_context=S, max_prefill_tokens=8 * S, fp16=prec == "fp16")
    out = {}
    try:
        for B in (8, 4):
            lg = [run_prefill(m, ids[i:i + B], ax.AXON_LOGITS_LAST, V)[0] for i in range(0, N, B)]
            out[B] = np.concatenate(lg).reshape(N, V)
        assert ax.axon_check_device(m)[0] == 0
    finally:
        ax.axon_free(m)
    assert np.any(out[8] != out[4])  # two kernels
    return [float(np.sqrt(np.mean((out[B] - ref)**2))) for B in (8, 4)]


# 1.64: the scores' spread at 8B width with matrices of N(0, 0.02); 2.5: a sharper attention
@pytest.mark.parametrize("spread", [1.0, 1.64, 2.5])
def test_error_no_larger_than_the_smaller_kernel(spread):
    tc, mma = errors(spread, "fp16")
    print(f"spread {spread}: rms {tc:.3e} (mma.sync {mma:.3e}), ratio {tc / mma:.4f}")
    # 131,072 values in 1,024 independent (prompt, head) groups: the ratio of two rms errors of
    # equal expectation has a standard deviation below 0.7 / sqrt(1024 * 8) = 0.8 %
    assert tc <= 1.008 * mma
