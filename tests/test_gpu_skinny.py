"""GPU parity of the few-token projections (weights as the 128-row MMA operand,
K split over a cluster) against the oracle: token counts around every MMA width
(16, 32, 64, 128), weight rows that end inside a 128-row tile, a K that the
cluster does not divide, and an odd vocabulary. The shape's attention projections
are wide enough for the kernel to take any number of tokens."""
import numpy as np
import pytest

import synth_inputs as si
from helpers import LOGIT_TOL, create, gpu_weights, oracle_for
from test_gpu_parity import _ax, check, decode_steps, oracle_decode, run_prefill
from test_gpu_tile_widths import rounding_bound

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# 2112 = 16.5 tiles of 128 rows and 33 K blocks; gate/up 640 rows; 1003 = 7.8 tiles
WIDE = dict(L=1, D=2112, H=32, G=8, d=128, F=320, V=1003, tie=False, bias=True, theta=1e4, eps=1e-5)
# fp16 operands keep three more mantissa bits than bf16 ones
TOL = {"bf16": LOGIT_TOL, "fp16": LOGIT_TOL / 8}


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2608_19889_gb300 import build
    build.build()


@pytest.fixture(scope="module")
def oracle():
    w = gpu_weights(WIDE)
    return w, oracle_for(WIDE, w)


@pytest.mark.parametrize("prec", ["bf16", "fp16"])
def test_prompts_of_every_width(prec, oracle):
    ax = _ax()
    w, o = oracle
    m = create(WIDE, w, max_batch=1, max_context=128, max_prefill_tokens=128, fp16=prec == "fp16")
    try:
        for S in (1, 2, 15, 16, 17, 32, 33, 64, 65, 127, 128):
            ids = si.make_ids(1, S, WIDE["V"], seed=S)
            lg, nxt = run_prefill(m, ids, ax.AXON_LOGITS_ALL, WIDE["V"])
            check(lg, o.prefill(ids, o.new_contiguous_cache(1, 128)), tol=TOL[prec], what=f"S={S} ({prec})")
            assert np.array_equal(nxt, lg[:, -1].argmax(-1))
        assert ax.axon_check_device(m)[0] == 0
    finally:
        ax.axon_free(m)


@pytest.mark.parametrize("prec", ["bf16", "fp16"])
@pytest.mark.parametrize("B", [7, 16, 33, 64])
def test_decode_batches(B, prec, oracle, monkeypatch):
    ax = _ax()
    monkeypatch.setenv("AXON_NO_PERSIST", "1")
    w, o = oracle
    m = create(WIDE, w, max_batch=B, max_context=32, fp16=prec == "fp16")
    try:
        ids = si.make_ids(B, 9, WIDE["V"], seed=B)
        lg, nxt = run_prefill(m, ids, ax.AXON_LOGITS_LAST, WIDE["V"])
        cache = o.new_contiguous_cache(B, 32)
        check(lg, o.prefill(ids, cache, last_only=True)[:, -1], tol=TOL[prec], what=f"B={B} prefill")
        dl, fed = decode_steps(m, nxt, [9] * B, 2, WIDE["V"])
        check(dl, oracle_decode(o, cache, fed, [9] * B), tol=TOL[prec], what=f"B={B} decode ({prec})")
        assert ax.axon_check_device(m)[0] == 0
    finally:
        ax.axon_free(m)


@pytest.mark.parametrize("prec", ["bf16", "fp16"])
def test_more_rows_than_a_token_tile(prec, oracle):
    """129-300 rows: the O projection (17 weight tiles, K = 4096) runs on two or
    three token tiles, the last one ragged."""
    ax = _ax()
    w, o = oracle
    m = create(WIDE, w, max_batch=2, max_context=160, max_prefill_tokens=300, fp16=prec == "fp16")
    try:
        for B, S in ((1, 129), (2, 128), (2, 150)):
            ids = si.make_ids(B, S, WIDE["V"], seed=S)
            lg, _ = run_prefill(m, ids, ax.AXON_LOGITS_ALL, WIDE["V"])
            check(lg, o.prefill(ids, o.new_contiguous_cache(B, 160)), tol=TOL[prec], what=f"B={B} S={S} ({prec})")
        assert ax.axon_check_device(m)[0] == 0
    finally:
        ax.axon_free(m)


@pytest.mark.parametrize("prec", ["bf16", "fp16"])
def test_qkv_too_wide_for_the_kernel(prec):
    """41,472 weight rows of QKV are more 128-row tiles than the kernel takes: few tokens
    run it on the GEMM's general layout, the other projections on the kernel."""
    ax = _ax()
    shape = dict(L=1, D=64, H=288, G=18, d=128, F=128, V=304, tie=False, bias=True, theta=1e4, eps=1e-5)
    w = gpu_weights(shape)
    o = oracle_for(shape, w)
    m = create(shape, w, max_batch=9, max_context=80, fp16=prec == "fp16")
    try:
        for S in (9, 17, 64):
            ids = si.make_ids(1, S, shape["V"], seed=S)
            lg, _ = run_prefill(m, ids, ax.AXON_LOGITS_ALL, shape["V"])
            ref = o.prefill(ids, o.new_contiguous_cache(1, 80))
            check(lg, ref, tol=rounding_bound(ref, prec), what=f"S={S} ({prec})")
        ids = si.make_ids(9, 5, shape["V"], seed=3)
        _, nxt = run_prefill(m, ids, ax.AXON_LOGITS_LAST, shape["V"])
        cache = o.new_contiguous_cache(9, 80)
        o.prefill(ids, cache)
        dl, fed = decode_steps(m, nxt, [5] * 9, 2, shape["V"])
        ref = oracle_decode(o, cache, fed, [5] * 9)
        check(dl, ref, tol=rounding_bound(ref, prec), what=f"decode of 9 ({prec})")
        assert ax.axon_check_device(m)[0] == 0
    finally:
        ax.axon_free(m)
