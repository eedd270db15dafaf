"""The persistent decode step's exchange of flagged words against the oracle:
operands that stage in several pieces (an MLP wide enough at head_dim 64), steps
of different batch sizes in turn on one model (what an earlier, larger batch left
in the buffers must not be taken for this step's), and several layers and steps
(flags of earlier layers and launches)."""
import ctypes

import numpy as np
import pytest

import synth_inputs as si
from helpers import create, gpu_weights, oracle_for, tiny_tol
from test_gpu_parity import _ax, check, decode_steps, oracle_decode, run_prefill
from test_gpu_persistent import _kinds

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# down projection K = 4928: 8 bf16 rows (or 4 rows of two fp16 terms) are 79 KB, the staging region 64 KB
PIECES = dict(L=3, D=128, H=4, G=2, d=64, F=4928, V=500, tie=False, bias=True, theta=1e4, eps=1e-5)


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2608_19889_gb300 import build
    build.build()


@pytest.mark.parametrize("prec,B", [("bf16", 8), ("bf16", 7), ("fp16", 4), ("fp16", 6), ("fp16", 1)])
def test_operand_staged_in_pieces(prec, B):
    ax = _ax()
    w = gpu_weights(PIECES)
    m = create(PIECES, w, max_batch=B, max_context=64, fp16=prec == "fp16")
    try:
        assert "decode_persistent" in _kinds(m, B, [20] * B)
        ids = si.make_ids(B, 20, PIECES["V"], seed=B)
        lg, nxt = run_prefill(m, ids, ax.AXON_LOGITS_LAST, PIECES["V"])
        o = oracle_for(PIECES, w)
        cache = o.new_contiguous_cache(B, 64)
        check(lg, o.prefill(ids, cache, last_only=True)[:, -1], tol=tiny_tol(prec), what="prefill")
        dl, fed = decode_steps(m, nxt, [20] * B, 6, PIECES["V"])
        check(dl, oracle_decode(o, cache, fed, [20] * B), tol=tiny_tol(prec), what=f"B={B} decode ({prec})")
        assert ax.axon_check_device(m)[0] == 0
    finally:
        ax.axon_free(m)


@pytest.mark.parametrize("prec", ["bf16", "fp16"])
def test_batch_sizes_in_turn(prec):
    """Sequence b of a step with fewer sequences is the same sequence b: its
    tokens are fed to the oracle in the same order."""
    ax = _ax()
    shape = dict(PIECES, F=192)
    B = 6
    w = gpu_weights(shape)
    m = create(shape, w, max_batch=B, max_context=64, fp16=prec == "fp16")
    try:
        ids = si.make_ids(B, 9, shape["V"], seed=5)
        run_prefill(m, ids, ax.AXON_LOGITS_LAST, shape["V"])
        o = oracle_for(shape, w)
        caches = [o.new_contiguous_cache(1, 64) for _ in range(B)]
        for b in range(B):
            o.prefill(ids[b:b + 1], caches[b], last_only=True)
        lens = np.full(B, 9)
        rng = np.random.Generator(np.random.PCG64(3))
        for n in (6, 1, 4, 2, 6, 3, 1, 5):
            tok = rng.integers(0, shape["V"], n).astype(np.int32)
            ctx = torch.from_numpy(lens[:n].astype(np.int32)).cuda()
            logits = torch.empty(n, shape["V"], device="cuda")
            nxt = torch.empty(n, dtype=torch.int32, device="cuda")
            ax.axon_decode_step(m, torch.from_numpy(tok).cuda(), ctx, logits=logits, next_tokens=nxt)
            ref = np.stack([o.decode_step(tok[b:b + 1], caches[b], lens[b:b + 1])[0] for b in range(n)])
            check(logits.cpu().numpy(), ref, tol=tiny_tol(prec), what=f"step of {n} ({prec})")
            lens[:n] += 1
            assert ctx.cpu().numpy().tolist() == lens[:n].tolist()
        assert ax.axon_check_device(m)[0] == 0
    finally:
        ax.axon_free(m)


@pytest.mark.parametrize("prec", ["bf16", "fp16"])
def test_position_outside_the_cache_is_reported_and_nothing_else(prec):
    """A sequence whose cache is full: DEVERR_POS (4) and no wait that ran out (8),
    while the other sequences of the step are as without it."""
    ax = _ax()
    shape = dict(PIECES, F=192, L=6)
    w = gpu_weights(shape)
    m = create(shape, w, max_batch=3, max_context=32, fp16=prec == "fp16")
    try:
        ids = si.make_ids(3, 9, shape["V"], seed=5)
        _, nxt = run_prefill(m, ids, ax.AXON_LOGITS_LAST, shape["V"])
        ref, _ = decode_steps(m, nxt, [9] * 3, 1, shape["V"])
        for full in (32, 40):
            tok, ctx = torch.from_numpy(nxt).cuda(), torch.tensor([9, full, 9], dtype=torch.int32, device="cuda")
            logits = torch.empty(3, shape["V"], device="cuda")
            ax.axon_decode_step(m, tok, ctx, logits=logits, next_tokens=torch.empty_like(tok))
            assert ax.axon_check_device(m)[1] == 4
            assert np.array_equal(logits.cpu().numpy()[[0, 2]], ref[[0, 2], 0])
            assert ctx.tolist() == [10, full + 1, 10]
    finally:
        ax.axon_free(m)


def test_flags_start_anew_before_they_wrap():
    """Steps on both sides of the 32-bit wrap, the ones after it with more sequences than
    any before (words that nothing has written yet): bit-identical to a model whose
    flags are far from it."""
    ax = _ax()
    shape = dict(PIECES, F=192)
    w = gpu_weights(shape)
    ids = si.make_ids(8, 9, shape["V"], seed=5)
    runs = []
    for epoch in (None, 2**32 - 9):  # steps of L + 1 = 4 flags: two fit
        m = create(shape, w, max_batch=8, max_context=32)
        try:
            _, nxt = run_prefill(m, ids, ax.AXON_LOGITS_LAST, shape["V"])
            if epoch is not None:
                assert ax.lib().axon_internal_persist_epoch(m, ctypes.c_uint32(epoch)) == 0
            out, lens = [], np.full(8, 9, dtype=np.int32)
            for n in (2, 1, 8, 3, 8):
                tok, ctx = torch.from_numpy(nxt[:n].copy()).cuda(), torch.from_numpy(lens[:n].copy()).cuda()
                logits = torch.empty(n, shape["V"], device="cuda")
                ax.axon_decode_step(m, tok, ctx, logits=logits, next_tokens=torch.empty_like(tok))
                out.append(logits.cpu().numpy())
                lens[:n] += 1
            assert ax.axon_check_device(m)[0] == 0
            runs.append(out)
        finally:
            ax.axon_free(m)
    for a, b in zip(*runs):
        assert np.array_equal(a, b)
