"""GPU parity of the tensor-core prefill attention at the edges of its tiles
(128 query rows = PW positions x H/G heads, two tiles per CTA, 128 keys per
step) against the oracle: every grouping of heads, lengths around a tile, a
pair of tiles and a key step, a window that starts inside a key step, and
chunks after a past that is not a multiple of a cache block."""
import pytest

import synth_inputs as si
from helpers import create, gpu_weights, oracle_for, tiny_tol
from test_gpu_parity import _ax, check, run_prefill
from test_gpu_varlen import _case, _run_varlen

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2608_19889_gb300 import build
    build.build()


def _shape(H, G, d, **over):
    return dict(dict(L=2, D=128, H=H, G=G, d=d, F=128, V=304, tie=False, bias=True, theta=1e4, eps=1e-5), **over)


def _lengths(H, G):
    pw = 128 // (H // G)
    return sorted({1, 16, pw, pw + 1, 2 * pw, 2 * pw + 1, 65, 127, 128, 129, 273})


@pytest.mark.parametrize("prec", ["bf16", "fp16"])
@pytest.mark.parametrize("H,G,d", [(2, 2, 64), (3, 1, 64), (7, 1, 64), (16, 1, 64), (4, 1, 128), (5, 1, 128),
                                   (6, 3, 128)])
def test_every_position_at_tile_edges(H, G, d, prec):
    # one packed batch with a prompt of every length (above 64 rows: the tensor-core kernel)
    ax = _ax()
    shape = _shape(H, G, d)
    w = gpu_weights(shape)
    o = oracle_for(shape, w)
    lens = _lengths(H, G)
    m = create(shape, w, max_batch=len(lens), max_context=288, max_prefill_tokens=sum(lens), fp16=prec == "fp16")
    try:
        chunks = [si.make_ids(1, S, shape["V"], seed=S)[0] for S in lens]
        lg, _, cu = _run_varlen(m, chunks, torch.zeros(len(lens), dtype=torch.int32, device="cuda"),
                                ax.AXON_LOGITS_ALL, shape["V"])
        for i, c in enumerate(chunks):
            ref = o.prefill(c[None], o.new_contiguous_cache(1, 288))[0]
            check(lg[cu[i]:cu[i + 1]], ref, tol=tiny_tol(prec), what=f"H/G {H}/{G} S={len(c)}")
        assert ax.axon_check_device(m)[0] == 0
    finally:
        ax.axon_free(m)


@pytest.mark.parametrize("B,S,window", [(2, 385, 0), (1, 512, 0), (1, 400, 1), (1, 400, 100), (1, 400, 128),
                                        (2, 433, 130), (9, 256, 0)])
def test_prompts_of_one_length_with_and_without_window(B, S, window):
    ax = _ax()
    shape = _shape(4, 1, 128, window=window)
    w = gpu_weights(shape)
    o = oracle_for(shape, w)
    m = create(shape, w, max_batch=B, max_context=512, max_prefill_tokens=B * S)
    try:
        ids = si.make_ids(B, S, shape["V"], seed=9)
        lg, _ = run_prefill(m, ids, ax.AXON_LOGITS_ALL, shape["V"])
        check(lg, o.prefill(ids, o.new_contiguous_cache(B, 512)), tol=tiny_tol("bf16"), what=f"window {window}")
    finally:
        ax.axon_free(m)


@pytest.mark.parametrize("layout", ["contiguous", "paged"])
def test_chunks_after_odd_pasts(layout):
    # more than 32 sequences: the work items are found over two scans of the offsets
    first = [1, 17, 127, 128, 129] + [3] * 30
    second = [129, 1, 64, 1, 65] + [1, 2, 5] * 10
    _case(_shape(3, 1, 64), layout, "fp16", first=first, second=second, max_ctx=288)
