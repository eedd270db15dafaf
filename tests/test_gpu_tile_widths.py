"""Output tiles of 192 and 224 columns of the prefill GEMM against the oracle: row
counts and widths at which a pass of 2,100 rows (17 row blocks on 152 SMs, the last of
them ragged) has every projection take one of them, with whole and with cut last
tiles. Widths of 256 and 128 are what the other prefill tests take."""
import ctypes

import pytest

import synth_inputs as si
from helpers import create, gpu_weights, oracle_for
from test_gpu_parity import _ax, check, run_prefill

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

BASE = dict(L=1, d=64, V=1000, tie=False, theta=1e4, eps=1e-5)
# QKV 1280 rows, O and down 1280, gate/up 1280: tiles of 192, the last one of 128 columns
W192 = dict(BASE, D=1280, H=12, G=4, F=640, bias=True)
# QKV 1792 rows (whole tiles of 224), O, down and gate/up 1664 (the last one of 96 columns)
W224 = dict(BASE, D=1664, H=20, G=4, F=832, bias=False)


def rounding_bound(ref, prec):
    """Bound on max |delta logit| from the 16-bit roundings of one layer.

    A rounding to unit roundoff u (2^-8 bf16, 2^-11 fp16) has a relative error of
    u / sqrt(3) * sqrt(E[1/m^2]) = 0.42 u rms over log-uniform mantissas m in [1, 2).
    Nine values are rounded (the operands of QKV, gate/up and the LM head, q, k, v, P, o and the
    gate's product u); the seven before the MLP enter the product of gate and up through
    both factors, so count twice: 7 * 2 + 2 = 16 independent terms of the size of the output, hence
    4 * 0.42 u relative to the logits' spread. Of 2.1 million logits none is expected
    beyond 6 standard deviations (4e-3 of them). Observed rms errors, kernels with
    tiles of 128 and 256 / these: D = 1664 bf16 4.71e-3 / 4.72e-3 and fp16 5.27e-4 /
    5.30e-4 of logits of spread 0.818, i.e. 3.5 and 3.2 times 0.42 u."""
    u = {"bf16": 2.0**-8, "fp16": 2.0**-11}[prec]
    return 6 * 4 * 0.42 * u * float(ref.std())


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2608_19889_gb300 import build
    build.build()


@pytest.mark.parametrize("prec", ["bf16", "fp16"])
@pytest.mark.parametrize("shape,width", [(W192, 192), (W224, 224)], ids=["192", "224"])
def test_middle_tile_widths(shape, width, prec):
    ax = _ax()
    B, S = 4, 525
    w = gpu_weights(shape)
    m = create(shape, w, max_batch=B, max_context=528, fp16=prec == "fp16", max_prefill_tokens=B * S)
    try:
        # QKV, O and down, gate/up: all take the width that the case is about
        for n in ((shape["H"] + 2 * shape["G"]) * shape["d"], shape["D"], 2 * shape["F"]):
            assert ax.lib().axon_internal_gemm_tile_n(m, ctypes.c_int32(B * S), ctypes.c_int32(n)) == width
        ids = si.make_ids(B, S, shape["V"], seed=7)
        lg, _ = run_prefill(m, ids, ax.AXON_LOGITS_ALL, shape["V"])
        o = oracle_for(shape, w)
        ref = o.prefill(ids, o.new_contiguous_cache(B, 528))
        check(lg, ref, tol=rounding_bound(ref, prec), what=f"D={shape['D']} ({prec})")
        assert ax.axon_check_device(m)[0] == 0
    finally:
        ax.axon_free(m)
