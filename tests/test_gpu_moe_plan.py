"""The routing launches of the mixture-of-experts layer at the row counts where
they change: up to 32 slots (rows x experts per token) one CTA routes, sorts
and gathers, up to 256 rows it routes and sorts, beyond that routing is its
own launch; 1,024 slots are one round of the sort. The oracle takes the
GPU's own choices, which have to be valid top-k sets."""
import pytest

import synth_inputs as si
from helpers import create, gpu_weights, oracle_for, tiny_tol
from test_gpu_moe import MOE2, _check_routing, _moe_layers
from test_gpu_parity import _ax, check, run_prefill

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2608_19889_gb300 import build
    build.build()


@pytest.mark.parametrize("prec", ["bf16", "fp16"])
@pytest.mark.parametrize("rows", [1, 8, 9, 256, 257])
def test_rows_at_the_edges_of_the_routing_launches(rows, prec):
    ax = _ax()
    shape = MOE2  # 4 experts per token
    w = gpu_weights(shape)
    m = create(shape, w, max_batch=1, max_context=288, fp16=prec == "fp16")
    try:
        rec = torch.full((shape["L"], rows, shape["top_k"]), -1, dtype=torch.int32, device="cuda")
        ax.axon_moe_routing_record(m, rec, rows)
        ids = si.make_ids(1, rows, shape["V"], seed=rows)
        lg, _ = run_prefill(m, ids, ax.AXON_LOGITS_ALL, shape["V"])
        route = rec.cpu().numpy()
        o = oracle_for(shape, w)
        o.forced_routing = {l: route[l] for l in _moe_layers(shape)}
        ref = o.prefill(ids, o.new_contiguous_cache(1, 288))
        _check_routing(o, route, shape, f"{rows} rows {prec}")
        check(lg, ref, tol=tiny_tol(prec), what=f"{rows} rows ({prec})")
    finally:
        ax.axon_free(m)


@pytest.mark.parametrize("S", [3, 20, 150])
def test_token_whose_router_logits_are_not_numbers(S):
    """It is routed to valid, distinct experts, and the other sequence is as without it."""
    ax = _ax()
    shape = MOE2
    w = gpu_weights(shape)
    ids = si.make_ids(2, S, shape["V"] - 1, seed=S)
    w["model.embed_tokens.weight"][shape["V"] - 1] = float("nan")
    m = create(shape, w, max_batch=2, max_context=160, max_prefill_tokens=2 * S)
    try:
        rec = torch.full((shape["L"], 2 * S, shape["top_k"]), -1, dtype=torch.int32, device="cuda")
        ref, _ = run_prefill(m, ids, ax.AXON_LOGITS_LAST, shape["V"])
        ids[0, -1] = shape["V"] - 1
        ax.axon_moe_routing_record(m, rec, 2 * S)
        lg, _ = run_prefill(m, ids, ax.AXON_LOGITS_LAST, shape["V"])
        assert ax.axon_check_device(m)[0] == 0
        for l in _moe_layers(shape):
            for row in rec[l].tolist():
                assert len(set(row)) == shape["top_k"] and 0 <= min(row) and max(row) < shape["n_experts"]
        assert (lg[0] != lg[0]).all() and (lg[1] == ref[1]).all()
    finally:
        ax.axon_free(m)
