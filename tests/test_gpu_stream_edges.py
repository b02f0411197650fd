"""Edges of the per-sequence engine's streaming passes against the oracle:
slices around a thread's batch of units (one group of 256 units, several, a
ragged last unit), rows at every 16-byte offset, one to four rows in play.

The comparison and its tolerances are those of the parity tests.
"""
import pytest
import torch

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2410_18234_gb300 import mds  # noqa: E402
from synth import WorkloadSpec, make_workload, host_copy  # noqa: E402
from oracle.verify import oracle_verify  # noqa: E402
from parity import compare, check  # noqa: E402

DEV = "cuda:0"


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("V,cluster,models", [(7, 1, 1), (1024, 1, 1), (2049, 1, 2), (4095, 2, 3), (8192, 1, 1),
                                              (9001, 1, 3), (16384, 1, 2), (16392, 1, 1), (33003, 2, 1)])
def test_stream_edges(V, cluster, models, dtype):
    spec = WorkloadSpec(f"v{V}", B=6, K=3, L=2, V=V, dtype=dtype, model_ids=[k % models for k in range(3)],
                        target_scale=3.0, draft_sigma=[0.8, 1.2, 0.6][:models], t_target=0.8,
                        t_draft=[0.8, 1.1, 1.0][:models], data_seed=V)
    w = make_workload(spec, device=DEV)
    for scheme in ("single", "WIS", "WIS0", "SpecTr", "IS"):
        v = mds.Verifier(spec.B, spec.K, spec.L, V, dtype=dtype, cluster=cluster, omega0=10)
        out, acc, diag = v.verify(w.target, w.draft_list(), w.model_ids, w.tokens, w.temps, scheme, 31, diag=True)
        torch.cuda.synchronize()
        bits, _ = v.status()
        v.close()
        o_out, o_acc, recs = oracle_verify(*host_copy(w), scheme, 31, omega0=10)
        res = compare(out.cpu().numpy(), acc.cpu().numpy(), o_out, o_acc, recs, g_diag=diag.cpu().numpy(), scheme=scheme)
        check(res, scheme)
        assert bits == 0


@pytest.mark.parametrize("V,dtype", [(98304, "bf16"), (98305, "bf16"), (49152, "f32"), (49153, "f32")])
def test_single_draft_either_side_of_the_engine_rule(V, dtype):
    """One CTA a sequence (a batch of 304 at most): slices of 192 KB and just above."""
    spec = WorkloadSpec(f"v{V}", B=4, K=2, L=2, V=V, dtype=dtype, model_ids=[0, 0], target_scale=3.0,
                        draft_sigma=[0.8], t_target=0.8, t_draft=[0.8], data_seed=V)
    w = make_workload(spec, device=DEV)
    v = mds.Verifier(304, spec.K, spec.L, V, dtype=dtype)
    out, acc, diag = v.verify(w.target, w.draft_list(), w.model_ids, w.tokens, w.temps, "single", 31, diag=True)
    torch.cuda.synchronize()
    bits, _ = v.status()
    assert (v.cluster_size > 0) == (V * w.target.element_size() <= 192 * 1024), v.cluster_size
    v.close()
    o_out, o_acc, recs = oracle_verify(*host_copy(w), "single", 31)
    res = compare(out.cpu().numpy(), acc.cpu().numpy(), o_out, o_acc, recs, g_diag=diag.cpu().numpy(), scheme="single")
    check(res, "single")
    assert bits == 0
