"""Rows masked with the storage type's lowest finite value, as samplers and
grammars mask them, against the oracle: a masked token has probability 0
wherever the mask lies (a thread's, a warp's or a slice's whole share, whose
own maximum is then the mask, and times log2(e) / T is -inf).  With -inf
masks besides, and a NaN inside a masked stretch, which the status reports.

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


def masked(V, dtype, kind, models=1):
    """A workload whose rows keep some tokens, the draft tokens among them, and the rest masked."""
    spec = WorkloadSpec(f"v{V}", B=6, K=3, L=2, V=V, dtype=dtype, model_ids=[k % models for k in range(3)],
                        target_scale=3.0, draft_sigma=[0.6, 1.0][:models], t_target=0.9, t_draft=[0.9, 1.1][:models],
                        data_seed=V)
    w = make_workload(spec, device=DEV)
    ids = torch.arange(V, device=DEV)
    if kind == "sparse":
        keep = ids % 97 == 3
    elif kind == "second-half":
        keep = ids >= V // 2
    else:                         # one stretch of 256 tokens in eight
        keep = (ids // 256) % 8 == 5
    keep[w.tokens.reshape(-1).long()] = True
    low = float("-inf") if kind == "stretches-inf" else torch.finfo(w.target.dtype).min
    for t in (w.target, w.drafts):
        t.masked_fill_(~keep, low)
    return w, keep


def run(w, scheme, cluster):
    s = w.spec
    v = mds.Verifier(s.B, s.K, s.L, s.V, dtype=s.dtype, omega0=10, cluster=cluster, acc_prob=0)
    out, acc, diag = v.verify(w.target, w.draft_list(), w.model_ids, w.tokens, w.temps, scheme, 31, diag=True)
    torch.cuda.synchronize()
    bits, _ = v.status()
    v.close()
    return out, acc, diag, bits


@pytest.mark.parametrize("cluster", [0, 2])
@pytest.mark.parametrize("kind", ["sparse", "second-half", "stretches", "stretches-inf"])
@pytest.mark.parametrize("V,dtype,models", [(20000, "bf16", 1), (33003, "bf16", 2), (16384, "f32", 1), (9001, "f32", 2)])
def test_masked_rows(V, dtype, models, kind, cluster):
    w, _ = masked(V, dtype, kind, models)
    for scheme in ("single", "WIS", "WIS0", "SpecTr", "IS"):
        out, acc, diag, bits = run(w, scheme, cluster)
        o_out, o_acc, recs = oracle_verify(*host_copy(w), scheme, 31, omega0=10)
        res = compare(out.cpu().numpy(), acc.cpu().numpy(), o_out, o_acc, recs, g_diag=diag.cpu().numpy(), scheme=scheme)
        check(res, scheme)
        assert bits == 0, (scheme, bits)


@pytest.mark.parametrize("scheme", ["single", "WIS"])
def test_nan_in_a_masked_stretch(scheme):
    w, keep = masked(20000, "bf16", "stretches-inf")
    at = int(torch.nonzero(~keep)[300])
    w.target[..., at] = float("nan")
    assert run(w, scheme, 0)[3] & mds.MDS_ST_NONFINITE
