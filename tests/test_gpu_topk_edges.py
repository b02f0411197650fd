"""The top-k kernel's selection where its bound fails or ties: flat rows, rows
of few values (more tokens at the bound than it sets aside), rows with fewer
finite logits than k or all of them past the first units, odd lengths in both
storage types, k = 1, 10 and 16.  Against the oracle with the same
restriction; the comparison and its tolerances are those of the parity tests.
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
NEG = float("-inf")


def shape(t, kind):
    """The rows of t (any leading shape) turned into the kind's."""
    V = t.shape[-1]
    ids = torch.arange(V, device=t.device)
    if kind == "flat":
        t.fill_(0.25)
    elif kind == "two-values":
        t.copy_((t.float() > 0).float() * 2.0)
    elif kind == "three-finite":
        t.masked_fill_((ids % (V // 3 + 1) != 7), NEG)
    elif kind == "late":          # the first half of the row is masked
        t.masked_fill_(ids < V // 2, NEG)
    elif kind == "one-warp":      # the large logits lie in every sixteenth 512-byte stretch
        per = 512 // t.element_size()
        t.copy_(torch.where((ids // per) % 16 == 3, torch.full_like(t, 9.0), t.float().clamp(max=5.0).to(t.dtype)))


@pytest.mark.parametrize("V,dtype", [(20000, "bf16"), (33001, "bf16"), (9003, "f32")])
@pytest.mark.parametrize("kind", ["plain", "flat", "two-values", "three-finite", "late", "one-warp"])
def test_selection_edges(kind, V, dtype):
    spec = WorkloadSpec(kind, B=3, K=2, L=2, V=V, dtype=dtype, model_ids=[0, 0], target_scale=3.0, draft_sigma=[0.5],
                        t_target=1.0, t_draft=[1.0], data_seed=V)
    w = make_workload(spec, device=DEV)
    shape(w.target, kind)
    shape(w.drafts, kind)
    for k in (1, 10, 16):
        v = mds.Verifier(spec.B, spec.K, spec.L, V, dtype=dtype, top_k=k)
        for scheme in ("single", "WIS"):
            out, acc, diag = v.verify(w.target, w.draft_list(), w.model_ids, w.tokens, w.temps, scheme, 5, diag=True)
            torch.cuda.synchronize()
            o_out, o_acc, recs = oracle_verify(*host_copy(w), scheme, 5, top_k=k)
            res = compare(out.cpu().numpy(), acc.cpu().numpy(), o_out, o_acc, recs, g_diag=diag.cpu().numpy(),
                          scheme=scheme)
            check(res, f"{scheme} top-{k}")
        assert v.status()[0] == 0
        v.close()
