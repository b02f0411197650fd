"""One Verifier for calls of different schemes and numbers of draft models:
each call's slices, and so the workspace's layout, differ from the one
before.  Every call must give what a Verifier of its own gives, bit for bit.
"""
import pytest
import torch

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2410_18234_gb300 import mds  # noqa: E402
from synth import WorkloadSpec, make_workload  # noqa: E402

DEV = "cuda:0"


def workload(B, V, models):
    return make_workload(WorkloadSpec(f"m{models}", B=B, K=2, L=2, V=V, dtype="bf16",
                                      model_ids=[k % models for k in range(2)], target_scale=4.0,
                                      draft_sigma=[0.5, 1.0][:models], t_target=1.0, t_draft=[1.0, 1.3][:models],
                                      data_seed=3), device=DEV)


@pytest.mark.parametrize("B,V", [(256, 128256), (128, 50272)])
def test_calls_of_other_layouts(B, V):
    ws = {m: workload(B, V, m) for m in (1, 2)}

    def call(v, scheme, models):
        w = ws[models]
        out = v.verify(w.target, w.draft_list(), w.model_ids, w.tokens, w.temps, scheme, 9, diag=True)
        torch.cuda.synchronize()
        assert v.status()[0] & ~mds.MDS_ST_OMEGA0 == 0, (scheme, models)
        return out

    one = mds.Verifier(B, 2, 2, V)
    for scheme, models in [("WIS", 1), ("WIS0", 1), ("single", 1), ("WIS", 2), ("WIS0", 2), ("WIS", 1), ("single", 2),
                           ("WIS0", 1)]:
        got = call(one, scheme, models)
        own = mds.Verifier(B, 2, 2, V)
        want = call(own, scheme, models)
        own.close()
        for g, x in zip(got[:2], want[:2]):
            assert torch.equal(g, x), (scheme, models)
        # the depths a walk visited (the others' diagnostics are not written)
        seen = torch.arange(3, device=DEV)[None] <= want[1][:, None]
        assert torch.equal(got[2][seen], want[2][seen]), (scheme, models)
    one.close()


@pytest.mark.parametrize("scheme", ["single", "WIS", "WIS0"])
def test_small_calls_on_a_large_context(scheme):
    """Tasks are grouped by the call's batch, slices by the context's: a call
    of a batch's first sequences gives their results, bit for bit."""
    B, V = 400, 100000
    w = workload(B, V, 1)
    v = mds.Verifier(B, 2, 2, V)

    def call(n):
        out = v.verify(w.target[:n], [d[:n] for d in w.draft_list()], w.model_ids, w.tokens[:n], w.temps[:n], scheme, 9,
                       diag=True)
        torch.cuda.synchronize()
        assert v.status()[0] & ~mds.MDS_ST_OMEGA0 == 0
        return out

    want = call(B)
    for n in (1, 5, 64, 150, B):
        got = call(n)
        seen = torch.arange(3, device=DEV)[None] <= want[1][:n, None]
        assert torch.equal(got[0], want[0][:n]) and torch.equal(got[1], want[1][:n]), n
        assert torch.equal(got[2][seen], want[2][:n][seen]), n
    v.close()
