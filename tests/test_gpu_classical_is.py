"""Classical importance sampling at the edges of its binned law: the ratios
q/p in one window of bins, over several, over more bins than the residual's
table holds (direct sums), masked tokens (q = 0 or p = 0), several models and
cluster sizes, and coarse quadrature steps.  Tokens, p_I(Y) and the residual
mass of every visited depth against the oracle.

Residual mass: a probability 2^a is off by 2^-24 |a| ln 2 (the scale
log2(e) / T and the argument are rounded to 24 bits), so |d(q - p_I)| <=
1e-7 |a| (q + p_I) / 2 and the sum by at most 1e-7 |a|: 1e-5 for |a| <= 100,
3e-5 for the widest rows, whose |a| reaches 240.
"""
import numpy as np
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
# name: target scale, draft noise, draft temperature, models, V, dtype
SPREADS = {
    "one-window": (2.0, 0.05, 1.0, 1, 2048, "bf16"),
    "equal-rows": (3.0, 0.0, 1.0, 1, 1031, "f32"),
    "several-windows": (4.0, 3.0, 1.0, 1, 3001, "bf16"),
    "two-models": (4.0, 1.5, 2.0, 2, 2500, "f32"),
    "past-the-table": (14.0, 10.0, 0.6, 3, 1500, "f32"),
}


def run(spec, cluster, is_h, mask=0, tol=1e-5):
    w = make_workload(spec, device=DEV)
    if mask:
        # tokens neither side can draw, and tokens only the drafts can
        ids = torch.arange(spec.V, device=DEV)
        free = torch.ones(spec.V, dtype=torch.bool, device=DEV)
        free[w.tokens.reshape(-1).long()] = False
        w.target[..., free & (ids % mask == 1)] = float("-inf")
        w.drafts[..., free & (ids % (2 * mask) == 1)] = float("-inf")
    v = mds.Verifier(spec.B, spec.K, spec.L, spec.V, dtype=spec.dtype, cluster=cluster, is_h=is_h, acc_prob=1)
    out, acc, diag = v.verify(w.target, w.draft_list(), w.model_ids, w.tokens, w.temps, "IS", 21, diag=True)
    torch.cuda.synchronize()
    bits, _ = v.status()
    v.close()
    o_out, o_acc, recs = oracle_verify(*host_copy(w), "IS", 21, is_h=is_h)
    d = diag.cpu().numpy()
    res = compare(out.cpu().numpy(), acc.cpu().numpy(), o_out, o_acc, recs, g_diag=d, scheme="IS")
    check(res, "IS")
    assert bits == 0
    for b, rr in recs.items():
        for r in rr:
            if r.j == spec.L:
                break
            assert abs(d[b, r.j, 2] - r.R) <= tol, (b, r.j, d[b, r.j, 2], r.R)
            if r.band:
                break


def spec_of(name, B=6, K=3, L=2):
    scale, sigma, td, models, V, dtype = SPREADS[name]
    return WorkloadSpec(name, B=B, K=K, L=L, V=V, dtype=dtype, model_ids=[k % models for k in range(K)],
                        target_scale=scale, draft_sigma=[sigma, 0.5 * sigma, 1.5 * sigma][:models],
                        t_target=1.0, t_draft=[td, 1.0, 1.4][:models], data_seed=5)


@pytest.mark.parametrize("cluster", [0, 1, 4])
@pytest.mark.parametrize("name", sorted(SPREADS))
def test_ratio_spreads(name, cluster):
    run(spec_of(name), cluster, 0.25, tol=3e-5 if name == "past-the-table" else 1e-5)


@pytest.mark.parametrize("is_h", [0.1, 1.0])
def test_quadrature_steps(is_h):
    run(spec_of("two-models"), 0, is_h)


def test_masked_tokens():
    run(spec_of("one-window", K=2), 0, 0.25, mask=7)
