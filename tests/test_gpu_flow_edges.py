"""Edges of the slice-dataflow engine's warp-wise passes against the oracle:
vocabularies around the slice lengths (a ragged last unit, last warp, last
slice), rows at every 16-byte offset (odd lengths), rows of ties (more tokens
at a warp's threshold than it may set aside, so the bound is raised), flat
rows, rows with a few finite logits, long lists (Omega_0 of 62).

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


def spec_of(V, dtype, B=8, K=3, L=3, models=1):
    return WorkloadSpec(f"v{V}", B=B, K=K, L=L, V=V, dtype=dtype, model_ids=[k % models for k in range(K)],
                        target_scale=4.0, draft_sigma=[0.8, 1.2][:models], t_target=0.8, t_draft=[0.8, 1.1][:models],
                        data_seed=V)


def run(w, scheme, omega0=20, uncertified=False):
    """One call against the oracle.  `uncertified`: the list cannot certify the
    cut of Omega_0 (ties at it), which the status must say; the walk is then
    another than the exact cut's, and what holds for every cut is checked."""
    s = w.spec
    v = mds.Verifier(s.B, s.K, s.L, s.V, dtype=s.dtype, omega0=omega0)
    out, acc, diag = v.verify(w.target, w.draft_list(), w.model_ids, w.tokens, w.temps, scheme, 31, diag=True)
    torch.cuda.synchronize()
    bits, _ = v.status()
    v.close()
    o_out, o_acc, recs = oracle_verify(*host_copy(w), scheme, 31, omega0=omega0)
    res = compare(out.cpu().numpy(), acc.cpu().numpy(), o_out, o_acc, recs, g_diag=diag.cpu().numpy(), scheme=scheme)
    if uncertified:
        assert bits == mds.MDS_ST_OMEGA0
        a = acc.cpu()
        assert bool(((a >= 0) & (a <= s.L)).all())
        for b in range(s.B):
            n = int(a[b])
            assert bool(((out[b, :n + 1] >= 0) & (out[b, :n + 1] < s.V)).all()) and bool((out[b, n + 1:] == -1).all())
            d = diag[b, :n + 1, :3]
            assert bool(torch.isfinite(d).all()) and bool((d >= 0).all()) and bool((d <= 1 + 1e-5).all())
        return
    check(res, scheme)
    assert bits == 0


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("V", [2047, 2048, 2049, 4096, 8191, 8200, 16385, 20000, 33003])
def test_slice_edges(V, dtype):
    w = make_workload(spec_of(V, dtype, models=2 if V % 2 == 0 else 1), device=DEV)
    for scheme in ("single", "WIS", "WIS0"):
        run(w, scheme)


@pytest.mark.parametrize("V", [8192, 20000])
def test_long_lists(V):
    w = make_workload(spec_of(V, "f32"), device=DEV)
    run(w, "WIS0", omega0=mds.MDS_MAX_OMEGA0)


@pytest.mark.parametrize("kind", ["integers", "two-values", "flat", "few-finite"])
def test_ties_and_flat_rows(kind):
    spec = spec_of(9000, "bf16", B=4, K=2, L=2)
    w = make_workload(spec, device=DEV)
    for t in (w.target, w.drafts):
        if kind == "integers":
            t.copy_(t.float().round())
        elif kind == "two-values":
            t.copy_((t.float() > 6.0).float() * 3.0)
        elif kind == "flat":
            t.fill_(1.5)
        else:
            keep = torch.zeros(spec.V, dtype=torch.bool, device=DEV)
            keep[w.tokens.reshape(-1).long()] = True
            keep[[5, 4099, 8999]] = True
            t.masked_fill_(~keep, float("-inf"))
    for scheme in ("single", "WIS"):
        run(w, scheme)
    run(w, "WIS0", uncertified=kind == "flat")


def test_large_noalloc_batch_fits_the_scratch():
    """Slice records with 64 run masses (T = 16384) at a batch near the scratch's end."""
    B, V = 2300, 131072
    g = torch.Generator(device=DEV).manual_seed(5)
    target = torch.randn(B, 1, 2, V, generator=g, device=DEV, dtype=torch.bfloat16)
    draft = torch.randn(B, 1, V, generator=g, device=DEV, dtype=torch.bfloat16)
    tok = torch.randint(V, (B, 1, 1), generator=g, device=DEV, dtype=torch.int32)
    temps = torch.ones(B, 2, device=DEV)
    res = []
    v = mds.Verifier(B, 1, 1, V, omega0=20)
    o, a, _ = v.verify(target, [draft], [0], tok, temps, "WIS0", 9)
    res.append((o.clone(), a.clone()))
    v.close()
    o, a = torch.empty_like(o), torch.empty_like(a)
    mds.mds_verify_noalloc(B, 1, 1, V, target, [draft], [0], tok, temps, "WIS0", 9, o, a, omega0=20)
    torch.cuda.synchronize()
    assert torch.equal(o, res[0][0]) and torch.equal(a, res[0][1])
