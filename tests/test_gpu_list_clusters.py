"""Rows whose large logits lie next to each other, as tokenizers that number
by frequency place them: the truncated alphabet's exact cut needs the largest
tokens of a slice wherever they lie in it (as many of them as a slice's list
holds, 16), so its status must stay 0.  Ties and heavier clusters beside, on
which the weighted scheme's stages fall back to full passes.  Against the
oracle; the comparison and its tolerances are those of the parity tests.
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


def clustered(V, dtype, near, B=4):
    """A workload whose 30 largest logits are the ids `near` and as many apart as that leaves."""
    spec = WorkloadSpec(f"v{V}", B=B, K=3, L=2, V=V, dtype=dtype, model_ids=[0, 0, 0], target_scale=2.0,
                        draft_sigma=[0.5], t_target=1.0, t_draft=[1.0], data_seed=V)
    w = make_workload(spec, device=DEV)
    far = [int((i + 0.5) * V / (30 - len(near))) for i in range(30 - len(near))]
    ids = torch.tensor(list(near) + far, device=DEV)
    step = torch.arange(30, device=DEV).float() * 0.25
    for t in (w.target, w.drafts):
        t[..., ids] = (14.0 + step.flip(0) + 0.3 * t[..., ids].float()).to(t.dtype)
    g = torch.Generator(device=DEV).manual_seed(V)
    pick = torch.randint(30, w.tokens.shape, generator=g, device=DEV)
    w.tokens.copy_(ids[pick].to(w.tokens.dtype))
    return w


def run(w, scheme, omega0=20):
    s = w.spec
    v = mds.Verifier(s.B, s.K, s.L, s.V, dtype=s.dtype, omega0=omega0)
    out, acc, diag = v.verify(w.target, w.draft_list(), w.model_ids, w.tokens, w.temps, scheme, 31, diag=True)
    torch.cuda.synchronize()
    bits, _ = v.status()
    v.close()
    o_out, o_acc, recs = oracle_verify(*host_copy(w), scheme, 31, omega0=omega0)
    res = compare(out.cpu().numpy(), acc.cpu().numpy(), o_out, o_acc, recs, g_diag=diag.cpu().numpy(), scheme=scheme)
    check(res, scheme)
    assert bits == 0, (scheme, bits)


NEAR = {
    "units": range(256, 508, 21),      # twelve units of one stretch of 256 ids
    "unit": range(1000, 1008),         # one 16-byte unit of 16-bit logits
    "lanes": range(2048, 2062),        # neighbours: two units
    "places": range(512, 740, 16),     # the same place of fifteen units
}


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("V", [32000, 128256])
@pytest.mark.parametrize("near", sorted(NEAR))
def test_large_logits_close_together(near, V, dtype):
    w = clustered(V, dtype, NEAR[near])
    for scheme in ("WIS", "WIS0"):
        run(w, scheme)


@pytest.mark.parametrize("B", [4, 300])
@pytest.mark.parametrize("dtype", ["bf16", "f32"])
def test_more_large_logits_than_a_slice_lists(dtype, B):
    """A descending head of ids and forty equal logits: the weighted scheme stays exact."""
    w = clustered(20000, dtype, range(0, 20), B)
    for t in (w.target, w.drafts):
        t[..., 4096:4352] += (torch.arange(256, device=DEV).flip(0) / 32.0).to(t.dtype)
        t[..., 9000:9160:4] = 9.0
    run(w, "WIS")
