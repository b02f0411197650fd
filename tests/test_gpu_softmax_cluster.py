"""Whole softmax rows of the per-sequence engine against the oracle: the row
statistics it exports at every depth a walk visits, evaluated at every token
of the row as the kernel does, to the tolerance of test_gpu_softmax.  Single
draft calls take this engine in production; a set cluster size keeps them
there while the export is on.
"""
import math

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2410_18234_gb300 import mds  # noqa: E402
from synth import WORKLOADS, make_workload  # noqa: E402
from oracle.verify import softmax_t  # noqa: E402

RTOL = 1e-5          # the fp32 kernel against the fp64 oracle
FLOOR = 1e-30        # below fp32's normal range the kernel's exponent is 0


@pytest.mark.parametrize("cluster", [1, 4])
@pytest.mark.parametrize("name,kw", [("serving-152k", dict(B=4, K=2, L=2, model_ids=[0, 0], temp_per_seq=None,
                                                           t_target=0.5, t_draft=[0.5])),
                                     ("two-models-50k", dict(B=4, K=3, L=2, V=10007, dtype="f32", model_ids=[0, 1, 2],
                                                             draft_sigma=[0.5, 1.0, 1.5], t_target=0.5,
                                                             t_draft=[2.0, 1.0, 0.7]))])
def test_softmax_rows_match_oracle(name, kw, cluster):
    spec = WORKLOADS[name].with_(**kw)
    w = make_workload(spec, device="cuda:0")
    v = mds.Verifier(spec.B, spec.K, spec.L, spec.V, dtype=spec.dtype, omega0=20, cluster=cluster)
    stats = torch.empty(spec.B, spec.L + 1, mds.DEBUG_ROWS, 4, dtype=torch.float32, device="cuda:0")
    mds.mds_debug_row_stats(v.ctx, stats)
    out = torch.empty(spec.V, dtype=torch.float32, device="cuda:0")
    for scheme in ("single", "SpecTr", "WIS", "WIS0"):
        stats.fill_(float("nan"))
        _, acc, _ = v.verify(w.target, w.draft_list(), w.model_ids, w.tokens, w.temps, scheme, spec.verify_seed)
        torch.cuda.synchronize()
        assert v.cluster_size == cluster
        st = stats.cpu().numpy()
        for b in range(spec.B):
            for j in range(spec.L + 1):
                written = [r for r in range(mds.DEBUG_ROWS) if not math.isnan(st[b, j, r, 3])]
                # every visited depth, the target's row first, and nothing beyond
                assert (0 in written) == (j <= int(acc[b])), (scheme, b, j)
                if scheme == "WIS0" or j == spec.L:
                    assert written in ([], [0]), (scheme, b, j, written)
                for r in written:
                    M, iz, c, src = (float(x) for x in st[b, j, r])
                    row, T = ((w.target[b, int(src), j], float(w.temps[b, 0])) if src < 100 else
                              (w.drafts[int(src) - 100][b, j], float(w.temps[b, 1 + int(src) - 100])))
                    assert c == pytest.approx(math.log2(math.e) / T, rel=1e-6)
                    assert M == float(row.float().max())
                    mds.mds_debug_probs(row.contiguous(), M, iz, c, out)
                    torch.cuda.synchronize()
                    g = out.cpu().numpy().astype(np.float64)
                    o = softmax_t(row.float().cpu().numpy(), T)
                    big = o >= FLOOR
                    rel = np.abs(g[big] - o[big]) / o[big]
                    assert rel.max() <= RTOL, (scheme, b, j, r, float(rel.max()))
                    assert np.all(np.abs(g[~big] - o[~big]) <= FLOOR)
    mds.mds_debug_row_stats(v.ctx, None)
    assert v.status()[0] == 0
    v.close()


@pytest.mark.parametrize("V,cluster,scale", [(4096, 16, 3.0), (32003, 8, 4.0)])
def test_normaliser_error(V, cluster, scale):
    """1/Z against 64 bits over 640 rows: as near as the dataflow engine's on
    the same rows (root mean squares within 15%; both are a few tenths of a
    unit in the last place, set by the last few additions)."""
    rms = {}
    for cl in (0, cluster):
        err = []
        for seed in range(20):
            g = torch.Generator(device="cuda:0").manual_seed(seed)
            target = torch.randn(16, 1, 2, V, generator=g, device="cuda:0") * scale
            draft = target[:, 0, :1] + torch.randn(16, 1, V, generator=g, device="cuda:0")
            tokens = torch.randint(V, (16, 1, 1), generator=g, device="cuda:0", dtype=torch.int32)
            v = mds.Verifier(16, 1, 1, V, dtype="f32", cluster=cl)
            stats = torch.empty(16, 2, mds.DEBUG_ROWS, 4, device="cuda:0")
            mds.mds_debug_row_stats(v.ctx, stats)
            v.verify(target, [draft], [0], tokens, torch.ones(16, 2, device="cuda:0"), "single", 1)
            torch.cuda.synchronize()
            assert v.cluster_size == cl
            v.close()
            st = stats.double().cpu().numpy()
            for r, rows in ((0, target[:, 0, 0]), (1, draft[:, 0])):
                want = torch.softmax(rows.double(), 1).amax(1).cpu().numpy()
                mc = st[:, 0, r, 0] * st[:, 0, r, 2]   # the largest token's exponent is mc - round(mc)
                got = st[:, 0, r, 1] * np.exp2(mc - mc.astype(np.float32).astype(np.float64))
                err.append(got / want - 1.0)
        rms[cl] = float(np.sqrt(np.mean(np.square(err))))
    assert rms[cluster] <= 1.15 * rms[0], rms
