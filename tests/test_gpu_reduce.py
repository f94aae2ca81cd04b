"""The reduction over path counts around its tile and CTA edges, against the oracle's estimates.

Synthetic records (moments of correlated per-path values) of batches whose
systems straddle the edges: 128-path CTAs, 32 CTAs per system, powers of two of
the sort, and the 16384-path limit of the sort in shared memory.  Sums run in
another order than numpy's: relative 1e-9 (differences of moments lose up to
1e4 of the 1e-16), 1e-7 for jackknife errors.
"""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1305_6758_gb300 as mp  # noqa: E402


def records(P, rng):
    e, m, mz = -1.0 + 0.05 * rng.standard_normal(P), 0.5 + 0.1 * rng.random(P), 0.3 * rng.standard_normal(P)
    r = np.zeros((P, mp.NREC))
    r[:, :13] = np.stack([e, e * e + 1e-3, m, m * m + 1e-3, m ** 4 + 1e-3, mz[::-1], e + m, mz, mz * mz + 1e-3, abs(mz),
                          e * m + 1e-4, e * mz, m * mz], 1)
    r[:, 17], r[:, 18] = rng.random(P), 1e-7 * rng.random(P)
    return r


@pytest.mark.parametrize("counts", [(1, 2, 3, 5), (127, 128, 129), (4095, 4096, 4097), (16383, 16384, 8191),
                                    (16385, 3, 40000), (32768, 65537)])
def test_estimates_at_path_count_edges(counts):
    rng = np.random.default_rng(sum(counts))
    recs = [records(P, rng) for P in counts]
    systems = [mp.System(8, 1.0 + 0.1 * k, n_paths=P) for k, P in enumerate(counts)]
    got = mp.reduce_records(systems, 3, 4, torch.from_numpy(np.concatenate(recs)).cuda())
    for s, r, g in zip(systems, recs, got):
        ref = O.estimates(r, s.N, s.T)
        for k, v in ref.items():
            if np.isnan(v):
                assert np.isnan(g[k]), (s.n_paths, k)
            elif not (s.n_paths < 3 and k.startswith("r_")):
                tol = 1e-7 if k.endswith("_se") or k == "start_z" else 1e-9
                assert g[k] == pytest.approx(v, rel=tol, abs=1e-10), (s.n_paths, k)
        assert g["norm_max"] == r[:, 18].max()
