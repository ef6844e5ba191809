"""Ensembles in free-running passes share their CTAs out among the instances by
pass length: every CTA count, from fewer CTAs than pass lengths to more
processing elements than tiles, advances every tile, and later calls of the
modes that share out evenly continue exactly."""
import pytest

from gpu_util import gpu_ensemble_run
from test_gpu_ensemble import check_against_oracle, small_ensemble

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K", [1, 4])
@pytest.mark.parametrize("max_ctas", [1, 2, 3, 5, 0])
@pytest.mark.parametrize("bounds", [(1, 2, 3), (3, 3, 1), (2, 2, 2), (0, 1, 3)])
def test_shared_out_passes_replay_in_the_oracle(bounds, max_ctas, K):
    from paper_1911_05769_gb300 import AT_FREE
    M = 256
    inst = small_ensemble(n_inst=6, seed=91, M=M)
    for j, d in enumerate(inst):
        d["L"] = bounds[j % 3]
    steps = 90
    res = gpu_ensemble_run(inst, M=M, order=2, steps=steps, dtype="f64", mode=AT_FREE, record=True,
                           max_ctas=max_ctas, steps_per_pass=max(bounds) + 1, tile_subdomains=K, calls=[31, 59])
    rec = res["rec"]
    p0 = 0
    for d in inst:
        Pj = d["n"] // M
        r = rec[:, p0:p0 + Pj, :]
        assert r.min() >= 0 and r.max() <= d["L"]
        p0 += Pj
    check_against_oracle(inst, res, M=M, order=2, steps=steps, mode="replay", dtype="f64", delays=rec)
