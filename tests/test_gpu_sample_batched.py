"""The batched sampler (two products per site for all samples) draws what the oracle's sampler draws."""
import numpy as np
import pytest

from oracle import gbs
from oracle import observables as oobs
from paper_2410_18740_gb300 import inputs

pytestmark = pytest.mark.gpu


# (M, D, d, chi, samples): local basis and Fock basis, more samples than SMs, ragged bonds at the ends
@pytest.mark.parametrize("M,D,d,chi,ns", [(7, 11, 5, 70, 37), (6, 6, 6, 96, 200), (5, 24, 6, 36, 400)])
def test_batched_draws_match_the_oracle(ctx, M, D, d, chi, ns):
    from paper_2410_18740_gb300 import vtn
    w = inputs.workload("large", 17 + M, M=M, D=D, d=d)
    m = vtn.vtn_build_mpo(ctx, w.r, w.U, D, d)
    rng = np.random.default_rng(M)
    dims = [min(chi, d ** s, d ** (M - s)) for s in range(M + 1)]
    sites = [(rng.standard_normal((dims[s], d, dims[s + 1])) + 1j * rng.standard_normal((dims[s], d, dims[s + 1])))
             / np.sqrt(2 * d * dims[s + 1]) for s in range(M)]
    mps = vtn.vtn_mps_from_host(ctx, m, sites)
    got = vtn.vtn_sample(ctx, m, mps, seed=77, n_samples=ns)
    isos = None
    if d != D:
        S_list, _, _ = gbs.lbo_transform(w.r, w.U)
        isos = [gbs.lbo_isometry(S, D, d) for S in S_list]
    assert np.array_equal(got, oobs.sample(sites, isos, seed=77, n_samples=ns))
    vtn.vtn_mps_free(mps)
    vtn.vtn_mpo_free(m)
