"""The FP64 assembly spread over CTAs (csrc/occri_api.cu, ace_factor_kernel and ace_k_kernel) at
its edges: one share of the Gram matrix or several, AO counts around the tiles of 16 and 32, the
smallest and largest nocc, E_x over several k, and the failure of one k. K and E_x against
numpy on the build's own K_{mu i}."""
import numpy as np
import pytest

from workloads import small_workload

pytestmark = pytest.mark.gpu

CASES = [
    dict(mesh=(1, 1, 1), counts=(2, 1), nocc=1),              # nao 10: one tile of 16
    dict(mesh=(1, 1, 1), counts=(5, 1), nocc=7),              # nao 16: a whole tile
    dict(mesh=(1, 2, 1), counts=(4, 3, 1, 1), nocc=5),        # nao 50: ragged tiles of 16
    dict(mesh=(3, 3, 3), counts=(4, 3, 1, 1), nocc=3),        # 81 tiles of 32 a k
    dict(mesh=(1, 1, 2), counts=(6, 4, 2, 2), nocc=32),       # nao 84: 21 shares wanted, 16 taken
]


@pytest.mark.parametrize("case", range(len(CASES)))
@pytest.mark.parametrize("want_k", [True, False])
def test_k_and_ex_from_kc(case, want_k):
    import torch
    import paper_2207_09028_gb300 as occri
    w = small_workload(grid=(12, 12, 12), lo=0.2, hi=8.0, seed=60 + case, **CASES[case])
    plan = occri.Plan.from_workload(w, precision="fp64")
    C = torch.from_numpy(w.C).cuda()
    KC, K, Ex = plan.build(C, want_k=want_k)
    kc = KC.cpu().numpy()
    m = np.conj(np.swapaxes(w.C, 1, 2)) @ kc
    ex = np.trace(m, axis1=1, axis2=2).real.sum() / w.nk
    # FP64 sums of at most nao nocc nk = 2,700 products, each rounded at 1.1e-16 of its size
    assert abs(float(Ex.cpu()[0]) - ex) <= 1e-12 * np.abs(m).max() * w.nocc
    if not want_k:
        assert K is None
        return
    k = K.cpu().numpy()
    assert np.array_equal(k, np.conj(np.swapaxes(k, 1, 2)))   # the tiles below are copies
    m = 0.5 * (m + np.conj(np.swapaxes(m, 1, 2)))
    ref = kc @ np.linalg.solve(m, np.conj(np.swapaxes(kc, 1, 2)))
    # the solve carries the condition of M: a few times cond(M) 1.1e-16
    bar = 1e-13 + 20 * 1.1e-16 * max(np.linalg.cond(x) for x in m)
    assert np.abs(k - ref).max() <= bar * np.abs(ref).max()


def test_failure_of_one_k_leaves_the_others():
    import torch
    import paper_2207_09028_gb300 as occri
    w = small_workload(mesh=(1, 1, 3), grid=(8, 8, 8), counts=(2, 1), nocc=2, seed=71)
    plan = occri.Plan.from_workload(w, precision="fp64")
    good = plan.build(torch.from_numpy(w.C).cuda())[1]
    bad = w.C.copy()
    bad[1, :, 1] = bad[1, :, 0]   # a repeated orbital: M of k = 1 is singular
    with pytest.raises(occri.OccriError) as e:
        plan.build(torch.from_numpy(bad).cuda())
    assert e.value.status == occri.OCCRI_ENOTPD and e.value.bad_k == 1
    # the counters are back at zero: the next build is the first one again
    assert torch.equal(plan.build(torch.from_numpy(w.C).cuda())[1], good)
