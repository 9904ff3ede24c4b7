"""Couplings that are not all +-1, against the oracle bit for bit: bonds of weight 0, 1 and 2
in every mixture (odd and even total weights, sites without a bond), word edges, thresholds
that are all zero, and every kernel that takes such lattices."""
import numpy as np
import pytest

from oracle import oracle as o
from paper_2501_17267_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sg():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    torch.cuda.init()
    from paper_2501_17267_gb300 import sg
    return sg


def _couplings(L, kind):
    J3 = wl.random_couplings(31 + L, L, jmax=2, allow_zero=True)
    if kind == "double":
        J3 = np.where(J3 < 0, -2, 2)
    elif kind == "sparse":
        J3 = np.where(np.arange(J3.size).reshape(J3.shape) % 3 == 0, J3, 0)
    return np.ascontiguousarray(J3.astype(np.int8))


@pytest.mark.parametrize("kind", ["mixed", "double", "sparse"])
@pytest.mark.parametrize("L,n", [(2, 3), (4, 33), (6, 64), (10, 100), (12, 256)])
def test_general_couplings_match_oracle(sg, L, n, kind):
    J3 = _couplings(L, kind)
    inst = sg.Instance.from_couplings(L, J3, e_gs=-1)
    reps = sorted({0, 1, n // 2, n - 1})
    for b0, b1 in [(0.05, 1.5), (1.0, 40.0)]:
        args = dict(replicas=n, sweeps=9, beta0=b0, beta1=b1, schedule="linear", seed=5, instance_id=2)
        spins, E = o.sa_run(L, J3, 5, 2, 9, b0, b1, False, reps=reps)
        one = sg.sa_run(inst, spins="host", **args)
        other = dict(args, sweeps=4, instance_id=3)  # unequal members: the plane kernel
        two = sg.sa_run_batch([inst, inst], [args, other], spins="host")
        for got in (one, two[0]):
            assert np.array_equal(got["spins"][reps], spins) and np.array_equal(got["E"][reps], E)
    K = min(n, 256)
    res = sg.pt_run(inst, K, 7, 0.05, 2.0, seed=7, instance_id=2, spins="host")
    ref = o.pt_run(L, J3, 7, 2, K, 7, 0.05, 2.0)
    for k in ("spins", "E", "perm", "accepts"):
        assert np.array_equal(res[k], ref[k]), k
    assert res["minE"] == ref["minE"]
