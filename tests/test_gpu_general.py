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


# (L, C): one pair a thread and several, slabs of one plane, of unequal height, a block alone
@pytest.mark.parametrize("L,C", [(2, 1), (2, 2), (4, 3), (6, 1), (10, 5), (12, 12), (16, 2), (16, 16), (22, 4), (24, 7),
                                 (32, 2)])
def test_general_couplings_on_clusters_equal_row_kernel(sg, monkeypatch, L, C):
    for kind, n, (b0, b1, schedule) in [("mixed", 40, (0.1, 3.0, "linear")), ("double", 3, (0.5, 30.0, "geometric")),
                                        ("sparse", 65, (20.0, 0.1, "linear"))]:
        inst = sg.Instance.from_couplings(L, _couplings(L, kind), e_gs=-1)
        args = dict(replicas=n, sweeps=9, beta0=b0, beta1=b1, schedule=schedule, seed=5, instance_id=2, spins="host")
        monkeypatch.setenv("SG_SA_CLUSTER", "1")
        monkeypatch.setenv("SG_SA_CLUSTER_C", str(C))
        a = sg.sa_run(inst, **args)
        monkeypatch.delenv("SG_SA_CLUSTER_C")
        monkeypatch.setenv("SG_SA_CLUSTER", "0")
        b = sg.sa_run(inst, **args)
        assert np.array_equal(a["spins"], b["spins"]) and np.array_equal(a["E"], b["E"])
