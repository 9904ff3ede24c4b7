"""Every wait of a cluster kernel for other blocks is bounded: with the limit at 0 the waits give up,
the blocks stop once nothing is on its way to them, the call reports it, and the next call is right."""
import numpy as np
import pytest

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


def _gives_up_then_runs(sg, monkeypatch, call, want):
    monkeypatch.setenv("SG_WAIT_LIMIT", "0")
    with pytest.raises(sg.SGError) as e:
        call()
    assert e.value.code == sg.SG_ETIMEOUT
    monkeypatch.delenv("SG_WAIT_LIMIT")
    for a, b in zip(call(), want):
        assert np.array_equal(a["E"], b["E"]) and np.array_equal(a["spins"], b["spins"])


# a second set of warps drawing, one pair a thread, two, columns; slabs of unequal height; 16 blocks
@pytest.mark.parametrize("L,C", [(4, 2), (16, 4), (18, 3), (34, 4), (22, 3), (32, 16)])
@pytest.mark.parametrize("general", [False, True])
def test_annealing(sg, monkeypatch, L, C, general):
    inst = sg.Instance.from_couplings(L, wl.random_couplings(3, L), e_gs=-1) if general else sg.Instance.create(L, 3)
    args = dict(replicas=40, sweeps=9, beta0=0.1, beta1=3.0, seed=5, spins="host")
    monkeypatch.setenv("SG_SA_CLUSTER", "0")
    want = sg.sa_run(inst, **args)
    monkeypatch.setenv("SG_SA_CLUSTER", "1")
    monkeypatch.setenv("SG_SA_CLUSTER_C", str(C))
    _gives_up_then_runs(sg, monkeypatch, lambda: [sg.sa_run(inst, **args)], [want])


# one word of slots and two; one block a word (which waits for the energies alone)
@pytest.mark.parametrize("L,C,K", [(4, 2, 32), (16, 4, 32), (18, 3, 32), (34, 4, 32), (32, 16, 32), (4, 1, 40), (16, 4, 40),
                                   (32, 8, 64)])
def test_tempering(sg, monkeypatch, L, C, K):
    insts = [sg.Instance.create(L, 8 + k) for k in range(2)]
    ps = [dict(temps=K, sweeps=9, beta_min=0.2, beta_max=3.0, seed=5, instance_id=k) for k in range(2)]
    monkeypatch.setenv("SG_PT_CLUSTER", "0")
    want = sg.pt_run_batch(insts, ps, spins="host")
    monkeypatch.setenv("SG_PT_CLUSTER", "1")
    monkeypatch.setenv("SG_PT_CLUSTER_C", str(C))
    _gives_up_then_runs(sg, monkeypatch, lambda: sg.pt_run_batch(insts, ps, spins="host"), want)


@pytest.mark.parametrize("n_small", [4, 200])
def test_batch_on_clusters(sg, monkeypatch, n_small):
    """After a give-up the persistent kernel passes over the planes that are left."""
    sides = [24, 20, 32] + [(4, 8, 12, 16)[k % 4] for k in range(n_small)]
    insts = [sg.Instance.create(L, 900 + k) for k, L in enumerate(sides)]
    ps = [dict(replicas=40, sweeps=(6, 11)[k % 2], beta0=0.1, beta1=3.0, schedule="linear", seed=2,
               instance_id=k) for k in range(len(sides))]
    monkeypatch.setenv("SG_BATCH_WG", "1")
    want = sg.sa_run_batch(insts, ps, spins="host")
    monkeypatch.setenv("SG_BATCH_WG", "0")
    _gives_up_then_runs(sg, monkeypatch, lambda: sg.sa_run_batch(insts, ps, spins="host"), want)


def test_trial_that_gives_up_is_not_chosen(sg, monkeypatch, tmp_path):
    """The batch's tuner times its forms; one whose waits gave up is no candidate, nor kept as one."""
    sides = [48] * 12 + [24, 40]
    insts = [sg.Instance.create(L, 400 + k) for k, L in enumerate(sides)]
    ps = [dict(replicas=64, sweeps=(40, 60)[k % 2], beta0=0.1, beta1=3.0, schedule="linear", seed=2, instance_id=k)
          for k in range(len(sides))]
    monkeypatch.setenv("SG_BATCH_WG", "1")
    want = sg.sa_run_batch(insts, ps, spins="host")
    monkeypatch.delenv("SG_BATCH_WG")
    monkeypatch.setenv("SG_AUTOTUNE_CACHE", str(tmp_path / "tune.json"))
    monkeypatch.setenv("SG_WAIT_LIMIT", "0")
    for a, b in zip(sg.sa_run_batch(insts, ps, spins="host"), want):
        assert np.array_equal(a["E"], b["E"]) and np.array_equal(a["spins"], b["spins"])


def test_served_chunks(sg, monkeypatch):
    """A chunk whose waits gave up ends its request; the server serves the next one."""
    reqs = [sg.request(sg.SG_REQ_SA, 32, 4, 32, 0.1, 3.0, 0.0, 40, sweeps_per_restart=40),
            sg.request(sg.SG_REQ_PT, 16, 4, 32, 0.2, 3.0, 0.0, 40)]
    monkeypatch.setenv("SG_SA_CLUSTER_C", "4")
    monkeypatch.setenv("SG_PT_CLUSTER_C", "4")
    with sg.Server(1 << 30, chunk_sweeps=20) as srv:
        want = [srv.poll(srv.submit(q)) for q in reqs]
        monkeypatch.setenv("SG_WAIT_LIMIT", "0")
        assert [srv.poll(srv.submit(q))["status"] for q in reqs] == [sg.SG_ETIMEOUT] * 2
        monkeypatch.delenv("SG_WAIT_LIMIT")
        got = [srv.poll(srv.submit(q)) for q in reqs]
    for a, b in zip(got, want):
        assert a["status"] == sg.SG_OK and a["minE"] == b["minE"] and a["sweeps"] == b["sweeps"]
