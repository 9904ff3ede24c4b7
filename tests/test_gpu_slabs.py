"""Lattices held in the shared memory of thread-block clusters, against the row kernels, bit
for bit: every cluster size at the edges of the block forms (one pair of sites a thread, two
pairs, columns), sides whose columns do not fill a warp, slabs of one plane, and schedules
through all three ways a sweep's thresholds can decide."""
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


# (L, C): pairs a block = L^3 / 2C, up to 512 one a thread, up to 1024 two, else columns
SLABS = [(2, 1), (2, 2), (4, 1), (4, 4), (6, 3), (8, 1), (8, 8), (10, 1), (10, 5), (12, 1), (12, 6), (14, 1), (14, 7),
         (16, 2), (16, 4), (18, 3), (20, 2), (22, 2), (24, 8), (26, 2), (34, 2), (48, 6), (50, 5)]
BETAS = [(0.1, 3.0, "linear"), (0.5, 30.0, "geometric"), (20.0, 0.1, "linear")]


@pytest.mark.parametrize("L,C", SLABS)
def test_annealing_on_clusters_equals_row_kernel(sg, monkeypatch, L, C):
    R, S = (40, 12) if L <= 26 else (5, 7)
    inst = sg.Instance.create(L, 300 + L)
    for k, (b0, b1, schedule) in enumerate(BETAS):
        args = dict(replicas=R, sweeps=S, beta0=b0, beta1=b1, schedule=schedule, seed=11 + k, instance_id=3, spins="host")
        monkeypatch.setenv("SG_SA_CLUSTER", "1")
        monkeypatch.setenv("SG_SA_CLUSTER_C", str(C))
        a = sg.sa_run(inst, **args)
        monkeypatch.delenv("SG_SA_CLUSTER_C")
        monkeypatch.setenv("SG_SA_CLUSTER", "0")
        b = sg.sa_run(inst, **args)
        assert np.array_equal(a["spins"], b["spins"]) and np.array_equal(a["E"], b["E"])


@pytest.mark.parametrize("L,C", SLABS + [(60, 6), (64, 8)])
def test_tempering_on_clusters_equals_row_kernels(sg, monkeypatch, L, C):
    K, S = (32, 9) if L > 26 else (13 if L % 4 else 32, 20)
    insts = [sg.Instance.create(L, 500 + 10 * L + k) for k in range(2 if L <= 26 else 1)]
    ps = [dict(temps=K, sweeps=S, beta_min=0.2, beta_max=3.0, seed=5, instance_id=k) for k in range(len(insts))]
    monkeypatch.setenv("SG_PT_CLUSTER", "1")
    monkeypatch.setenv("SG_PT_CLUSTER_C", str(C))
    a = sg.pt_run_batch(insts, ps, spins="host")
    monkeypatch.delenv("SG_PT_CLUSTER_C")
    monkeypatch.setenv("SG_PT_CLUSTER", "0")
    b = sg.pt_run_batch(insts, ps, spins="host")
    for x, y in zip(a, b):
        for key in ("spins", "E", "perm", "accepts"):
            assert np.array_equal(x[key], y[key]), key
        assert x["minE"] == y["minE"]


# C that does not divide L: slabs differ by a plane
@pytest.mark.parametrize("L,C", [(4, 3), (6, 4), (8, 5), (10, 7), (14, 4), (18, 5), (22, 3), (26, 8), (34, 7), (50, 7)])
def test_slabs_of_unequal_height(sg, monkeypatch, L, C):
    test_annealing_on_clusters_equals_row_kernel(sg, monkeypatch, L, C)
    test_tempering_on_clusters_equals_row_kernels(sg, monkeypatch, L, C)


# more blocks than a portable cluster has
@pytest.mark.parametrize("L,C", [(16, 16), (24, 12), (26, 13), (32, 11), (32, 16), (50, 10)])
def test_clusters_of_more_than_eight_blocks(sg, monkeypatch, L, C):
    test_annealing_on_clusters_equals_row_kernel(sg, monkeypatch, L, C)
    test_tempering_on_clusters_equals_row_kernels(sg, monkeypatch, L, C)


# two words of slots, each on C blocks of the cluster: word edges, every block form, C = 1
@pytest.mark.parametrize("L,C,K", [(4, 1, 33), (8, 1, 64), (8, 4, 40), (10, 3, 63), (16, 4, 48), (16, 2, 33), (22, 7, 64),
                                   (32, 8, 48), (40, 8, 50)])
def test_tempering_with_two_words_of_slots(sg, monkeypatch, L, C, K):
    S = 20 if L <= 26 else 7
    insts = [sg.Instance.create(L, 500 + 10 * L + k) for k in range(2)]
    ps = [dict(temps=K, sweeps=S, beta_min=0.2, beta_max=3.0, seed=5, instance_id=k) for k in range(2)]
    monkeypatch.setenv("SG_PT_CLUSTER", "1")
    monkeypatch.setenv("SG_PT_CLUSTER_C", str(C))
    a = sg.pt_run_batch(insts, ps, spins="host")
    monkeypatch.delenv("SG_PT_CLUSTER_C")
    monkeypatch.setenv("SG_PT_CLUSTER", "0")
    b = sg.pt_run_batch(insts, ps, spins="host")
    for x, y in zip(a, b):
        for key in ("spins", "E", "perm", "accepts"):
            assert np.array_equal(x[key], y[key]), key
        assert x["minE"] == y["minE"]


def test_batch_whose_sides_share_no_divisor(sg, monkeypatch, tmp_path):
    sides = [22, 40, 44, 10, 26]
    insts = [sg.Instance.create(L, 700 + k) for k, L in enumerate(sides)]
    ps = [dict(replicas=40, sweeps=(6, 11)[k % 2], beta0=0.1, beta1=3.0, schedule="linear", seed=2, instance_id=k)
          for k in range(len(sides))]
    monkeypatch.setenv("SG_AUTOTUNE_CACHE", str(tmp_path / "tune.json"))
    runs = []
    for wg in ("0", "1"):  # clusters; planes of one word, a block each
        monkeypatch.setenv("SG_BATCH_WG", wg)
        runs.append(sg.sa_run_batch(insts, ps, spins="host"))
    for x, y in zip(*runs):
        assert np.array_equal(x["spins"], y["spins"]) and np.array_equal(x["E"], y["E"])


@pytest.mark.parametrize("n_small", [40, 200])
def test_batch_of_small_lattices_on_clusters_and_single_blocks(sg, monkeypatch, tmp_path, n_small):
    """Few small planes are annealed by whole clusters, enough of them by single blocks."""
    sides = [24, 20] + [(4, 8, 12, 16)[k % 4] for k in range(n_small)]
    insts = [sg.Instance.create(L, 900 + k) for k, L in enumerate(sides)]
    ps = [dict(replicas=40, sweeps=(6, 11)[k % 2], beta0=0.1, beta1=3.0, schedule="linear", seed=2, instance_id=k)
          for k in range(len(sides))]
    monkeypatch.setenv("SG_AUTOTUNE_CACHE", str(tmp_path / "tune.json"))
    runs = []
    for wg in ("0", "1"):  # clusters; planes of one word, a block each
        monkeypatch.setenv("SG_BATCH_WG", wg)
        runs.append(sg.sa_run_batch(insts, ps, spins="host"))
    for x, y in zip(*runs):
        assert np.array_equal(x["spins"], y["spins"]) and np.array_equal(x["E"], y["E"])


def test_loaded_server_equals_requests_one_at_a_time(sg):
    """With many requests in service chunks run on clusters of any size, alone through the row
    kernels: both kinds, one and two words, restarts shorter than the cap, a chunk that does not
    divide them."""
    reqs = [sg.request(kind, L, 40 + 7 * L + k, 40 if kind == sg.SG_REQ_SA and k % 2 else 32, 0.1 + 0.1 * kind, 3.0, 0.002,
                       70, run_seed=k, sweeps_per_restart=50)
            for k, L in enumerate((24, 32, 40, 20, 64, 48) * 4) for kind in (sg.SG_REQ_SA, sg.SG_REQ_PT)]
    results = []
    for active in (64, 1):
        with sg.Server(4 << 30, max_active=active, chunk_sweeps=15) as srv:
            tickets = [srv.submit(q) for q in reqs]
            results.append([srv.poll(t) for t in tickets])
    for a, b in zip(*results):
        for key in ("status", "reached", "sweeps", "minE", "e_gs"):
            assert a[key] == b[key], key
        assert a["status"] == sg.SG_OK


@pytest.mark.parametrize("L,probs,gauge", [(2, wl.UNIFORM, True), (4, (0, 0, 1), False), (6, (0.3, 0.7, 0), True),
                                           (12, (1, 0, 0), True), (40, wl.UNIFORM, True)])
def test_server_generates_the_host_generators_instance(sg, L, probs, gauge):
    """E_gs and the lowest energies of requests, whose instances are made on the device, against
    runs of the instances that the host generator makes."""
    reqs = [sg.request(kind, L, 2 ** 33 + 17 * L, 32, 0.3, 3.0, 0.0, 20, run_seed=9, sweeps_per_restart=20,
                       class_prob=probs, gauge=gauge) for kind in (sg.SG_REQ_SA, sg.SG_REQ_PT)]
    with sg.Server(1 << 30, max_active=4, chunk_sweeps=20) as srv:
        tickets = [srv.submit(q) for q in reqs]
        sa, pt = [srv.poll(t) for t in tickets]
    inst = sg.Instance.create(L, 2 ** 33 + 17 * L, probs, gauge)
    assert sa["e_gs"] == pt["e_gs"] == inst.e_gs
    assert sa["minE"] == sg.sa_run(inst, 32, 20, 0.3, 3.0, seed=9)["E"].min()
    assert pt["minE"] == sg.pt_run(inst, 32, 20, 0.3, 3.0, seed=9)["minE"]
