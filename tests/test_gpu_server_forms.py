"""The forms a server's chunks take, and its host side."""
import os
import subprocess
import sys
import threading
import time

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def sg():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    torch.cuda.init()
    from paper_2501_17267_gb300 import sg
    return sg


def _one(sg, req, chunk):
    with sg.Server(4 << 30, chunk_sweeps=chunk) as srv:
        return srv.poll(srv.submit(req))


# Items a lane of a block with so many threads sums in its nine-bit counters: 175, 128, 85 and 42.
@pytest.mark.parametrize("L,C,threads", [(56, 8, 64), (64, 8, 128), (34, 1, 256), (64, 8, 512)])
def test_chunk_energies_with_any_number_of_threads(sg, monkeypatch, L, C, threads):
    """A chunk on clusters reports the lowest energy sg_sa_run gives, however many items a thread
    of its blocks has: of a hot lattice (about half the bonds satisfied) and of a cold one."""
    for beta in (0.01, 3.0):
        req = sg.request(sg.SG_REQ_SA, L, 60 + L, 32, 0.01, beta, 0.0, 12, run_seed=5, sweeps_per_restart=12)
        want = sg.sa_run(sg.Instance.create(L, 60 + L), 32, 12, 0.01, beta, seed=5)["E"].min()
        monkeypatch.setenv("SG_SA_CLUSTER_C", str(C))
        monkeypatch.setenv("SG_SA_CLUSTER_THREADS", str(threads))
        got = _one(sg, req, 12)
        monkeypatch.delenv("SG_SA_CLUSTER_C")
        monkeypatch.delenv("SG_SA_CLUSTER_THREADS")
        assert got["status"] == sg.SG_OK and got["minE"] == want


# the cost model takes clusters for a lone L = 32 and row kernels for a lone L = 64
@pytest.mark.parametrize("L,clusters", [(32, True), (64, False)])
def test_annealing_knob_reaches_the_server(sg, monkeypatch, L, clusters):
    """SG_SA_CLUSTER turns the cluster kernel off, or takes it, for chunks too: with waits that give
    up at once a chunk on clusters times out, one through the row kernels does not."""
    req = sg.request(sg.SG_REQ_SA, L, 4, 32, 0.1, 3.0, 0.0, 40, sweeps_per_restart=40)
    want = _one(sg, req, 20)
    assert want["status"] == sg.SG_OK
    monkeypatch.setenv("SG_WAIT_LIMIT", "0")
    assert (_one(sg, req, 20)["status"] == sg.SG_ETIMEOUT) == clusters
    monkeypatch.setenv("SG_SA_CLUSTER", "1")
    assert _one(sg, req, 20)["status"] == sg.SG_ETIMEOUT
    monkeypatch.setenv("SG_SA_CLUSTER", "0")
    got = _one(sg, req, 20)
    assert got["status"] == sg.SG_OK and got["minE"] == want["minE"]


# Pinned memory comes with whatever it held; here an energy, a status, a ground state and the first
# token a server writes.
_PINNED = """
#define _GNU_SOURCE
#include <dlfcn.h>
#include <stddef.h>
int cudaHostAlloc(void** p, size_t n, unsigned flags)
{
    static int (*real)(void**, size_t, unsigned);
    if (!real) {
        void* lib = dlopen("libcudart.so.13", RTLD_NOW | RTLD_NOLOAD);
        *(void**)&real = dlsym(lib ? lib : RTLD_NEXT, "cudaHostAlloc");
    }
    const int rc = real ? real(p, n, flags) : 1;
    if (rc == 0 && n == 64) {
        long long* w = (long long*)*p;
        w[0] = -1000000000, w[1] = 0, w[2] = -1, w[3] = 1;
    }
    return rc;
}
"""
_SOLVE = """
from paper_2501_17267_gb300 import sg
inst = sg.Instance.create(40, 7)
want = int(sg.sa_run(inst, 32, 400, 0.1, 3.0, seed=5)["E"].min())
req = sg.request(sg.SG_REQ_SA, 40, 7, 32, 0.1, 3.0, 0.0, 400, run_seed=5, sweeps_per_restart=400)
with sg.Server(1 << 30, chunk_sweeps=400) as srv:
    got = srv.poll(srv.submit(req))
assert got["e_gs"] == inst.e_gs and got["minE"] == want, (got, want)
"""


def test_report_words_start_clean(tmp_path):
    """What the words of a chunk's report held before is no report (in a process of its own)."""
    (tmp_path / "pinned.c").write_text(_PINNED)
    lib = str(tmp_path / "pinned.so")
    subprocess.run(["gcc", "-shared", "-fPIC", str(tmp_path / "pinned.c"), "-o", lib, "-ldl"], check=True)
    env = dict(os.environ, LD_PRELOAD=lib, SG_SA_CLUSTER_C="8")
    r = subprocess.run([sys.executable, "-c", _SOLVE], cwd=ROOT, env=env, capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr[-2000:]


def _fine_ladder(sg, beta):
    """A request whose exchange tables have some 70 million entries (half a second of host work) and
    whose device memory no small budget covers."""
    return sg.request(sg.SG_REQ_PT, 128, 1, 64, beta, beta * (1.0 + 63 * 2e-5), 0.0, 10)


def test_submit_does_not_wait_for_another_callers_tables(sg):
    with sg.Server(16 << 20) as srv:
        spent = []

        def submit():
            t0 = time.perf_counter()
            with pytest.raises(sg.SGError):
                srv.submit(_fine_ladder(sg, 1.0))
            spent.append(time.perf_counter() - t0)

        other = threading.Thread(target=submit)
        other.start()
        time.sleep(0.05)
        t0 = time.perf_counter()
        ticket = srv.submit(sg.request(sg.SG_REQ_PT, 4, 2, 8, 0.3, 2.0, 0.0, 10))
        took = time.perf_counter() - t0
        other.join()
        assert spent[0] > 0.2  # long enough to tell
        assert took < spent[0] / 4
        srv.poll(ticket)


def test_tables_kept_between_requests_are_bounded(sg):
    """Requests that are gone leave no unbounded tables behind."""
    def resident():
        with open("/proc/self/statm") as f:
            return int(f.read().split()[1]) * os.sysconf("SC_PAGE_SIZE")

    with sg.Server(16 << 20) as srv:
        sizes = []
        for k in range(5):
            with pytest.raises(sg.SGError) as e:
                srv.submit(_fine_ladder(sg, 1.0 + 0.01 * k))
            assert e.value.code == sg.SG_ENOMEM
            sizes.append(resident())
    assert sizes[-1] - sizes[0] < 100 << 20  # one table set is about 280 MB


def test_poll_of_a_request_that_never_ran_holds_nobody_up(sg):
    """The planted energy of a large request cancelled in the queue is host work of the caller
    that asks for it, not of everybody."""
    busy = sg.request(sg.SG_REQ_PT, 16, 1, 16, 0.02, 0.1, 0.0, 10 ** 9)  # (too hot to reach anything)
    large = sg.request(sg.SG_REQ_SA, 256, 3, 1, 0.1, 3.0, 0.0, 10, sweeps_per_restart=10)
    with sg.Server(8 << 30, max_active=1, chunk_sweeps=10) as srv:
        running = srv.submit(busy)
        tickets = [srv.submit(large) for _ in range(4)]
        for t in tickets:
            srv.cancel(t)
        spent, got = [], []

        def ask():
            for t in tickets:
                t0 = time.perf_counter()
                got.append(srv.poll(t))
                spent.append(time.perf_counter() - t0)

        other = threading.Thread(target=ask)
        other.start()
        waits = []
        while other.is_alive():
            t0 = time.perf_counter()
            assert srv.poll(running, timeout_ms=0) is None
            waits.append(time.perf_counter() - t0)
            time.sleep(1e-3)
        other.join()
        srv.cancel(running)
        assert all(r["status"] == sg.SG_ECANCELED and r["e_gs"] == got[0]["e_gs"] for r in got)
    assert min(spent) > 0.01  # long enough to tell
    assert sorted(waits)[len(waits) // 2] < min(spent) / 3
