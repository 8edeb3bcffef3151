"""sim_run_noalloc (the entry point for callers that cannot allocate device memory) against the
regular sim_load_csr + sim_run path and the CPU oracle.

Callers such as a serving process whose GPU memory is entirely reserved by its own pool, or a
latency-sensitive loop that must not make synchronising allocation calls, use sim_run_noalloc:
it keeps all of its scratch in a fixed device array inside the library.  This file is collected
last so that a run stopping at the first failure has already run every other test.
"""
import numpy as np
import pytest

from tests.gpu_helpers import FIELDS, n_threads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g
    g.build()


def _regular(pol, w):
    """sim_load_csr + sim_run with default options (tie seed 0 for every instance, as the
    allocation-free entry point uses)."""
    from paper_2508_14544_gb300 import Simulator
    with Simulator(pol, w.M, w.n_instances) as sim:
        sim.load(w.offsets, w.arrival, w.prompt, w.lower, w.upper, w.true_o)
        return sim.run()


def _oracle(pol, w):
    from oracle import plain
    return plain.run_batch(pol, w.M, w.offsets, w.arrival, w.prompt, w.lower, w.upper, w.true_o,
                           n_threads=n_threads(), tie_seeds=np.zeros(w.n_instances, np.uint64))


def _dev(w):
    import torch
    return [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (w.arrival, w.prompt, w.lower, w.upper, w.true_o)]


def _noalloc(pol, w, dev, out):
    import torch

    from paper_2508_14544_gb300 import _lib as L
    rc = L.sim_run_noalloc(pol, w.M, np.ascontiguousarray(w.offsets, dtype=np.int64), *dev, out)
    assert rc == L.SIM_OK, L.sim_last_error(None)
    torch.cuda.synchronize()
    return out.cpu().numpy().view(L.RESULT_DTYPE).reshape(-1)[: w.n_instances].copy()


def _check(got, ref, tag):
    for f in FIELDS:
        assert np.array_equal(got[f], ref[f]), (tag, f)


def test_noalloc_matches_sim_run_and_oracle_calls_in_a_row():
    import torch

    from paper_2508_14544_gb300 import workloads as W
    from paper_2508_14544_gb300 import _lib as L
    w = W.make_workload("c2", list(range(0, 1024, 11)))  # 94 instances, all four alphas
    dev = _dev(w)
    out = torch.zeros(w.n_instances * L.RESULT_DTYPE.itemsize, dtype=torch.uint8, device="cuda")
    for pol in (L.SIM_AMIN, L.SIM_AMAX, L.SIM_HSF, L.SIM_AMIN):  # calls in a row share the fixed scratch
        got = _noalloc(pol, w, dev, out)
        _check(got, _regular(pol, w), f"sim_run pol={pol}")
        _check(got, _oracle(pol, w), f"oracle pol={pol}")
        assert np.all(got["status"] == 0)


def test_noalloc_empty_instances():
    import torch

    from paper_2508_14544_gb300 import workloads as W
    from paper_2508_14544_gb300 import _lib as L
    rng = np.random.default_rng(3)
    parts = []
    for i in range(40):
        n = 0 if i % 3 == 0 else int(rng.integers(1, 300))
        o = rng.integers(1, 60, n)
        l = np.array([rng.integers(1, x + 1) for x in o], dtype=np.int64)
        parts.append(dict(a=np.sort(rng.integers(0, 50, n)), s=rng.integers(1, 20, n), l=l, u=o + 5, o=o))
    w = W.concat_instances("with-empty", 900, parts)
    dev = _dev(w)
    out = torch.zeros(w.n_instances * L.RESULT_DTYPE.itemsize, dtype=torch.uint8, device="cuda")
    for pol in (L.SIM_AMIN, L.SIM_AMAX, L.SIM_HSF):
        got = _noalloc(pol, w, dev, out)
        _check(got, _regular(pol, w), f"sim_run pol={pol}")
        _check(got, _oracle(pol, w), f"oracle pol={pol}")
        assert np.all(got["total_latency"][::3] == 0)


def test_noalloc_rejects_oversize_inputs():
    import torch

    from paper_2508_14544_gb300 import _lib as L
    n = 2049  # one instance above the 2048-request limit
    dev = [torch.ones(n, dtype=torch.int32, device="cuda") for _ in range(5)]
    out = torch.zeros(L.RESULT_DTYPE.itemsize, dtype=torch.uint8, device="cuda")
    rc = L.sim_run_noalloc(L.SIM_HSF, 10_000, np.array([0, n], dtype=np.int64), *dev, out)
    assert rc == L.SIM_E_INVAL
    assert "2048" in L.sim_last_error(None)
    # 300 instances of 1000 requests: each within the per-instance limit, 300,000 in total
    off = np.arange(301, dtype=np.int64) * 1000
    dev = [torch.ones(300_000, dtype=torch.int32, device="cuda") for _ in range(5)]
    out = torch.zeros(300 * L.RESULT_DTYPE.itemsize, dtype=torch.uint8, device="cuda")
    rc = L.sim_run_noalloc(L.SIM_AMIN, 10_000, off, *dev, out)
    assert rc == L.SIM_E_INVAL
    assert "262144" in L.sim_last_error(None)


@pytest.mark.parametrize("pol", [0, 1, 2])
def test_noalloc_sets_beyond_shared_memory(pol):
    """Instances whose active set outgrows the shared-memory slots (one-token prompts, up to 2000 jobs at
    once) between small ones: the second launch simulates exactly those."""
    import torch

    from paper_2508_14544_gb300 import workloads as W
    from paper_2508_14544_gb300 import _lib as L
    rng = np.random.default_rng(17)
    parts = []
    for n in (2000, 30, 513, 512, 511, 1, 2048, 0, 700, 64):
        o = rng.integers(1, 6, n)
        a = np.sort(rng.integers(0, 3, n))
        parts.append(dict(a=a, s=np.ones(n, np.int64), l=np.ones(n, np.int64), u=o + 2, o=o))
    w = W.concat_instances("wide", 6000, parts)
    out = torch.zeros(w.n_instances * L.RESULT_DTYPE.itemsize, dtype=torch.uint8, device="cuda")
    dev = _dev(w)
    for _ in range(2):
        _check(_noalloc(pol, w, dev, out), _oracle(pol, w), f"wide pol={pol}")


def test_noalloc_more_instances_than_warps():
    """16384 instances (the limit), several per simulating warp, with queues that spill to their own
    buffers."""
    import torch

    from paper_2508_14544_gb300 import workloads as W
    from paper_2508_14544_gb300 import _lib as L
    rng = np.random.default_rng(18)
    parts = []
    for i in range(16384):
        n = 300 if i % 64 == 0 else int(rng.integers(0, 12))
        o = rng.integers(1, 30, n)
        l = rng.integers(1, o + 1)
        parts.append(dict(a=np.sort(rng.integers(0, 40, n)), s=rng.integers(1, 9, n), l=l, u=o + 5, o=o))
    w = W.concat_instances("many", 120, parts)
    out = torch.zeros(w.n_instances * L.RESULT_DTYPE.itemsize, dtype=torch.uint8, device="cuda")
    _check(_noalloc(L.SIM_AMIN, w, _dev(w), out), _oracle(L.SIM_AMIN, w), "many")


@pytest.mark.parametrize("pol", [0, 1, 2])
def test_noalloc_every_request_active_at_once(pol):
    """Sets that fill the shared-memory slots (512), or the array's (2048), to the last one."""
    import torch

    from paper_2508_14544_gb300 import workloads as W
    from paper_2508_14544_gb300 import _lib as L
    rng = np.random.default_rng(19)
    for n in (128, 511, 512, 513, 2047, 2048):
        o = rng.integers(1, 9, n)
        w = W.concat_instances("full", 100_000, [dict(a=np.zeros(n, np.int64), s=np.ones(n, np.int64),
                                                      l=np.maximum(o // 2, 1), u=o + 2, o=o)] * 3)
        out = torch.zeros(w.n_instances * L.RESULT_DTYPE.itemsize, dtype=torch.uint8, device="cuda")
        _check(_noalloc(pol, w, _dev(w), out), _oracle(pol, w), f"full pol={pol} n={n}")


@pytest.mark.parametrize("pol", [0, 1, 2])
def test_noalloc_captured_with_other_sizes(pol):
    """A captured call copies the offsets again on every replay: instances that have grown past the sizes at
    capture are staged all the same (their sets fit the slots), and those that reach past the arrays' limits
    get SIM_E_INVAL."""
    import torch

    from paper_2508_14544_gb300 import workloads as W
    from paper_2508_14544_gb300 import _lib as L
    rng = np.random.default_rng(27)

    def workload(sizes):
        parts = []
        for n in sizes:
            o = rng.integers(1, 40, n)
            l = rng.integers(1, o + 1)
            parts.append(dict(a=rng.integers(0, 30, n), s=rng.integers(1, 9, n), l=l, u=o + 5, o=o))
        return W.concat_instances("replay", 300, parts)

    room, off = 8192, torch.zeros(5, dtype=torch.int64).pin_memory()
    dev = [torch.zeros(room, dtype=torch.int32, device="cuda") for _ in range(5)]
    out = torch.zeros(4 * L.RESULT_DTYPE.itemsize, dtype=torch.uint8, device="cuda")

    def put(w):
        off.numpy()[:] = w.offsets
        for d, x in zip(dev, (w.arrival, w.prompt, w.lower, w.upper, w.true_o)):
            d[: x.size].copy_(torch.from_numpy(np.ascontiguousarray(x)))

    small = workload((10, 7, 0, 9))
    put(small)
    _check(_noalloc(pol, small, dev, out), _oracle(pol, small), "plain")
    graph, side = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=side):
        rc = L.sim_run_noalloc(pol, small.M, off.numpy(), *dev, out, stream=side.cuda_stream)
    assert rc == L.SIM_OK, L.sim_last_error(None)
    for sizes in ((10, 7, 0, 9), (17, 300, 1, 16), (2048, 5, 33, 600)):
        w = workload(sizes)
        put(w)
        torch.cuda.synchronize()
        graph.replay()
        torch.cuda.synchronize()
        got = out.cpu().numpy().view(L.RESULT_DTYPE).reshape(-1).copy()
        _check(got, _oracle(pol, w), f"replay pol={pol} {sizes}")
    off.numpy()[:] = [0, 10, 10 + 2049, 2060, 2070]
    graph.replay()
    torch.cuda.synchronize()
    assert out.cpu().numpy().view(L.RESULT_DTYPE)["status"].reshape(-1)[1] == L.SIM_E_INVAL
