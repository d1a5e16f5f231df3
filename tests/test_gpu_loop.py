"""The one-launch iteration (and the separate kernels just past it) against the CPU oracle
at the edges of their range: a single warp per curve and 64 threads per curve
(512 / 513 unknowns), the largest grid of the one launch and the first past
it, thin and masked domains, both precision modes.

Tolerances as in test_gpu_parity.py: FP64 1e-12, FP32 + refinement 1e-5, both
of max |u|."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2411_11041_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _problem(nx, ny, field, mask, seed=5):
    rng = np.random.default_rng(seed)
    if field == "sheared":
        b1, b2 = W.sheared_beta(nx, ny)
    else:
        b1, b2 = np.full((ny, nx), field[0]), np.full((ny, nx), field[1])
    y1 = (ny - 1) / (nx - 1)
    f = W.random_field(rng, nx, ny)
    return W.Problem(nx, ny, 3e-3, 0.8, b1, b2, f, W.make_mask(mask, nx, ny), y1=y1)


CASES = [
    (31, 9, (1.0, 0.37), "square"),
    (40, 40, (1.0, 0.0), "square"),      # aligned: curves on grid lines
    (65, 64, "sheared", "square"),
    (90, 90, (-0.6, 0.8), "disc"),
    (514, 24, (1.0, 0.0), "square"),     # 512 unknowns: one warp a curve
    (515, 24, (1.0, 0.0), "square"),     # 513: 64 threads
    (1026, 11, (1.0, 0.0), "square"),    # 1024 unknowns, the longest of 64 threads
    (1027, 11, (1.0, 0.0), "square"),    # past it: separate kernels
    (300, 290, "sheared", "L"),
    (512, 512, "sheared", "square"),     # the largest grid of the one launch
    (512, 513, "sheared", "square"),     # the first of the separate kernels
]


@pytest.mark.parametrize("nx,ny,field,mask", CASES)
@pytest.mark.parametrize("prec", [0, 1])
def test_fixed_steps_match_oracle(nx, ny, field, mask, prec):
    import torch
    from paper_2411_11041_gb300 import Solver
    p = _problem(nx, ny, field, mask)
    if field == "sheared" and mask == "L":
        p.beta2[:] = np.abs(p.beta2)
    o = O.Oracle(p)
    s = Solver(p, tol=0.0, max_iter=3, prec=prec)
    u, it, st, code = s.solve_stationary(want_iter=True)
    ref, refit, k, rel, _ = o.solve_stationary(tol=0.0, max_iter=3)
    tol = 1e-12 if prec == 0 else 1e-5
    assert st["iters"] == k == 3
    assert np.abs(u.cpu().numpy() - ref).max() <= tol * np.abs(ref).max()
    assert np.abs(it.cpu().numpy() - refit).max() <= tol * np.abs(refit).max()
    assert abs(st["rel_update"] - rel) <= (1e-9 if prec == 0 else 1e-3) * rel + 1e-13
    # a caller's own split step, in place
    v = torch.tensor(np.random.default_rng(1).normal(size=(ny, nx)) * o.interior(), device="cuda:0")
    rh, rn = o.split_step(0.5, 0.02, v.cpu().numpy())
    uh, un = s.split_step(v, 0.02)
    assert np.abs(uh.cpu().numpy() - rh).max() <= tol * np.abs(rh).max()
    assert np.abs(un.cpu().numpy() - rn).max() <= tol * np.abs(rn).max()


def test_two_streams_solve_at_once():
    """Two handles on two streams from two threads: each launch waits for the
    SMs it needs, and both answers are the single solves'."""
    import threading

    import torch
    from paper_2411_11041_gb300 import Solver
    ps = [_problem(120, 120, "sheared", "square", seed=k) for k in (1, 2)]
    ref = [Solver(p, tol=1e-9, max_iter=5000).solve_stationary()[0].clone() for p in ps]
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in ps]
    out = [None, None]

    def work(i):
        with torch.cuda.stream(streams[i]):
            s = Solver(ps[i], tol=1e-9, max_iter=5000, stream=streams[i])
            for _ in range(5):
                out[i] = s.solve_stationary()[0]

    th = [threading.Thread(target=work, args=(i,)) for i in range(2)]
    [t.start() for t in th]
    [t.join() for t in th]
    torch.cuda.synchronize()
    for u, r in zip(out, ref):
        assert torch.equal(u, r)


def test_threads_with_different_launch_shapes():
    """Handles whose launches want different amounts of shared memory (rows per
    thread 4 and 16), solved from two threads at once, many short solves each."""
    import threading

    import torch
    from paper_2411_11041_gb300 import Solver
    ps = [_problem(60, 60, "sheared", "square", seed=3), _problem(240, 240, "sheared", "square", seed=4)]
    rows = (4, 16)
    ref = [Solver(p, tol=0.0, max_iter=2, rows_per_thread=r).solve_stationary()[0].clone() for p, r in zip(ps, rows)]
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in ps]
    bad = [None, None]

    def work(i):
        try:
            with torch.cuda.stream(streams[i]):
                s = Solver(ps[i], tol=0.0, max_iter=2, rows_per_thread=rows[i], stream=streams[i])
                bad[i] = sum(not torch.equal(s.solve_stationary()[0], ref[i]) for _ in range(100))
        except Exception as e:  # reported by the assertion below
            bad[i] = e

    th = [threading.Thread(target=work, args=(i,)) for i in range(2)]
    [t.start() for t in th]
    [t.join() for t in th]
    assert bad == [0, 0]


def _beside_a_busy_stream(call, mine):
    """call() on stream mine while another stream keeps one block of the device
    busy for about 50 ms; whether it came back before that stream was done."""
    import torch
    other = torch.cuda.Stream()
    with torch.cuda.stream(mine):
        call()  # first use: buffers, factors, kernels
    torch.cuda.synchronize()
    with torch.cuda.stream(other):
        torch.cuda._sleep(100_000_000)
    with torch.cuda.stream(mine):
        call()  # returns when its results are there
    first = not other.query()
    torch.cuda.synchronize()
    return first


@pytest.mark.parametrize("n", [33, 129, 300])
def test_split_step_does_not_wait_for_other_streams(n):
    """A split step needs no empty device: it runs beside another stream's kernel."""
    import torch
    from paper_2411_11041_gb300 import Solver
    mine = torch.cuda.Stream()
    s = Solver(_problem(n, n, "sheared", "square"), stream=mine)
    u = torch.rand((n, n), dtype=torch.float64, device="cuda:0")
    torch.cuda.synchronize()
    assert _beside_a_busy_stream(lambda: s.split_step(u, 0.05), mine)


@pytest.mark.parametrize("n", [33, 129, 300])
def test_solve_does_not_wait_for_other_streams(n):
    """The one launch takes part of an SM's registers: it starts beside another
    stream's kernel."""
    import torch
    from paper_2411_11041_gb300 import Solver
    mine = torch.cuda.Stream()
    s = Solver(_problem(n, n, "sheared", "square"), tol=0.0, max_iter=10, stream=mine)
    torch.cuda.synchronize()
    assert _beside_a_busy_stream(lambda: s.solve_stationary(), mine)


@pytest.mark.parametrize("n,k", [(64, 4), (129, 4), (257, 2)])
def test_small_solves_overlap(n, k):
    """k handles of one size on k streams: their launches fit the device side by
    side, so all of them take little longer than one (below 1.5 of it; one
    after the other k of it)."""
    import threading
    import time

    import torch
    from paper_2411_11041_gb300 import Solver
    streams = [torch.cuda.Stream() for _ in range(k)]
    hs = [Solver(_problem(n, n, "sheared", "square", seed=i), tol=0.0, max_iter=2000, stream=streams[i])
          for i in range(k)]
    torch.cuda.synchronize()

    def seconds(m):
        go = threading.Barrier(m + 1)

        def work(i):
            with torch.cuda.stream(streams[i]):
                go.wait()
                hs[i].solve_stationary()

        th = [threading.Thread(target=work, args=(i,)) for i in range(m)]
        [t.start() for t in th]
        go.wait()
        t0 = time.perf_counter()
        [t.join() for t in th]
        return time.perf_counter() - t0

    seconds(k)
    one, all_ = min(seconds(1) for _ in range(3)), min(seconds(k) for _ in range(3))
    assert all_ < 1.5 * one, (one, all_)


@pytest.mark.parametrize("nx,ny,field", [
    (300, 300, "sheared"),               # the largest grid of the one launch
    (301, 300, "sheared"),               # the first of the separate kernels
    (400, 400, "sheared"),
    (401, 400, "sheared"),
    (17, 2200, (0.8, 0.6)),              # near three slices a group
    (17, 2400, (0.8, 0.6)),              # past them: separate kernels
    (600, 260, (1.0, 0.0)),              # 64 threads a curve, two groups a block
])
@pytest.mark.parametrize("prec", [0, 1])
def test_fixed_steps_match_oracle_at_the_rules_edges(nx, ny, field, prec):
    test_fixed_steps_match_oracle(nx, ny, field, "square", prec)


REFUSED = """
import sys
import numpy as np
import torch
from tests.test_gpu_loop import _problem
from paper_2411_11041_gb300 import Solver
for prec in (0, 1):
    s = Solver(_problem(90, 70, "sheared", "square"), tol=0.0, max_iter=7, prec=prec)
    for _ in range(2):
        u, _, st, _ = s.solve_stationary()
        assert st["iters"] == 7
    np.save(sys.argv[1] + "%d.npy" % prec, u.cpu().numpy())
"""


def test_a_refused_launch_takes_the_graph(tmp_path):
    """Where the runtime refuses the cooperative launch (the blocks do not fit the
    part of the device the process may use; here a library in front of the
    runtime answers so), the solve runs as the graph of separate kernels."""
    import os
    import subprocess
    import sys

    from paper_2411_11041_gb300 import Solver
    src, so = tmp_path / "refuse.c", tmp_path / "refuse.so"
    src.write_text("int cudaLaunchCooperativeKernel() { return 720; }\n")  # cudaErrorCooperativeLaunchTooLarge
    subprocess.run(["gcc", "-shared", "-fPIC", "-o", str(so), str(src)], check=True)
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", REFUSED, str(tmp_path / "u")], cwd=root, capture_output=True, text=True,
                       timeout=300, env=dict(os.environ, LD_PRELOAD=str(so)))
    assert r.returncode == 0, r.stderr[-2000:]
    for prec in (0, 1):
        u = Solver(_problem(90, 70, "sheared", "square"), tol=0.0, max_iter=7, prec=prec).solve_stationary()[0]
        assert np.array_equal(u.cpu().numpy(), np.load(tmp_path / f"u{prec}.npy"))


def _partition_stream(sms):
    """A stream on a partition of about sms SMs (a green context of this process)."""
    import ctypes as C

    import torch
    torch.zeros(1, device="cuda:0")  # the primary context
    cu = C.CDLL("libcuda.so.1")

    def ok(code, what):
        if code:
            pytest.skip(f"no partition of the SMs here: {what} gave {code}")

    size = 4 + 92 + 48  # CUdevResource; the SM count is the first word of its union
    whole, part, rest = (C.create_string_buffer(size) for _ in range(3))
    groups, desc, ctx, st = C.c_uint(1), C.c_void_p(), C.c_void_p(), C.c_void_p()
    ok(cu.cuDeviceGetDevResource(0, whole, 1), "cuDeviceGetDevResource")
    ok(cu.cuDevSmResourceSplitByCount(part, C.byref(groups), whole, rest, 0, C.c_uint(sms)), "cuDevSmResourceSplitByCount")
    ok(cu.cuDevResourceGenerateDesc(C.byref(desc), part, 1), "cuDevResourceGenerateDesc")
    ok(cu.cuGreenCtxCreate(C.byref(ctx), desc, 0, 1), "cuGreenCtxCreate")
    ok(cu.cuGreenCtxStreamCreate(C.byref(st), ctx, 1, 0), "cuGreenCtxStreamCreate")
    return torch.cuda.ExternalStream(st.value), int.from_bytes(part.raw[96:100], "little")


@pytest.mark.parametrize("n", [64, 129, 300])
def test_solve_on_a_partition_of_the_sms(n):
    """A stream that has a few of the SMs: as many blocks as those hold, or the
    graph, and the same states as on the whole device."""
    import torch
    from paper_2411_11041_gb300 import Solver
    p = _problem(n, n, "sheared", "square")
    ref = Solver(p, tol=0.0, max_iter=20).solve_stationary()[0].clone()
    st, sms = _partition_stream(16)
    assert 1 <= sms < torch.cuda.get_device_properties(0).multi_processor_count
    torch.cuda.synchronize()
    with torch.cuda.stream(st):
        s = Solver(p, tol=0.0, max_iter=20, stream=st)
        for _ in range(2):
            u, _, stats, _ = s.solve_stationary()
    torch.cuda.synchronize()
    assert stats["iters"] == 20 and torch.equal(u, ref)


@pytest.mark.parametrize("n", [64, 257, 385])
@pytest.mark.parametrize("prec", [0, 1])
def test_tuned_handle_is_no_slower(n, prec):
    """The shapes adr_autotune keeps are the fastest of what a solve then runs:
    a tuned handle takes at most the untuned one's time per step, and 8 % for
    the spread of single runs."""
    from paper_2411_11041_gb300 import Solver
    s = Solver(_problem(n, n, "sheared", "square"), tol=0.0, max_iter=200, prec=prec)

    def us_per_step():
        s.solve_stationary()
        return min(s.solve_stationary()[2]["ms"] for _ in range(5)) / 200 * 1e3

    before = us_per_step()
    rows, blocks, ms = s.autotune()
    assert rows in (4, 8, 16) and blocks in (2, 4, 8)
    after = us_per_step()
    assert after <= 1.08 * before, (before, after, rows, blocks)


@pytest.mark.parametrize("prec", [0, 1])
def test_barrier_timeout_is_reported_and_the_handle_recovers(prec):
    """A bound of one poll makes the grid barriers of the one-launch iteration give
    up: the blocks leave, and the solve and the time steps report ADR_ETIMEOUT.
    With the default bound restored the same handle solves as before, bit for
    bit."""
    import torch
    from paper_2411_11041_gb300 import AdrError, Solver
    p = _problem(129, 120, "sheared", "square")
    s = Solver(p, tol=0.0, max_iter=25, prec=prec)
    u0, _, st0, _ = s.solve_stationary()
    u0 = u0.clone()
    s.set_wait_limit(1)
    with pytest.raises(AdrError, match="ETIMEOUT"):
        s.solve_stationary()
    for mode in (0, 1):
        with pytest.raises(AdrError, match="ETIMEOUT"):
            s.step_parabolic(u0.clone(), 1e-3, 3, mode)
    with pytest.raises(AdrError, match="EINVAL"):
        s.set_wait_limit(-1)
    s.set_wait_limit(0)
    u, _, st, _ = s.solve_stationary()
    assert torch.equal(u, u0)
    assert (st["iters"], st["rel_update"], st["max_correction"]) == (25, st0["rel_update"], st0["max_correction"])


@pytest.mark.parametrize("nx,ny,opts,one", [
    (64, 64, {}, True),
    (300, 300, {}, True),                          # the largest grid of the one launch
    (301, 300, {}, False),
    (400, 400, {}, False),
    (64, 64, dict(transfer=1), False),
    (64, 64, dict(anderson=2), False),
    (290, 290, dict(rows_per_thread=4), False),    # 128 threads a curve
    (290, 290, dict(rows_per_thread=16), True),
    (1000, 60, {}, True),                          # 1.5 slices a group
    (1000, 80, {}, False),                         # as many, and more nodes
    (1400, 64, {}, False),
    (80, 1500, {}, False),
    (2000, 50, {}, False),                         # nearly three
])
def test_route_of_a_solve(nx, ny, opts, one):
    """What the handle reports is what a solve then does: only the one launch
    waits at barriers, so a bound of one poll ends it and nothing else."""
    from paper_2411_11041_gb300 import AdrError, Solver
    s = Solver(_problem(nx, ny, "sheared", "square"), tol=0.0, max_iter=5, **opts)
    assert s.one_launch() == one
    s.set_wait_limit(1)
    if one:
        with pytest.raises(AdrError, match="ETIMEOUT"):
            s.solve_stationary()
    else:
        assert s.solve_stationary()[2]["iters"] == 5


def test_large_solves_share_the_device():
    """Eight handles of 385^2 on eight streams: separate kernels, whose steps take
    turns at the device's full rate (below five times one handle's time; as
    single launches, at most two of which fit the device at once, 6.3)."""
    import threading
    import time

    import torch
    from paper_2411_11041_gb300 import Solver
    streams = [torch.cuda.Stream() for _ in range(8)]
    hs = [Solver(_problem(385, 385, "sheared", "square", seed=i), tol=0.0, max_iter=1000, stream=streams[i])
          for i in range(8)]
    torch.cuda.synchronize()

    def seconds(m):
        go = threading.Barrier(m + 1)

        def work(i):
            with torch.cuda.stream(streams[i]):
                go.wait()
                hs[i].solve_stationary()

        th = [threading.Thread(target=work, args=(i,)) for i in range(m)]
        [t.start() for t in th]
        go.wait()
        t0 = time.perf_counter()
        [t.join() for t in th]
        return time.perf_counter() - t0

    seconds(8)
    one, all_ = min(seconds(1) for _ in range(3)), min(seconds(8) for _ in range(3))
    assert all_ < 5.0 * one, (one, all_)
