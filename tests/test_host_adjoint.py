"""Host side of the adjoint on the CPU: the library's objects linked with a CUDA runtime that runs
no kernel, notes every launch and its stream, and lets named calls fail (tests/helpers/
fake_cudart.cpp).  Each test is a child process with that library in place of libabp.so."""
import os
import shutil
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = os.path.join(ROOT, "tests", "helpers", "fake_cudart.cpp")

PRELUDE = r'''
import ctypes, os, sys
import numpy as np
sys.path.insert(0, os.environ["ABP_ROOT"])
from paper_1104_2499_gb300 import abp as A, workloads as W

L = A.lib()
L.fake_fail.argtypes = [ctypes.c_char_p, ctypes.c_long, ctypes.c_long]
L.fake_kernel.argtypes, L.fake_kernel.restype = [ctypes.c_long], ctypes.c_char_p
L.fake_ordered.argtypes = [ctypes.c_void_p, ctypes.c_long]
for f in ("fake_calls", "fake_launches", "fake_live", "fake_peak"):
    getattr(L, f).restype = ctypes.c_size_t if f in ("fake_live", "fake_peak") else ctypes.c_long


def integrated(n_traj=(300, 65, 1), n_steps=(203, 64, 7), K=8, ppt=2):
    n = len(n_traj)
    w = W.Workload(name="host", sets=[W.params(D=0.1)] * n, n_traj=list(n_traj), n_steps=list(n_steps), dt=1e-3, seed=1,
                   checkpoint_every=K)
    ctx = A.abp_create(A.make_config(w, particles_per_thread=ppt, schedule=1, steps_per_launch=max(n_steps)))
    A.abp_set_params(ctx, w.sets, w.n_traj, w.n_steps)
    A.abp_integrate(ctx)
    return ctx, np.zeros((n, 6)), np.zeros((sum(n_traj), 6))


def status(call, *a):
    try:
        call(*a)
    except A.AbpError as e:
        return e.status
    return A.ABP_OK


def kernels(i):
    return [L.fake_kernel(k).decode() for k in range(i, L.fake_launches())]
'''


@pytest.fixture(scope="module")
def child(tmp_path_factory):
    from paper_1104_2499_gb300 import build as B

    try:
        nvcc = B.nvcc()
    except RuntimeError:
        pytest.skip("nvcc not available to build libabp.so")
    if not shutil.which("g++"):
        pytest.skip("no C++ compiler")
    B.build()
    tmp = tmp_path_factory.mktemp("fake")
    lib = str(tmp / "libabp_fake.so")
    objs = [os.path.join(B.OUT, s.replace(".cu", ".o")) for s in B.SOURCES]
    subprocess.run(["g++", "-std=c++17", "-O1", "-Wall", "-Werror", "-fPIC", "-shared", "-o", lib, SRC] + objs +
                   ["-I", os.path.join(os.path.dirname(os.path.dirname(nvcc)), "include"), "-Wl,-Bsymbolic",
                    "-Wl,-z,defs", "-ldl", "-lpthread", "-lrt"], check=True)

    def run(code, **env):
        e = {k: v for k, v in os.environ.items() if not k.startswith("ABP_")}
        e.update(ABP_LIB=lib, ABP_ROOT=ROOT, **env)
        r = subprocess.run([sys.executable, "-c", PRELUDE + code], env=e, capture_output=True, text=True, timeout=300)
        assert r.returncode == 0, r.stderr[-4000:]

    return run


def test_readout_follows_a_backward(child):
    child('''
ctx, grad, dv = integrated()
assert status(A.abp_backward_traj, ctx, dv) == A.ABP_ESTATE
A.abp_backward(ctx, None, grad)
assert status(A.abp_backward_traj, ctx, dv) == A.ABP_OK
# a call refused for its arguments leaves the sums of the last one readable
assert status(A.abp_backward, ctx, None, None) == A.ABP_EINVAL
assert status(A.abp_backward, ctx, None, grad, 7) == A.ABP_EINVAL
assert status(A.abp_backward_traj, ctx, dv) == A.ABP_OK
''')


# small buffers first (the noise drawn again), then a larger form that finds no memory at all
def test_readout_is_refused_after_a_backward_without_scratch(child):
    child('''
os.environ["ABP_ADJ_HANDOFF_BYTES"] = "0"
ctx, grad, dv = integrated()
A.abp_backward(ctx, None, grad)
del os.environ["ABP_ADJ_HANDOFF_BYTES"]
L.fake_fail(b"cudaMalloc", 0, 1000)
assert status(A.abp_backward, ctx, None, grad) == A.ABP_ENOMEM
L.fake_fail(None, 0, 0)
n = L.fake_launches()
assert status(A.abp_backward_traj, ctx, dv) == A.ABP_ESTATE
assert L.fake_launches() == n  # no kernel on a scratch that is gone
A.abp_backward(ctx, None, grad)
assert status(A.abp_backward_traj, ctx, dv) == A.ABP_OK
''')


@pytest.mark.parametrize("call", ["cudaMemsetAsync", "cudaEventRecord", "cudaStreamWaitEvent", "launch", "cudaMemcpyAsync"])
def test_readout_is_refused_after_a_backward_that_broke_off(child, call):
    child('''
ctx, grad, dv = integrated()
A.abp_backward(ctx, None, grad)
L.fake_fail(CALL, 0, 1000)
assert status(A.abp_backward, ctx, None, grad) == A.ABP_ECUDA
L.fake_fail(None, 0, 0)
assert status(A.abp_backward_traj, ctx, dv) == A.ABP_ESTATE
'''.replace("CALL", repr(call.encode())))


# the runtime keeps a failed call's error until it is asked for: a call that reported it has to
# take it away, or the next one, which checks its launches by it, reports it a second time
@pytest.mark.parametrize("call", ["cudaMemsetAsync", "cudaEventRecord", "cudaStreamWaitEvent"])
def test_an_error_is_reported_by_one_call_only(child, call):
    child('''
ctx, grad, dv = integrated()
L.fake_fail(CALL, 0, 1)
first = status(A.abp_backward, ctx, None, grad)
if CALL == b"cudaMemsetAsync":  # the work queue clears its counters too
    assert first == A.ABP_ECUDA
    w = W.Workload(name="q", sets=[W.params()], n_traj=[600], n_steps=[100], dt=1e-3, seed=1)
    q = A.abp_create(A.make_config(w, particles_per_thread=2, schedule=2, steps_per_launch=50))
    A.abp_set_params(q, w.sets, w.n_traj, w.n_steps)
    L.fake_fail(CALL, 0, 1)
    assert status(A.abp_integrate, q) == A.ABP_ECUDA
    A.abp_reset(q, 1)
    assert status(A.abp_integrate, q) == A.ABP_OK
assert first == A.ABP_ECUDA
assert status(A.abp_backward, ctx, None, grad) == A.ABP_OK
'''.replace("CALL", repr(call.encode())))


# one group of tiles and two; state rows in one launch and in several, the noise hand-off, the
# noise drawn again
@pytest.mark.parametrize("sms", [152, 2])
@pytest.mark.parametrize("form", [{}, {"ABP_ADJ_STATE_BYTES": "700000"},
                                  {"ABP_ADJ_STATE_BYTES": "0", "ABP_ADJ_HANDOFF_BYTES": "200000"},
                                  {"ABP_ADJ_HANDOFF_BYTES": "0"}], ids=["states", "states-several", "handoff", "redraw"])
def test_the_callers_stream_follows_every_launch(child, sms, form):
    # whichever call fails, and whether once or from then on, the caller's stream is ordered after
    # every kernel that was launched, and a failure is never reported as success
    child('''
L.fake_sms(SMS)
ctx, grad, dv = integrated(K=24)
A.abp_backward(ctx, None, grad)  # streams, events and scratch are there
names = set()
for call in (b"none", b"cudaEventRecord", b"cudaStreamWaitEvent", b"launch"):
    for n in (1, 1000):
        i, more = 0, True
        while more:
            n0 = L.fake_launches()
            L.fake_fail(call, i, n)
            s = status(A.abp_backward, ctx, None, grad)
            more = L.fake_calls() > i
            L.fake_fail(None, 0, 0)
            assert s == (A.ABP_ECUDA if more else A.ABP_OK), (call, i, n, s)
            for k in range(n0, L.fake_launches()):
                assert L.fake_ordered(None, k), (call, i, n, k - n0, L.fake_kernel(k))
            names |= set(kernels(n0))
            i += 1
        assert i > (0 if call == b"none" else 2)
assert any(KERNEL in k for k in names), names
'''.replace("SMS", str(sms)).replace("KERNEL", repr("level1_pair" if "ABP_ADJ_HANDOFF_BYTES" in form else "states")), **form)


# the form a batch takes: every step's state up to 32,768 trajectories (24,576 where the run is one
# segment) and 512 MB of buffers, else
# the noise hand-off within its budget, else the noise drawn again; a launch over several segments
# has its own sweep
@pytest.mark.parametrize("n_traj,K,env,expect", [
    (32768, 24, {}, ["adjoint_states_kernel", "adjoint_sweep_kernel"]),
    (32769, 24, {}, ["adjoint_level1_pair_kernelILb1", "adjoint_reverse_pair_kernelILb1ELb1"]),
    (32768, 24, {"ABP_ADJ_STATE_BYTES": "0"}, ["adjoint_level1_pair_kernelILb1", "adjoint_reverse_pair_kernelILb1ELb1"]),
    (24576, 300, {}, ["adjoint_states_kernel", "adjoint_sweep_kernel"]),
    (24577, 300, {}, ["adjoint_level1_pair_kernelILb1", "adjoint_reverse_pair_kernelILb1ELb0"]),
    (24577, 200, {}, ["adjoint_states_kernel", "adjoint_sweep_kernel"]),
    (366, 24, {"ABP_ADJ_STATE_BYTES": "1"}, ["adjoint_level1_pair_kernelILb1", "adjoint_reverse_pair_kernelILb1ELb1"]),
    (366, 300, {"ABP_ADJ_STATE_BYTES": "0"}, ["adjoint_level1_pair_kernelILb1", "adjoint_reverse_pair_kernelILb1ELb0"]),
    (366, 24, {"ABP_ADJ_STATE_BYTES": "0", "ABP_ADJ_HANDOFF_BYTES": "0"},
     ["adjoint_level1_pair_kernelILb0", "adjoint_reverse_pair_kernelILb0ELb0"]),
    (366, 24, {"ABP_ADJ_HANDOFF_BYTES": "0"}, ["adjoint_level1_pair_kernelILb0", "adjoint_reverse_pair_kernelILb0ELb0"]),
])
def test_the_kernels_each_form_launches(child, n_traj, K, env, expect):
    child('''
ctx, grad, dv = integrated(n_traj=(N,), n_steps=(203,), K=KK)
n0 = L.fake_launches()
A.abp_backward(ctx, None, grad)
ks = kernels(n0)
assert "adjoint_final_kernel" in ks[-2] and "adjoint_set_kernel" in ks[-1], ks
names = EXPECT
assert all(any(n in k for n in names) for k in ks[:-2]) and all(any(n in k for k in ks) for n in names), ks
'''.replace("KK", str(K)).replace("(N,)", "(%d,)" % n_traj).replace("EXPECT", repr(expect)), **env)


# the query takes longer than a short backward's launches: only a scratch that has to grow asks
@pytest.mark.parametrize("K", [8, 50])
@pytest.mark.parametrize("form", [{}, {"ABP_ADJ_STATE_BYTES": "0"}], ids=["states", "handoff"])
def test_free_memory_is_asked_for_only_to_grow_the_scratch(child, form, K):
    child('''
ctx, grad, dv = integrated(K=KK)
L.fake_fail(b"cudaMemGetInfo", 0, 0)
A.abp_backward(ctx, None, grad)
assert L.fake_calls() == 1
n0 = L.fake_launches()
A.abp_backward(ctx, None, grad)
assert L.fake_calls() == 1
again = kernels(n0)
# a query that fails leaves the smallest form
ctx, grad, dv = integrated(K=KK)
L.fake_fail(b"cudaMemGetInfo", 0, 1)
n0 = L.fake_launches()
A.abp_backward(ctx, None, grad)
assert L.fake_calls() == 1 and any("reverse_pair_kernelILb0ELb0" in k for k in kernels(n0)), kernels(n0)
assert not any("ILb0ELb0" in k for k in again), again
'''.replace("KK", str(K)), **form)


# what a call takes and keeps: one buffer where one launch covers every segment, the streams and
# events of the groups in use
@pytest.mark.parametrize("form,step_bytes", [({}, 16), ({"ABP_ADJ_STATE_BYTES": "0"}, 0)], ids=["states", "handoff"])
def test_one_launch_takes_one_buffer(child, form, step_bytes):
    child('''
ctx, grad, dv = integrated(n_traj=(3000,), n_steps=(200,), K=40)
before, streams, events = L.fake_live(), L.fake_streams(), L.fake_events()
n0 = L.fake_launches()
A.abp_backward(ctx, None, grad)
assert len(kernels(n0)) == 4, kernels(n0)
used = L.fake_live() - before
if STEP:
    rows = STEP * 200 * 3000
else:  # five segments of 5 sub-checkpoints and 10 blocks of noise for the 12 blocks of 2 x 128 trajectories
    rows = 5 * 5 * 16 * 3000 + 12 * 5 * 10 * 2 * 128 * 16
# and 64 bytes per trajectory, the tile and set sums, each rounded to 256 bytes
assert rows + 64 * 3000 <= used <= rows + 64 * 3000 + 48 * 6 + 56 + 8 * 256, (used, rows)
assert (L.fake_streams() - streams, L.fake_events() - events) == (1, 6)
A.abp_backward(ctx, None, grad)
assert (L.fake_streams() - streams, L.fake_events() - events) == (1, 6)
# a batch of two groups adds the second one's, and a set-up that fails keeps what there was
L.fake_sms(2)
ctx, grad, dv = integrated(n_traj=(40000,), n_steps=(200,), K=40)
L.fake_fail(b"cudaEventCreateWithFlags", 3, 1)
assert status(A.abp_backward, ctx, None, grad) == A.ABP_ECUDA
L.fake_fail(None, 0, 0)
A.abp_backward(ctx, None, grad)
assert (L.fake_streams() - streams, L.fake_events() - events) == (1 + 3, 6 + 10)
A.abp_destroy(ctx)
assert (L.fake_streams() - streams, L.fake_events() - events) == (1, 6)
'''.replace("STEP", str(step_bytes)), **form)


# segments per launch with the hand-off, 152 SMs: level 1 of the next launch and the sweep each keep
# to schedulers of their own ((per + 1) T <= 38,912) while T <= 25,941; beyond, and for tiny
# batches, all ten segments at once
@pytest.mark.parametrize("n_traj,launches", [(100, 1), (3500, 1), (4000, 2), (8000, 4), (12000, 5), (16384, 10),
                                             (25941, 10), (25942, 1)])
def test_handoff_launches_leave_the_sweep_its_schedulers(child, n_traj, launches):
    child('''
ctx, grad, dv = integrated(n_traj=(N,), n_steps=(400,), K=40)
n0 = L.fake_launches()
A.abp_backward(ctx, None, grad)
assert sum("reverse_pair" in k for k in kernels(n0)) == COUNT, kernels(n0)
'''.replace("(N,)", "(%d,)" % n_traj).replace("COUNT", str(launches)), ABP_ADJ_STATE_BYTES="0")


# two groups of tiles: as many blocks of the paired sweep as SMs, and more than two launches or
# three times as many
@pytest.mark.parametrize("n_traj,K,groups", [(38000, 20, 1), (39000, 20, 2), (39000, 200, 1), (116000, 200, 1),
                                             (117000, 200, 2)])
def test_groups_of_tiles(child, n_traj, K, groups):
    child('''
ctx, grad, dv = integrated(n_traj=(N,), n_steps=(400,), K=KK)
n0, streams = L.fake_launches(), L.fake_streams()
A.abp_backward(ctx, None, grad)
assert L.fake_streams() - streams == (1 if GROUPS == 1 else 3), kernels(n0)
'''.replace("(N,)", "(%d,)" % n_traj).replace("KK", str(K)).replace("GROUPS", str(groups)),
          ABP_ADJ_HANDOFF_BYTES="0")
