"""Which integrator a window launches, on the CPU (tests/helpers/fake_cudart.cpp): windows of one
step take the plain kernel where the FP64 state is otherwise warp-specialised, windows of up to
eight steps one trajectory per thread where packed tiles otherwise hold two."""
import pytest

from test_host_adjoint import child  # noqa: F401  (the library linked with the fake runtime)

CODE = '''
w = W.Workload(name="win", sets=[W.params(D=0.1)] * SETS, n_traj=[TRAJ] * SETS, n_steps=[40] * SETS, dt=1e-3, seed=1, **MODE)
ctx = A.abp_create(A.make_config(w, particles_per_thread=1, schedule=1, steps_per_launch=40, state_fp64=FP64))
A.abp_set_params(ctx, w.sets, w.n_traj, w.n_steps)
got = []
for n in (1, 2, 8, 9, -1):
    n0 = L.fake_launches()
    A.abp_integrate(ctx, n)
    got.append([k for k in kernels(n0)])
for ks, want in zip(got, WANT):
    assert len(ks) == 1 and want in ks[0], got
'''


@pytest.mark.parametrize("sets,traj,mode,fp64,one,two,more", [
    (1, 4096, {}, True, "integrate_kernelIdLi1ELb0", "ws_kernelIdLb0", "ws_kernelIdLb0"),
    (70, 1, {}, True, "integrate_kernelIdLi1ELb1", "ws_kernelIdLb1", "ws_kernelIdLb1"),
    (1, 4096, {}, False, "ws_kernelIfLb0", "ws_kernelIfLb0", "ws_kernelIfLb0"),
    (3000, 20, {}, False, "integrate_kernelIfLi1ELb1", "integrate_kernelIfLi1ELb1",
     "integrate_kernelIfLi2ELb1"),
    (3000, 20, {"scheme": 1}, False, "integrate_kernelIfLi1ELb1", "integrate_kernelIfLi1ELb1",
     "integrate_kernelIfLi2ELb1"),
    (3000, 20, {"noise": 1}, False, "integrate_kernelIfLi1ELb1", "integrate_kernelIfLi1ELb1",
     "integrate_kernelIfLi1ELb1"),
    (3000, 20, {}, True, "integrate_kernelIdLi1ELb1", "integrate_kernelIdLi1ELb1",
     "integrate_kernelIdLi1ELb1"),
])
def test_kernel_of_a_window(child, sets, traj, mode, fp64, one, two, more):  # noqa: F811
    code = CODE.replace("SETS", str(sets)).replace("TRAJ", str(traj)).replace("MODE", repr(mode))
    child(code.replace("FP64", str(fp64)).replace("WANT", repr([one, two, two, more, more])))
