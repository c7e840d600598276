"""Adjoint sub-chunks on absolute multiples of 8 steps: segments that start or end inside a chunk
(checkpoint intervals and run lengths that are no multiple of 8) run it one step at a time and take
the noise hand-off for the whole ones, with the bits of the run that draws the noise again."""
import numpy as np
import pytest

from paper_1104_2499_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def abp():
    from paper_1104_2499_gb300 import abp as A
    from paper_1104_2499_gb300 import build as B

    B.build()
    A.lib()
    return A


def grads(abp, K, window=0):
    w = W.Workload(name="chunks", sets=[W.params(D=0.05), W.params(D=0.2, q=2.0), W.params(D=0.1, F0=0.3)],
                   n_traj=[300, 65, 1], n_steps=[203, 64, 7], dt=1e-3, seed=21, v0_mode=1, checkpoint_every=K)
    with abp.Ensemble(w) as ens:
        ens.run()
        return ens.backward(host=True, window=window).numpy(), ens.traj_grad(host=True).numpy()


# one step per segment; inside one chunk; odd; multiples of 4 and 8; longer than every run
@pytest.mark.parametrize("K", [1, 3, 8, 12, 50, 64, 77, 333])
def test_segments_of_any_length(abp, monkeypatch, K):
    ref = grads(abp, 64)[1]
    out = []
    for handoff in ("", "0"):
        monkeypatch.setenv("ABP_ADJ_HANDOFF_BYTES", handoff)
        out.append(grads(abp, K) + grads(abp, K, window=2 * K))
    for a, b in zip(*out):
        np.testing.assert_array_equal(a, b)
    # another K only regroups the FP32 partial sums of a segment: at most 333 terms, 2e-5
    # relative to the sum of their magnitudes
    np.testing.assert_allclose(out[0][1], ref, rtol=0, atol=1e-4 * np.abs(ref).max(axis=0).max())
