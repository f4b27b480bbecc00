"""The sum of a row's slices in the last launch of a values-only plan: few slices
(a thread per row), many (a block per row) and more than a block reads at a time,
with the roots in a workspace and written by the subtrees, against the FP64
oracle.  Tolerances as for every amplitude (1e-4 relative plus 2e-6) and value."""
import numpy as np
import pytest

from paper_2301_05451_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2301_05451_gb300 import build
    build.build()
    from paper_2301_05451_gb300 import api as _api
    return _api


@pytest.mark.parametrize("subtree", [1, 11])
@pytest.mark.parametrize("target,slices", [(8, 8), (7, 16), (6, 64), (5, 512)])
def test_sum_of_slices(api, orc, target, slices, subtree):
    import torch
    spec, _, _ = W.grid_u3cz(seed=1, rows=4, cols=4, depth=8)
    params = np.random.default_rng(slices).uniform(0, 2 * np.pi, (3, spec.n_params)).astype(np.float32)
    N = api.Network(api.Circuit(spec), "amplitude", 0, hyper=True)
    E = api.TreeExec(api.Plan(N, method="greedy", target_log2=target), 3, subtree_log2=subtree)
    assert E.config()["chunk"] == slices
    v, _ = E.run(torch.as_tensor(params).cuda())
    torch.cuda.synchronize()
    E.status()
    v = v.cpu().numpy()
    ref = orc.amplitudes(spec, W.resolve_angles(spec, params))[:, 0]
    assert np.all(np.abs(v[:, 0] + 1j * v[:, 1] - ref) <= 1e-4 * np.abs(ref) + 2e-6)


def test_sum_of_slices_of_a_value(api, orc):
    import torch
    spec, _, _ = W.grid_brickwork(rows=3, cols=3, layers=4, observed=4)
    params = np.random.default_rng(9).uniform(0, 2 * np.pi, (2, spec.n_params)).astype(np.float32)
    N = api.Network(api.Circuit(spec), "expval", 0, lightcone=True)
    E = api.TreeExec(api.Plan(N, method="greedy", target_log2=3), 2)
    assert E.config()["chunk"] == 512
    v, _ = E.run(torch.as_tensor(params).cuda())
    torch.cuda.synchronize()
    E.status()
    np.testing.assert_allclose(v.cpu().numpy(), orc.expvals(spec, W.resolve_angles(spec, params)), atol=1e-5)
