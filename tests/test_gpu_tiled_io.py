"""Tiles of the tiled sweep in and out of HBM: the read-out of states and
probabilities, and initial states, against the FP64 oracle.  Tolerances as for
every state: entries 1e-4 relative plus 2e-6 absolute, probabilities the same."""
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


@pytest.mark.parametrize("n,tile", [(5, 5), (6, 5), (8, 5), (10, 7), (11, 8), (12, 8), (13, 12), (15, 12)])
def test_tiled_state_read_out(api, orc, n, tile):
    """State and probabilities of the tiled sweep: the linear order it computes
    in turned back, below, at and above the tile of the read-out, FP32 values
    widened exactly (zeros among them: qubits that stay in a basis state)."""
    import torch
    spec = W.CircuitSpec(n)
    r = np.random.default_rng(600 + n)
    k = 0
    for _ in range(3):
        for q in range(n - 1):
            spec.add(("RY", "RX")[q & 1], [q], ("p", k))
            k += 1
        for _ in range(2 * n):
            a, b = r.choice(n - 1, 2, replace=False)
            spec.add("CNOT", [int(a), int(b)])
        spec.add("X", [n - 1])
    params = r.uniform(0, 2 * np.pi, (3, spec.n_params)).astype(np.float32)
    spec.z([0])
    ang = W.resolve_angles(spec, params)
    p = torch.as_tensor(params).cuda()
    for out in ("state", "probs"):
        E = api.Exec(api.Circuit(spec), 3, output=out, max_smem_qubits=1, tile_qubits=tile)
        v, _ = E.run(p)
        torch.cuda.synchronize()
        E.status()
        v = v.cpu().numpy()
        for b in range(3):
            ref = orc.statevector(spec, ang[b])
            if out == "state":
                assert np.array_equal(v[b], v[b].astype(np.float32).astype(np.float64))
                assert np.all(np.abs(v[b, 0::2] + 1j * v[b, 1::2] - ref) <= 1e-4 * np.abs(ref) + 2e-6)
            else:
                assert np.all(np.abs(v[b] - np.abs(ref) ** 2) <= 1e-4 * np.abs(ref) ** 2 + 2e-6)


@pytest.mark.parametrize("n,tile", [(6, 5), (9, 8), (13, 12)])
@pytest.mark.parametrize("shift", [0, 1])
def test_tiled_initial_state_at_any_alignment(api, orc, n, tile, shift):
    """The caller's initial state starts on a 16-byte boundary or 8 bytes off."""
    import torch
    spec, params, _ = W.random_circuit(n, 40, 700 + n, batch=2)
    r = np.random.default_rng(710 + n)
    init = r.normal(size=(2, 1 << n)) + 1j * r.normal(size=(2, 1 << n))
    init = (init / np.linalg.norm(init, axis=1, keepdims=True)).astype(np.complex64)
    buf = torch.zeros((2 << n) + 2, dtype=torch.complex64, device="cuda")
    psi0 = buf[shift:shift + (2 << n)].view(2, 1 << n)
    psi0.copy_(torch.as_tensor(init))
    assert psi0.data_ptr() % 16 == 8 * shift
    E = api.Exec(api.Circuit(spec), 2, output="state", max_smem_qubits=1, tile_qubits=tile)
    E.set_initial_state(psi0)
    v, _ = E.run(torch.as_tensor(params).cuda())
    torch.cuda.synchronize()
    E.status()
    v = v.cpu().numpy()
    ang = W.resolve_angles(spec, params)
    for b in range(2):
        ref = orc.statevector(spec, ang[b], init=init[b].astype(np.complex128))
        assert np.all(np.abs(v[b, 0::2] + 1j * v[b, 1::2] - ref) <= 1e-4 * np.abs(ref) + 2e-6)


@pytest.mark.parametrize("grad", ["none", "adjoint"])
@pytest.mark.parametrize("B", [100, 200, 700])
def test_tiled_passes_at_each_cta_shape(api, orc, B, grad):
    """Forward kernels of 256 and of 128 threads per CTA (12-bit tiles, 1.3 to 9
    tiles per SM), values and gradients of a few rows against the oracle."""
    import torch
    spec, params, _ = W.ladder20(batch=B, n=13, layers=3)
    E = api.Exec(api.Circuit(spec), B, grad=grad, max_smem_qubits=1, tile_qubits=12)
    v, g = E.run(torch.as_tensor(params).cuda())
    torch.cuda.synchronize()
    E.status()
    rows = [0, B // 2, B - 1]
    np.testing.assert_allclose(v.cpu().numpy()[rows], orc.expvals(spec, W.resolve_angles(spec, params[rows])), atol=1e-5)
    if grad == "adjoint":
        ref = orc.param_grads_param_shift(spec, params[B - 1].astype(np.float64))
        np.testing.assert_allclose(g[B - 1].cpu().numpy(), ref, atol=1e-4)


@pytest.mark.parametrize("B,n,tile", [(1, 7, 5), (3, 9, 5), (2, 11, 8)])
def test_shifted_copies_start_at_their_pass(api, orc, B, n, tile):
    """Parameter shift over two to a dozen tile passes, every copy taken over from
    the unshifted one at the pass that holds its angle (U3's three angles in
    passes of their own), against the oracle's shift rule."""
    import torch
    spec, params, _ = W.random_circuit(n, 12 * n, 800 + n, batch=B)
    E = api.Exec(api.Circuit(spec), B, grad="param_shift", max_smem_qubits=1, tile_qubits=tile)
    p = torch.as_tensor(params).cuda()
    for _ in range(2):
        v, g = E.run(p)
    torch.cuda.synchronize()
    E.status()
    np.testing.assert_allclose(v.cpu().numpy(), orc.expvals(spec, W.resolve_angles(spec, params)), atol=1e-5)
    for b in range(B):
        ref = orc.param_grads_param_shift(spec, params[b].astype(np.float64))
        np.testing.assert_allclose(g[b].cpu().numpy(), ref, atol=1e-4)
