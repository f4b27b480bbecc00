"""The kernels of a tree plan's steps, one chosen shape at a time: a path that
contracts two blocks of a circuit whose product has 2^nm x 2^nn entries, summed
over 2^nk, in a kernel of its own, against the FP64 oracle's amplitudes.
Tolerance as for every amplitude: 1e-4 relative plus 2e-6 (a step's sum rounds
like the unit-norm state's)."""
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


def _blocks(n, opened, nk, nn):
    """n qubits; block L: gates on all of them and the inputs of qubits
    `opened`..n-1; block R: gates on qubits 0..nk-1 and the outputs of qubits
    nn..nk-1.  L x R: nm = opened + n - nk, nn, nk."""
    c = W.CircuitSpec(n)
    p, left = 0, 0
    for width in (n, nk):
        left = left or len(c.gates)
        for q in range(width):
            c.add("RY", [q], ("p", p))
            c.add("RZ", [q], ("p", p + 1))
            p += 2
        for q in range(width - 1):
            c.add("CNOT", [q, q + 1])
        for q in range(width):
            c.add("RX", [q], ("p", p))
            p += 1
    c.amplitude([q & 1 for q in range(n)])
    return c, left


def _path(N, n, left, opened, nk, nn):
    T = [N.tensor(i) for i in range(N.n_tensors)]
    ends = {}
    groups = {"L": [], "R": [], "rest": []}
    n_in = n_out = 0
    for i, t in enumerate(T):
        if t["gate"] >= 0:
            groups["L" if t["gate"] < left else "R"].append(i)
        elif n_in < n:
            groups["L" if n_in >= opened else "rest"].append(i)
            n_in += 1
        else:
            groups["R" if nn <= n_out < nk else "rest"].append(i)
            n_out += 1
    assert n_in == n and n_out == n
    idx = {i: set(t["idx"]) for i, t in enumerate(T)}
    path, nxt = [], N.n_tensors

    def merge(a, b):
        nonlocal nxt
        path.append((a, b))
        idx[nxt] = idx[a] ^ idx[b]
        nxt += 1
        return nxt - 1

    def block(ids):
        ids = list(ids)
        cur = ids.pop(0)
        while ids:
            j = next((k for k in ids if idx[k] & idx[cur]), ids[0])
            ids.remove(j)
            cur = merge(cur, j)
        return cur

    a, b = block(groups["L"]), block(groups["R"])
    shape = (len(idx[a] - idx[b]), len(idx[b] - idx[a]), len(idx[a] & idx[b]))
    block([merge(a, b)] + groups["rest"])
    return path, shape


# (qubits, nm, nn, nk, batch): thread-, warp- and 64 x 64-tile shapes in 16 x 16
# and 32 x 32 tiles (k below, at and above a staged chunk), tiles narrower than
# their square on either side, tensor-core shapes on both sides of the size rule,
# k split over blocks with and without a sum of blocks
SHAPES = [(8, 5, 3, 3, 3), (8, 4, 4, 7, 2), (9, 9, 0, 6, 1), (8, 2, 6, 6, 5), (9, 1, 7, 8, 2), (7, 5, 5, 6, 1),
          (6, 5, 5, 5, 130), (7, 7, 6, 7, 1), (9, 8, 6, 7, 9), (10, 7, 7, 10, 1), (8, 5, 5, 8, 1), (8, 6, 5, 8, 160),
          (10, 5, 6, 9, 3), (8, 4, 4, 8, 2), (9, 0, 3, 9, 4), (8, 2, 2, 8, 3), (9, 6, 5, 5, 33), (8, 4, 4, 6, 400)]


@pytest.mark.parametrize("plain", [False, True])
@pytest.mark.parametrize("n,nm,nn,nk,B", SHAPES)
def test_step_shapes(api, orc, n, nm, nn, nk, B, plain):
    import torch
    spec, left = _blocks(n, nm - (n - nk), nk, nn)
    params = np.random.default_rng(100 * n + nm).uniform(0, 2 * np.pi, (B, spec.n_params)).astype(np.float32)
    N = api.Network(api.Circuit(spec), "amplitude", 0)
    path, shape = _path(N, n, left, nm - (n - nk), nk, nn)
    assert shape == (nm, nn, nk)
    E = api.TreeExec(api.Plan(N, path=path), B, plain=plain, subtree_log2=1)
    p = torch.as_tensor(params).cuda()
    for _ in range(2):
        v, _ = E.run(p)
    torch.cuda.synchronize()
    E.status()
    v = v.cpu().numpy()
    ref = orc.amplitudes(spec, W.resolve_angles(spec, params))[:, 0]
    assert np.all(np.abs(v[:, 0] + 1j * v[:, 1] - ref) <= 1e-4 * np.abs(ref) + 2e-6)


@pytest.mark.parametrize("B", [2, 67])
def test_step_shapes_with_hyperedges(api, orc, B):
    import torch
    spec, params, _ = W.random_circuit(9, 80, 5100 + B, batch=B, amplitudes=1,
                                       gates=("H", "RX", "RY", "RZ", "CZ", "RZZ", "CNOT"))
    N = api.Network(api.Circuit(spec), "amplitude", 0, hyper=True)
    E = api.TreeExec(api.Plan(N), B, subtree_log2=1)
    v, _ = E.run(torch.as_tensor(params).cuda())
    torch.cuda.synchronize()
    E.status()
    v = v.cpu().numpy()
    ref = orc.amplitudes(spec, W.resolve_angles(spec, params))[:, 0]
    assert np.all(np.abs(v[:, 0] + 1j * v[:, 1] - ref) <= 1e-4 * np.abs(ref) + 2e-6)


@pytest.mark.parametrize("target", [0, 3])
@pytest.mark.parametrize("B", [1, 310, 700])
def test_fused_gradient_row_counts(api, orc, B, target):
    """The one-CTA value and gradient at each of its thread counts, with one
    slice (outputs written by the CTA) and several (summed after it)."""
    import torch
    spec, params, _ = W.random_circuit(5, 30, 5200, batch=B)
    qs, coeff, _ = spec.terms[0]
    single = W.CircuitSpec(spec.n_qubits)
    single.gates, single.terms, single.n_groups = spec.gates, [(qs, coeff, 0)], 1
    N = api.Network(api.Circuit(spec), "expval", 0, hyper=True)
    E = api.TreeExec(api.Plan(N, target_log2=target), B, grad="adjoint")
    assert E.config()["reverse"] == 1
    v, g = E.run(torch.as_tensor(params).cuda().contiguous())
    torch.cuda.synchronize()
    E.status()
    rows = sorted({0, B // 2, B - 1})
    ang = W.resolve_angles(spec, params[rows])
    np.testing.assert_allclose(v.cpu().numpy()[rows, 0], orc.expvals(single, ang)[:, 0], atol=1e-5)
    for b in rows:
        ref = orc.param_grads_param_shift(single, params[b].astype(np.float64))
        np.testing.assert_allclose(g[b].cpu().numpy(), ref, atol=1e-4)
