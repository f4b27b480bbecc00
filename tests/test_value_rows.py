"""Expectations of a few rows of a small circuit, which come from a state of two
floats per number (k2_fine_row): on the host, compiled as
tests/test_specialised_host.py compiles the generated programs, and on the GPU.

Tolerance: what coefficients as good as sincos2's leave, with nothing lost in
the state.  The error d of a half angle's (sin, cos) shifts the angle by 2 d, so
a value moves by 2 d |gradient| (over the angles in quadrature); sincos2's d is
at most 2^-25.4, 2^-28.2 RMS (test_sincos2)."""
import math
import os
import subprocess

import numpy as np
import pytest

import oracle as orc
from paper_2301_05451_gb300 import workloads as W

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HERE = os.path.join(ROOT, "tests", "host_kernels")
KIND = {"H": 0, "X": 1, "Y": 2, "Z": 3, "RX": 4, "RY": 5, "RZ": 6, "U3": 7, "CNOT": 8, "CZ": 9, "RZZ": 10}
MAX_D, RMS_D = 2.0 ** -25.4, 2.0 ** -28.2


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("values") / "values")
    cmd = ["g++", "-std=c++20", "-O1", "-ffp-contract=off", "-fsanitize=address,undefined", "-fno-sanitize-recover=all",
           "-w", "-pthread", "-I" + HERE, "-I" + os.path.join(ROOT, "include"),
           "-I" + os.path.join(ROOT, "paper_2301_05451_gb300", "csrc"), os.path.join(HERE, "values.cpp"), "-o", out]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[:3000]
    return out


def _run(exe, words):
    r = subprocess.run([exe], input=" ".join(map(str, words)), capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[:3000]
    return r.stdout


@pytest.mark.parametrize("reach", [0.8, 2 * math.pi, 6000.0, 1e6])
def test_sincos2(exe, reach):
    """sin and cos as two floats each, near zero, over a turn, to the end of the
    float reduction and past it."""
    x = np.random.default_rng(int(reach)).uniform(-reach, reach, 100000).astype(np.float32)
    got = np.array(_run(exe, [0, len(x)] + [repr(float(v)) for v in x]).split(), dtype=np.float64).reshape(-1, 2)
    d = np.hypot(got[:, 0] - np.sin(x.astype(np.float64)), got[:, 1] - np.cos(x.astype(np.float64)))
    assert d.max() <= MAX_D
    assert np.sqrt(np.mean(d ** 2)) <= RMS_D


def _circuit(name):
    """(spec, rows): angles are parameters, one observable group per term."""
    if name == "hea6":
        spec, n, rows = W.CircuitSpec(6), 6, 24
        p = 0
        for _ in range(3):
            for q in range(n):
                spec.add("RY", [q], ("p", p))
                spec.add("RZ", [q], ("p", p + 1))
                p += 2
            for q in range(n):
                spec.add("CNOT", [q, (q + 1) % n])
        spec.z([0])
        return spec, rows
    n, gates = {"all1": (1, 12), "all2": (2, 30), "all5": (5, 70), "all10": (10, 90), "deep2": (2, 300)}[name]
    spec = W.random_circuit(n, gates, 40 + n, gates=tuple(k for k in KIND if n > 1 or KIND[k] < 8), batch=1,
                            observables=False)[0]
    for q in range(n):
        spec.add("RX", [q], ("p", spec.n_params))
        spec.z([q], 1.0, q)
    return spec, 3


def _reference(spec, params):
    """Values, and the bound of each row and group."""
    v = orc.expvals(spec, W.resolve_angles(spec, params))
    tol = np.zeros_like(v)
    for g in range(spec.n_groups):
        one = W.CircuitSpec(spec.n_qubits)
        one.gates, one.terms, one.n_groups = spec.gates, [(q, c, 0) for q, c, h in spec.terms if h == g], 1
        for b in range(len(params)):
            grad = orc.param_grads_param_shift(one, params[b].astype(np.float64))
            tol[b, g] = 2 * MAX_D * np.linalg.norm(grad) + 1e-12
    return v, tol


CASES = ["hea6", "all1", "all2", "all5", "all10", "deep2"]


@pytest.mark.parametrize("name", CASES)
def test_value_rows_on_the_host(exe, name):
    spec, rows = _circuit(name)
    n, P = spec.n_qubits, spec.n_params
    params = np.random.default_rng(n).uniform(0, 2 * math.pi, (rows, P)).astype(np.float32)
    words = [n, P, rows, spec.n_groups, len(spec.terms), len(spec.gates), 64 if n == 6 else 32]
    for g in spec.gates:
        q = list(g.qubits)
        words += [KIND[g.name], n - 1 - q[0], n - 1 - q[1] if len(q) > 1 else -1, len(g.angles)]
        words += [a[1] for a in g.angles] + [-1] * (3 - len(g.angles))
    for qs, coeff, group in sorted(spec.terms, key=lambda t: t[2]):
        words += [sum(1 << (n - 1 - q) for q in qs), coeff, group]
    out = _run(exe, words + [repr(float(v)) for v in params.reshape(-1)]).split("\n")
    assert out[0] == "status 0"
    v, tol = _reference(spec, params)
    assert np.all(np.abs(np.array(out[1].split(), dtype=np.float64).reshape(v.shape) - v) <= tol)


@pytest.mark.gpu
@pytest.mark.parametrize("rows", [1, 24, 72, 73])
def test_value_rows(rows):
    """A gradient launch with a CTA for the values of every row, up to half the
    SMs and past that (float values, 2e-5); another initial state; the gradients
    beside them."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2301_05451_gb300 import api, build
    build.build()
    spec, n = _circuit("hea6")[0], 6
    params = np.random.default_rng(n).uniform(0, 2 * math.pi, (rows, spec.n_params)).astype(np.float32)
    v, tol = _reference(spec, params)
    fine = 2 * rows + 8 <= torch.cuda.get_device_properties(0).multi_processor_count
    E = api.Exec(api.Circuit(spec), rows, grad="adjoint")
    p = torch.as_tensor(params).cuda()
    for _ in range(2):
        got, g = E.run(p)
    torch.cuda.synchronize()
    E.status()
    assert np.all(np.abs(got.cpu().numpy() - v) <= (tol if fine else 2e-5))
    for b in (0, rows - 1):
        ref = orc.param_grads_param_shift(spec, params[b].astype(np.float64))
        np.testing.assert_allclose(g[b].cpu().numpy(), ref, atol=5e-5)
    psi0 = np.zeros((rows, 1 << n), np.complex64)
    psi0[np.arange(rows), np.arange(rows) % (1 << n)] = 1j
    E.set_initial_state(torch.as_tensor(psi0).cuda())
    got, _ = E.run(p)
    E.status()
    ang = W.resolve_angles(spec, params)
    sign = 1 - 2.0 * (np.arange(1 << n) >> (n - 1))
    for b in (0, rows - 1):
        ref = (np.abs(orc.statevector(spec, ang[b], init=psi0[b].astype(np.complex128))) ** 2 * sign).sum()
        assert abs(got[b, 0].item() - ref) <= (2 * MAX_D * math.sqrt(spec.n_params) if fine else 2e-5)
