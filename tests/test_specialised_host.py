"""The specialised sweep programs run on the host: the generated source of a
circuit (tdq_sweep_source) is compiled with a host compiler against stand-ins
for the CUDA headers (tests/host_kernels) and run one CTA at a time, one host
thread per CUDA thread, with a guard behind the shared memory.  Values,
adjoint gradients and final states against the FP64 oracle: every gate kind,
CNOT circuits (whose gates pair far-apart indices in the linear frame), CZ
between register, group and tile bits, tied parameters, angles at the edges of
the two rotation forms, states smaller than a register group.

Tolerances: FP32 rounding of at most 200 gates on unit-norm states, 200 x 2^-24
x 4 = 5e-5 on gradients (which add two states' errors), 2e-5 on values and
amplitudes."""
import math
import os
import re
import subprocess

import numpy as np
import pytest

import oracle as orc
from paper_2301_05451_gb300 import workloads as W

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HERE = os.path.join(ROOT, "tests", "host_kernels")
KIND = {"H": 0, "X": 1, "Y": 2, "Z": 3, "RX": 4, "RY": 5, "RZ": 6, "U3": 7, "CNOT": 8, "CZ": 9, "RZZ": 10}


def _dense(n, n_gates, seed, kinds, batch=2):
    spec, params, _ = W.random_circuit(n, n_gates, seed, gates=kinds, batch=batch, observables=False)
    for q in range(n):  # ends in rotations: nothing to fold into the observable
        spec.add("RX", [q], ("p", spec.n_params))
    params = np.random.default_rng(seed).uniform(0, 2 * math.pi, size=(batch, spec.n_params)).astype(np.float32)
    for q in range(n):
        spec.z([q], 1.0, q)
    if n > 1:
        spec.z([0, n - 1], 0.5, 0)
    return spec, params


ALL = tuple(KIND)


def _case(name):
    """(spec, params, tile bits, adjoint)"""
    if name.startswith("all"):
        n, tile = {"all1": (1, 0), "all2": (2, 0), "all3": (3, 0), "all6": (6, 0), "all7_tiled": (7, 5),
                   "all9_tiled": (9, 5), "all10_tiled": (10, 7)}[name]
        return _dense(n, 12 * n, 70 + n, ALL if n > 1 else ("H", "X", "Y", "Z", "RX", "RY", "RZ", "U3")) + (tile, True)
    if name == "cnot8":
        return _dense(8, 90, 81, ("RY", "RZ", "CNOT")) + (0, True)
    if name == "cnot9_tiled":
        return _dense(9, 100, 82, ("RY", "RX", "RZ", "CNOT")) + (6, True)
    if name == "cz8":
        return _dense(8, 90, 83, ("RY", "RX", "RZ", "H", "CZ", "Z")) + (0, True)
    if name == "cz9_tiled":
        return _dense(9, 100, 84, ("RY", "H", "RZZ", "CZ", "U3")) + (6, True)
    if name == "real7":  # no phases: the scale is applied by itself
        return _dense(7, 60, 85, ("RY", "H", "CNOT")) + (0, True)
    if name in ("tied6", "tied7_tiled"):
        n, tile = (6, 0) if name == "tied6" else (7, 5)
        spec, params, _ = W.random_circuit_tied(n, 10 * n, 5, 86 + n, batch=2)
        for q in range(n):
            spec.add("RX", [q], ("p", q % 5))
        return spec, params, tile, True
    if name in ("edges5", "edges7_tiled"):  # angles where the rotation forms meet and their ends
        n, tile = (5, 0) if name == "edges5" else (7, 5)
        spec, params = _dense(n, 10 * n, 90 + n, ("RY", "RX", "RZ", "U3", "CNOT", "CZ"))
        e = np.array([0, math.pi / 2, -math.pi / 2, math.pi, -math.pi, 2 * math.pi, 3 * math.pi / 2, 1e-7, 0.75])
        return spec, e[np.random.default_rng(9).integers(len(e), size=params.shape)].astype(np.float32), tile, True
    if name in ("state6", "state9_tiled"):  # no observable: the final state, global phase kept
        n, tile = (6, 0) if name == "state6" else (9, 5)
        return W.random_circuit(n, 12 * n, 95 + n, gates=ALL, batch=2, observables=False)[:2] + (tile, False)
    raise AssertionError(name)


CASES = ["all1", "all2", "all3", "all6", "all7_tiled", "all9_tiled", "all10_tiled", "cnot8", "cnot9_tiled", "cz8",
         "cz9_tiled", "real7", "tied6", "tied7_tiled", "edges5", "edges7_tiled", "state6", "state9_tiled"]


@pytest.mark.parametrize("name", CASES)
def test_program_on_the_host(name, tmp_path):
    from paper_2301_05451_gb300 import api, build
    build.build()
    spec, params, tile, adj = _case(name)
    n, rows = spec.n_qubits, params.shape[0]
    src = api.Circuit(spec).specialised_source("adjoint" if adj else "none", tile_qubits=tile)
    (tmp_path / "gen.inc").write_text(src)
    head = open(os.path.join(ROOT, "paper_2301_05451_gb300", "csrc", "engine.cuh")).read()
    bits = [int(re.search(r"%s = (\d+);" % v, head).group(1)) for v in (
        "kTiledSpecFwdRegBits", "kTiledSpecRevRegBits")] if tile else [2, 2]  # whole states below 11 qubits
    fwd = re.findall(r"(tdq_k1f_\d+)\(", src)
    rev = re.findall(r"(tdq_k1r_\d+)\(", src)
    exe = str(tmp_path / "run")
    cmd = ["g++", "-std=c++20", "-O1", "-fsanitize=address,undefined", "-fno-sanitize-recover=all", "-w", "-pthread",
           "-DGENERATED=\"%s\"" % (tmp_path / "gen.inc"), "-I" + HERE, "-I" + os.path.join(ROOT, "include"),
           "-I" + os.path.join(ROOT, "paper_2301_05451_gb300", "csrc"), os.path.join(HERE, "run.cpp"), "-o", exe]
    cmd += ["-DFWD_KERNELS=" + ",".join(fwd), "-DREV_KERNELS=" + ",".join(rev or ["nullptr"])] if tile else ["-DWHOLE"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[:3000]
    P = spec.n_params
    ng = spec.n_groups
    words = [n, tile, bits[0], bits[1], int(adj), P, rows, ng, len(spec.terms), len(spec.gates)]
    for g in spec.gates:
        q = list(g.qubits)
        srcs = [a[1] if a[0] == "p" else -1 for a in g.angles] + [-1] * (3 - len(g.angles))
        words += [KIND[g.name], n - 1 - q[0], n - 1 - q[1] if len(q) > 1 else -1, len(g.angles)] + srcs + srcs
    for qs, coeff, group in sorted(spec.terms, key=lambda t: t[2]):
        words += [sum(1 << (n - 1 - q) for q in qs), coeff, group]
    words += [repr(float(v)) for v in params[:, :P].reshape(-1)]
    r = subprocess.run([exe], input=" ".join(map(str, words)), capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[:3000]
    lines = r.stdout.split("\n")
    assert lines[0] == "status 0"
    got = np.array(lines[1].split(), dtype=np.float64)
    ang = W.resolve_angles(spec, params)
    if not adj:
        for b in range(rows):
            v = got.reshape(rows, -1, 2)[b]
            np.testing.assert_allclose(v[:, 0] + 1j * v[:, 1], orc.statevector(spec, ang[b]), atol=2e-5)
        return
    np.testing.assert_allclose(got.reshape(rows, ng), orc.expvals(spec, ang), atol=2e-5)
    grads = np.array(lines[2].split(), dtype=np.float64).reshape(rows, -1)
    for b in range(rows):
        np.testing.assert_allclose(grads[b][:P], orc.param_grads_param_shift(spec, params[b].astype(np.float64)), atol=5e-5)
