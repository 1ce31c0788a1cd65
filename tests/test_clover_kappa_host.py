"""The clover force's per-link plaquette sum from the field that the library keeps,
kappa_k = Re tr(s_k K_mn) (hr_clover_leaf.cuh, KappaField, the native FP64 path of
the force kernel), compiled as plain C++ on the host, against the oracle's
leaf-by-leaf derivative."""

import shutil
import subprocess

import numpy as np
import pytest

import oracle
import synth
from oracle import clover as ocl
from tests.test_clover_leaf_host import CSRC, PLANES, PROGRAM

SIGMA = np.array([[[0, 1], [1, 0]], [[0, -1j], [1j, 0]], [[1, 0], [0, -1]]])


@pytest.mark.parametrize("dims", [(2, 2, 2, 4), (4, 2, 4, 2), (4, 4, 2, 6)])
def test_kappa_field_matches_leaf_by_leaf(tmp_path, dims):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no host C++ compiler")
    program = PROGRAM.replace("K(48 * V)", "K(18 * V)").replace("K.data(), rho", "KappaField{K.data(), V}, rho")
    assert program.count("KappaField") == 1 and "K(18 * V)" in program
    src, exe = tmp_path / "kappa.cpp", tmp_path / "kappa"
    src.write_text(program)
    subprocess.run([gxx, "-O2", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    V = int(np.prod(dims))
    rng = np.random.default_rng(711)
    q = synth.haar_links(dims, 712)
    lam = rng.normal(size=(V, 8, 8)) + 1j * rng.normal(size=(V, 8, 8))
    L4 = lam.reshape(V, 4, 2, 4, 2)
    K = np.stack([np.einsum("st,xtbsa->xba", ocl.sigma(mu, nu), L4) for mu, nu in PLANES])  # [6, V, 2, 2]
    kappa = np.einsum("kab,pxba->pkx", SIGMA, K).real
    inp, out = tmp_path / "in.bin", tmp_path / "out.bin"
    inp.write_bytes(np.asarray(dims, dtype=np.int32).tobytes() + np.ascontiguousarray(q).tobytes()
                    + np.ascontiguousarray(kappa).tobytes())
    subprocess.run([str(exe), str(inp), str(out)], check=True)
    F = np.fromfile(out, dtype=np.float64).reshape(4, V, 3)
    want = ocl.clover_derivative(dims, oracle.expand_links(dims, 2, q), lam)
    assert np.linalg.norm(F - want) <= 1e-13 * np.linalg.norm(want)
