"""The default method of complex128 states returns while its kernels run; what they report comes with a later call."""
import os
import shutil
import subprocess

import numpy as np
import pytest

import workloads as W
from conftest import ROOT


def test_reported_once(tmp_path):
    if shutil.which("g++") is None:
        pytest.skip("g++ not available")
    from paper_2008_13490_gb300 import _build
    lib = _build.build()
    libdir = os.path.dirname(lib)
    exe = tmp_path / "late_status_check"
    cuda_inc = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
    subprocess.run(["g++", "-O1", "-std=c++17", os.path.join(ROOT, "tests", "late_status_check.cpp"),
                    "-I", os.path.join(ROOT, "paper_2008_13490_gb300", "csrc"), "-I", os.path.join(ROOT, "include"),
                    "-I", cuda_inc, "-o", str(exe), "-L", libdir, "-lqsim", f"-Wl,-rpath,{libdir}"],
                   check=True, capture_output=True, text=True)
    assert subprocess.run([str(exe)]).returncode == 0


@pytest.mark.gpu
def test_complex128_calls_do_not_wait(qs):
    # 25 qubits, 40 layers: some 30 ms on the device, a few on the host.  Two states on streams of their own: the
    # second call returns while the first state's kernels still run
    import torch
    n = 25
    gates = qs.gates_array(W.layered_haar_cz(n, 40, seed=3))
    streams = [torch.cuda.Stream() for _ in range(2)]
    states = [qs.State(n, qs.QS_C128, stream=s) for s in streams]
    for st in states:   # buffers
        qs.sv_apply_circuit(st, gates)
    torch.cuda.synchronize()
    first = [qs.sv_probs(st, fp64=True, marg_mask=0xff)[0].cpu().numpy() for st in states]
    for st in states:
        qs.sv_set_basis(st, 0)
    stats = [qs.sv_apply_circuit(st, gates) for st in states]
    running = [not s.query() for s in streams]
    assert stats[0]["tile_launches"] == 0 and all(running)
    torch.cuda.synchronize()
    again = [qs.sv_probs(st, fp64=True, marg_mask=0xff)[0].cpu().numpy() for st in states]
    for st in states:
        st.close()
    assert np.allclose(again[0], again[1], rtol=0, atol=1e-12) and np.allclose(first[0], first[1], rtol=0, atol=1e-12)
    assert abs(again[0].sum() - 1) < 1e-12
