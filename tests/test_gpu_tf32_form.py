"""The library built with TF32 operator pairs (HPX_TC_F16=0): the adjoint of a batch whose
analysis runs on the tensor cores, against a plan that runs the sweeps."""

import os
import subprocess
import sys

import pytest

from helpers import ROOT

pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

RUN = r"""
import sys
import torch
import paper_1904_10514_gb300 as hp
hp.LIB_PATH = sys.argv[1]
ns, L, B = 32, 57, 16
g = torch.Generator(device="cuda")
g.manual_seed(3)
ops, sweeps = hp.Plan(ns, L, B, "fp32"), hp.Plan(ns, L, B, "fp32", sweeps=True, simt=True)
a = torch.randn(B, ops.nalm, dtype=torch.complex64, device="cuda", generator=g)
for name, tol in (("synthesize", 2e-5), ("analyze_vjp", 2e-5)):
    u, v = getattr(ops, name)(a), getattr(sweeps, name)(a)
    torch.cuda.synchronize()
    print(name, float(torch.linalg.vector_norm(u - v) / torch.linalg.vector_norm(v)) < tol)
"""


def test_tf32_form(tmp_path):
    from paper_1904_10514_gb300 import nvcc_build as nb
    if not all(os.path.exists(os.path.join(nb.OUT, os.path.splitext(s)[0] + ".o")) for s in nb.SOURCES):
        nb.build()
    obj, lib = str(tmp_path / "k_fused_tc.o"), str(tmp_path / "libhpx_tf32.so")
    subprocess.run([nb.NVCC, "-c", os.path.join(nb.CSRC, "k_fused_tc.cu"), "-o", obj, "-O3", "-std=c++17", "-Xcompiler",
                    "-fPIC", "-I" + nb.CSRC, "-DHPX_TC_F16=0"] + nb.ARCH, check=True, capture_output=True)
    objs = [obj if s == "k_fused_tc.cu" else os.path.join(nb.OUT, os.path.splitext(s)[0] + ".o") for s in nb.SOURCES]
    subprocess.run([nb.NVCC, "-shared", "-o", lib] + objs + nb.ARCH + ["-Xcompiler", "-fopenmp", "-lgomp"], check=True,
                   capture_output=True)
    r = subprocess.run([sys.executable, "-c", RUN, lib], cwd=ROOT, capture_output=True, text=True,
                       env=dict(os.environ, PYTHONPATH=ROOT))
    assert r.returncode == 0, r.stderr
    assert r.stdout.split() == ["synthesize", "True", "analyze_vjp", "True"], r.stdout
