"""Host logic of the products between parents (parent.cu): the planner's tables,
checked on the CPU in a harness compiled with the library's own source (see
tests/cpp/parent_plan_check.cu)."""
import os
import shutil
import subprocess

import pytest

from test_planner import ROOT, _meshes, _write_mesh


@pytest.mark.skipif(shutil.which("nvcc") is None, reason="needs nvcc to compile the host code")
def test_parent_tables(tmp_path):
    from paper_1911_10228_gb300 import build as B
    B.build()
    exe = tmp_path / "parent_plan_check"
    objs = [os.path.join(B.BUILD, n.replace(".cu", ".o")) for n in B.SOURCES if n != "flgf_api.cu"]
    subprocess.run(["nvcc", "-std=c++17", "--expt-relaxed-constexpr", "-gencode", "arch=compute_103a,code=sm_103a",
                    "-I", os.path.join(ROOT, "include"), "-o", str(exe),
                    os.path.join(ROOT, "tests", "cpp", "parent_plan_check.cu")] + objs + ["-lpthread"],
                   check=True, capture_output=True, timeout=900)
    for name, (N, problems) in _meshes().items():
        for ncomp in (1, 3):
            if ncomp > 1 and name == "batch":
                continue
            mesh = tmp_path / f"{name}{ncomp}.bin"
            _write_mesh(mesh, N, problems * ncomp)
            for pct in (0, 30, 100):
                for fp64 in (0, 1):
                    out = subprocess.run([str(exe), str(mesh), str(pct), str(fp64), str(ncomp)], capture_output=True,
                                         text=True, timeout=300)
                    assert out.returncode == 0 and out.stdout.strip().endswith("ok"), (name, ncomp, pct, fp64, out.stdout)
