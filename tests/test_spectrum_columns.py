"""Host logic of the block set's spectrum buffers: the device lists name spectrum
columns, which only the blocks with a spectrum of their own have, checked on
the CPU in a harness compiled with the library's own source (see
tests/cpp/spectrum_columns_check.cu)."""
import os
import shutil
import subprocess

import numpy as np
import pytest

from paper_1911_10228_gb300.inputs import box_coords
from test_planner import ROOT, _meshes, _write_mesh


@pytest.mark.skipif(shutil.which("nvcc") is None, reason="needs nvcc to compile the host code")
def test_spectrum_columns(tmp_path):
    from paper_1911_10228_gb300 import build as B
    B.build()
    exe = tmp_path / "spectrum_columns_check"
    objs = [os.path.join(B.BUILD, n.replace(".cu", ".o")) for n in B.SOURCES if n != "flgf_api.cu"]
    subprocess.run(["nvcc", "-std=c++17", "--expt-relaxed-constexpr", "-gencode", "arch=compute_103a,code=sm_103a",
                    "-I", os.path.join(ROOT, "include"), "-o", str(exe),
                    os.path.join(ROOT, "tests", "cpp", "spectrum_columns_check.cu")] + objs + ["-lpthread"],
                   check=True, capture_output=True, timeout=900)
    passes = 0
    meshes = _meshes()
    box = box_coords(14)
    meshes["scattered"] = (8, [[box[np.random.default_rng(0).random(len(box)) < 0.6]]])
    for name, (N, problems) in meshes.items():
        for ncomp in (1, 3):
            if ncomp > 1 and name == "batch":
                continue
            mesh = tmp_path / f"{name}{ncomp}.bin"
            _write_mesh(mesh, N, problems * ncomp)
            for pct in (30, 100):
                for fp64, mac in ((0, 1), (0, 2), (0, 0), (1, 1)):
                    for most in (0, 256 << 20):
                        out = subprocess.run([str(exe), str(mesh), str(pct), str(fp64), str(mac), str(ncomp), str(most)],
                                             capture_output=True, text=True, timeout=300)
                        what = (name, ncomp, pct, fp64, mac, most, out.stdout)
                        assert out.returncode == 0 and out.stdout.strip().endswith("ok"), what
                        if name == "scattered":
                            passes = max(passes, int(out.stdout.split("passes ")[1].split()[0]))
    assert passes > 2  # one phase and its adjoint: more where the bound cuts them
