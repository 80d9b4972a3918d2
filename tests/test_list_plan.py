"""The reach of FLGF_CTX_LIST_PCT, on the CPU (harness of test_planner.py)."""
import subprocess

from test_planner import _meshes, _write_mesh, harness  # noqa: F401 (fixture)


def test_every_tile_that_is_not_full_can_go_to_the_lists(harness, tmp_path):  # noqa: F811
    """At 100 the plans with products between parents list at least what the
    child-pair plan does: every tile with an absent block among its pairs."""
    for name, (N, problems) in _meshes().items():
        mesh = tmp_path / f"{name}.bin"
        _write_mesh(mesh, N, problems)
        listed = {}
        for fp64, mac in ((0, 0), (0, 1), (0, 2), (1, 0)):
            out = subprocess.run([str(harness), str(mesh), "100", "2", "4", "8", str(fp64), str(mac)],
                                 capture_output=True, text=True, timeout=300)
            assert out.returncode == 0, (name, out.stdout)
            listed[fp64, mac] = int(out.stdout.split("pair lists ")[1].split(")")[0])
        assert all(n >= listed[0, 0] for n in listed.values()), (name, listed)
