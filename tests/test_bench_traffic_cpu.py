"""bench.py reports the stored DRAM traffic of the kernel that it names: the
residual kernel of the degree-1 cycle, from that kernel's file."""
import json
import types

import bench


def test_traffic_of_the_named_kernel(tmp_path, monkeypatch):
    mesh = types.SimpleNamespace(entries=15000, prior_entries=7000)
    acc = {k: {"ms": 10.0, "iters": 4, "rhs_iters": 64, "launches": 1, "fine_ms": 2.0, "fine_launches": 4} for k in ("pair", "prior")}
    prm = types.SimpleNamespace(multigrid=1, mg_degree=1)
    kern, peak = bench.mg_kernel_table({"mesh": mesh, "N": 1000, "K": 8}, prm, acc, 2070.0, 152, 6000.0, 20.0)
    assert kern["pair"]["kernel"].startswith("k_level<double, 16, 1, 0, 1, 1>")
    (tmp_path / "profiles").mkdir()
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    monkeypatch.setattr(bench, "kernel_source_sha1", lambda files=None: "abc")
    for name, n in (("k_cheb", 1), ("k_level", 2)):
        (tmp_path / "profiles" / f"{name}_w_traffic.json").write_text(
            json.dumps({"source_sha1": "abc", "kernels": {"pair_fp64": {"dram_bytes_per_launch": n}}}))
    assert bench.mg_roofline(kern, "pair", peak, 6000.0, "measured", 2070.0, 152, "w")["traffic"] == 2
