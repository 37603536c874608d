"""The bench's issue-rate roofline of the FP64 kernels: a number only where the
kernels' instructions have been counted."""
import bench


def test_issue_roofline(monkeypatch):
    monkeypatch.setattr(bench, "WARP_INSTR_PER_32_TETS", {"fwd_fp64": 4000, "vjp_fp64": None})
    r = bench.issue_roofline("fwd_fp64", 10.0, 32_000_000, 100, 2000.0, default=True)
    assert r["peak"] == 800.0 and r["achieved"] == 400.0 and r["frac"] == 0.5
    # another formulation, a kernel changed since it was counted
    for key, default in (("fwd_fp64", False), ("vjp_fp64", True)):
        r = bench.issue_roofline(key, 10.0, 32_000_000, 100, 2000.0, default=default)
        assert r["achieved"] is None and r["frac"] is None and r["warp_instr_per_32_tets"] is None
