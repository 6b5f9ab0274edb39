"""bench.py's byte model and roofline of the CG on coefficients (no GPU)."""
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

import bench  # noqa: E402

FS = ("fs_x1i_cg_f32", "fs_p4_grad_f32", "fs_rows_cg_f32", "fs_p2_grad_f32", "fs_x1f_cg_f32", "fs_cg_rr_f32")


def test_byte_model():
    # 243^3: a spectrum of six components 24.1 B a voxel, a vector half of it
    b = bench.bytes_per_voxel(243)
    assert abs(sum(b[k + "_f32"] for k in bench.DC_KINDS) - 305.1) < 0.1
    f = bench.fs_bytes_per_voxel(243)
    assert abs(sum(f[k] for k in FS) - 362.2) < 0.2


def test_roofline():
    # 100 CG field-iterations, 5 Newton iterations, one tangent: P2 runs once
    # more for each of the tangent's six right-hand sides, P4 once for each
    # solution; every kernel at 1 ms per field launch
    eff = {"x1i_cg": 100, "rows_cg": 100, "x1f_cg": 100, "cg_rr": 100, "p2": 106, "p4": 111}
    prof = {k + "_f32": (float(n), n + 3) for k, n in eff.items()}
    rf = bench.cg_roofline(prof, 243, 100, 5, 1, "_f32", hbm=1000.0)
    assert set(rf["kernels"]) == set(eff)
    for k in eff:
        assert rf["kernels"][k]["ms"] == 1.0
        assert abs(rf["kernels"][k]["GB/s"] - bench.bytes_per_voxel(243)[k + "_f32"] * 243 ** 3 / 1e-3 / 1e9) < 0.1
    assert rf["matvec"]["ms_per_field_iter"] == 5.0 and rf["iteration"]["ms_per_field_iter"] == 6.0
    assert abs(rf["iteration"]["bytes_per_voxel"] - 305.1) < 0.2
