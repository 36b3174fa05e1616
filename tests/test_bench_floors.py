"""The bench's floors of the fixed-point kernels: the local terms are priced by the instructions that the kernels execute."""
import bench

INFO = dict(nx=512, ny=256, nz=4, px=1024, py=512, pz=8, bulk_layout=0, spectrum_bytes=25214976, tensor_bytes=33750528)
FMA = {"fp64": 1.06, "fp32": 73.0}   # TFLOP/s


def floors(precision):
    model = bench.algorithmic_model(INFO, 8)
    return {s: {k: v[0] / (v[1] * 1e6) for k, v in bench.fixed_point_work(model, INFO, s, precision, FMA, 13.2).items()}
            for s in ("xfwd_step", "yz_conv", "xinv_local_bb")}   # us


def test_local_terms_are_counted_instructions():
    f = floors("fp64")
    # 524 288 cells x 103 instructions at 0.53 T/s
    assert abs(f["xinv_local_bb"]["alu_local"] - 524288 * 103 / 0.53e6) < 1e-6
    assert 95 < f["xinv_local_bb"]["alu_local"] < 110 and f["yz_conv"]["alu_local"] == 0
    f = floors("f32x2")
    assert abs(f["xinv_local_bb"]["alu_local"] - 524288 * 1254 / 36.5e6) < 1e-6


def test_transforms_leave_the_local_terms_out():
    for p in ("fp64", "f32x2"):
        model = bench.algorithmic_model(INFO, 8)
        w = bench.fixed_point_work(model, INFO, "xinv_local_bb", p, FMA, 13.2)
        assert w["alu_int64"][0] == model["xinv_local_bb"]["flops"] - 90 * 524288
