"""bench.py's work per kernel class: a solve whose iterations have not been counted reports no work, and the counted
ones their own."""
import bench


def test_solve_classes():
    # 128x128x32 (524,288 nodes) with the Chebyshev solver iterates on FP32 corrections, 256x256 on cells
    assert bench.solve_class("cheb", 524288) == "uncounted"
    assert bench.solve_class("cheb", 65536) == "uncounted"
    assert bench.solve_class("cheb", 399999) == "cheb" and bench.solve_class("cheb", 400000) == "uncounted"
    assert bench.solve_class("dct", 524288) == "dct" and bench.solve_class("cg", 524288) == "cg"
    assert bench.class_work("uncounted", 6, 8.0)["cg"] == (None, None)
    for kind in ("cheb", "cg"):
        ops, byts = bench.class_work(kind, 6, 8.0)["cg"]
        assert ops == bench.CLASS_FP64_OPS[kind + "_iter"] * 8.0 * 24 and byts == bench.CLASS_BYTES[kind + "_iter"] * 8.0 * 24
    others = {k: v for k, v in bench.class_work("dct", 6, 1.0).items() if k != "cg"}
    assert others == {k: v for k, v in bench.class_work("uncounted", 6, 1.0).items() if k != "cg"}
