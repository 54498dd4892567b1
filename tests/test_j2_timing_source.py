"""hom_j2_time_kernels times the passes that the increments run (op_geom's), not the other solves'."""
import os

SRC = open(os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2110_00733_gb300", "csrc",
                        "hom_api.cu")).read()


def test_timed_passes_are_the_increments():
    impl = SRC[SRC.index("static int j2_time_impl("):SRC.index("int hom_j2_time_kernels(")]
    assert "op_geom(ctx, E)" in impl and "E.g," not in impl
    call = SRC[SRC.index("int hom_j2_time_kernels("):]
    call = call[:call.index("\n}\n")]
    assert call.index("ctx->j2_ops = true") < call.index("j2_time_impl<double>") < call.index("ctx->j2_ops = false")
