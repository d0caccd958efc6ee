"""How the units are compiled."""
from paper_1410_3464_gb300 import build


def test_fp64_unit_is_compiled_without_contraction():
    """Every instantiation of the FP64 kernels has to give the same bits."""
    for src in build.SOURCES:
        cmd = build.compile_command(src)
        assert ("-fmad=false" in cmd) == (src == "kernels_f64.cu"), src
        assert cmd[1:3] == ["-gencode", "arch=compute_103a,code=sm_103a"]
