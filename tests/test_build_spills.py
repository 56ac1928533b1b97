"""The build refuses register spills beyond what the kernels that fill the register file
are known to have."""
import pytest

from paper_1704_00512_gb300 import build

LINES = """ptxas info    : Compiling entry function '_ZN4cheb9k_colstepIfEEvNS_7ColArgsE' for 'sm_103a'
ptxas info    : Function properties for _ZN4cheb9k_colstepIfEEvNS_7ColArgsE
    48 bytes stack frame, {f32} bytes spill stores, 0 bytes spill loads
ptxas info    : Used 128 registers, used 1 barriers, 48 bytes cumulative stack size
ptxas info    : Function properties for _ZN4cheb9k_colstepIdEEvNS_7ColArgsE
    64 bytes stack frame, {f64} bytes spill stores, 12 bytes spill loads
"""


def test_spills_are_read_by_function():
    assert build.spills(LINES.format(f32=0, f64=8)) == {"_ZN4cheb9k_colstepIfEEvNS_7ColArgsE": 0,
                                                        "_ZN4cheb9k_colstepIdEEvNS_7ColArgsE": 8}


@pytest.mark.parametrize("f32,f64,ok", [(0, 0, True), (12, 0, True), (0, 4, False), (16, 0, False)])
def test_the_limits(f32, f64, ok):
    text = LINES.format(f32=f32, f64=f64)
    if ok:
        build.check_spills("csrc/colstep.cu", text)
    else:
        with pytest.raises(RuntimeError, match="spills"):
            build.check_spills("csrc/colstep.cu", text)
    build.check_spills("csrc/mlp.cu", text)  # (a source without limits)


def test_a_silent_compiler_is_refused():
    with pytest.raises(RuntimeError, match="no function"):
        build.check_spills("csrc/product.cu", "")
