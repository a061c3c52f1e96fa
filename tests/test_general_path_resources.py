"""The shape that the gross code runs keeps its state in registers: a few bytes of local memory in
the iteration loop cost it 1 % (CPU only: reads the `-Xptxas -v` report kept beside the object)."""
from test_kernel_resources import fused_resources, ptxas_report


def test_the_gross_codes_shape_does_not_spill():
    regs, st, ld = fused_resources(ptxas_report("relay_fused_f32_8_4"))[(256, 11, 4)]
    assert st == 0 and ld == 0, f"256 x 11: {regs} registers, spill {st}/{ld} bytes"
