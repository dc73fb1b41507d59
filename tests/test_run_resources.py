"""Registers and spills of the kernels that carry a gate, from the compiler's
resource report, built exactly as the library is.

The launch bounds fix how many CTAs share an SM and so the registers; what does
not fit is spilled, and more of it than was measured is a slower gate.  Runs on
the CPU: nvcc cross-compiles, nothing is launched.
"""
import pytest

from tests.test_kernel_resources import _find, _report

# kernel -> CTA size, CTAs per SM, bytes of spill stores and loads it was
# measured with
KERNELS = {
    "itpp_run.cu": {"k_run<1, false>": (256, 3, 844, 1692), "k_run<2, false>": (256, 2, 132, 268)},
    "itpp_run_wide.cu": {"k_run<1, true>": (256, 4, 1184, 2208), "k_run<2, true>": (256, 3, 1004, 1788)},
    "itpp_part.cu": {"k_gate_inplace<1, 256>": (256, 4, 0, 0), "k_gate_inplace<2, 128>": (128, 6, 276, 96)},
    "itpp_select.cu": {"k_sel_resolve<1>": (256, 2, 0, 0), "k_sel_resolve<2>": (256, 2, 0, 0)},
    "itpp_adjoint.cu": {"k_adj_recompute<1>": (256, 4, 0, 0), "k_adj_recompute<2>": (256, 4, 44, 36),
                        "k_adj_reverse<1>": (256, 4, 32, 32), "k_adj_reverse<2>": (256, 4, 68, 72)},
}


@pytest.mark.parametrize("src", sorted(KERNELS))
def test_registers_and_spills(src, tmp_path):
    res = _report(src, tmp_path)
    for name, (block, per_sm, stores, loads) in KERNELS[src].items():
        k = _find(res, name + "(")
        assert res[k + " regs"] <= 65536 // (block * per_sm) // 8 * 8, (k, res[k + " regs"])
        # a tenth more for another compiler of the same release
        assert res[k][1] <= 1.1 * stores, (k, res[k])
        assert res[k][2] <= 1.1 * loads, (k, res[k])
