"""Register and spill budgets, as in test_kernel_resources.py, of the FP64 steps and
fields in fixed point and of the one-row step."""
import pytest

from tests.test_kernel_resources import _entries, _find, reports  # noqa: F401 (fixture)

# (source, mangled-name pattern, register budget, spill budget in bytes)
BUDGETS = [
    # (2+1)-d, order 2 and on-lattice order 3: five blocks of 128 threads per SM; bilinear order 3: four
    ("step2x", r"k_step2xILi9E", 96, 0),
    ("step2x", r"k_step2xILi16ELi0E", 96, 0),
    ("step2x", r"k_step2xILi16ELi1E", 128, 0),
    ("step2x", r"k_fields2x", 64, 160),       # (eight; the spills lie beside the call of the FP64 frame)
    # (3+1)-d: six and five blocks per SM; the spills lie beside that call as well
    ("step3x", r"k_step3xILi2E", 80, 80),
    ("step3x", r"k_step3xILi3E", 96, 64),
    ("step3x", r"k_fields3xILi2E", 72, 64),
    ("step3x", r"k_fields3xILi3E", 80, 32),
    # (1+1)-d orders 3 and 5: seven and six blocks
    ("d1", r"k_step1xILi3E", 72, 0),
    ("d1", r"k_step1xILi5E", 80, 0),
    # the one-row step: a cluster of eight blocks of at most 256 threads
    ("step_row", r"k_row_steps", 255, 0),
]


@pytest.mark.parametrize("src,pattern,regs,spill", BUDGETS)
def test_kernel_stays_within_its_register_and_spill_budget(reports, src, pattern, regs, spill):  # noqa: F811
    for name, (r, st, ld) in _find(_entries(reports[src]), pattern).items():
        assert r <= regs, (name, r)
        assert st <= spill and ld <= spill, (name, st, ld)
