"""The build refuses a split kernel compiled to another register count than its
warpgroups' shares add up to (the launch would refuse it, at the user's call)."""
import pytest

from paper_1701_02011_gb300.build import check_registers

SOURCE = "constexpr int OZ_REGS = 168, OZ_REGS_SUM = 208;"


def _log(*counts):
    return "".join(f"ptxas info    : Compiling entry function '_Z11k_ozaki_mmaILi64ELi{k}EEv' for 'sm_103a'\n"
                   f"ptxas info    : Function properties for _Z11k_ozaki_mmaILi64ELi{k}EEv\n"
                   "    0 bytes stack frame, 0 bytes spill stores, 0 bytes spill loads\n"
                   f"ptxas info    : Used {n} registers, used 3 barriers, 4784 bytes smem\n"
                   "ptxas info    : Compiling entry function '_Z13k_ozaki_otherv' for 'sm_103a'\n"
                   "ptxas info    : Used 40 registers\n" for k, n in enumerate(counts, 1))


def test_register_count_of_the_split_kernel():
    check_registers(SOURCE, _log(168, 168))
    with pytest.raises(RuntimeError, match="166"):
        check_registers(SOURCE, _log(168, 166))
    with pytest.raises(RuntimeError, match="no registers"):
        check_registers(SOURCE, "")
