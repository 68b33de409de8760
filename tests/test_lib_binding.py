"""What the binding's pointer arguments take: integers and None.  Bytes, text
and other objects are refused before the library sees them (a bytes object
would reach the GPU as the address of its host buffer)."""

import pytest

import paper_1302_6189_gb300 as md


@pytest.mark.parametrize("call", [md.mdfft_exec, md.mdfft_exec_graph])
@pytest.mark.parametrize("bad", [b"0123456789abcdef", "text", 1.5, [1]])
def test_execution_pointers_are_integers(call, bad):
    plan = md.mdfft_plan((8, 8), 4, flags=md.MDFFT_PLAN_HOST_ONLY)
    try:
        for args in ((bad, 4096), (4096, bad), (4096, 8192, -1, 0, bad)):
            with pytest.raises(TypeError):
                call(plan, *args)
        with pytest.raises(md.MdfftError):  # integers reach the library, which refuses a host-only plan
            call(plan, 4096, 8192)
        with pytest.raises(md.MdfftError):
            call(plan, None, 8192)
    finally:
        md.mdfft_destroy(plan)
