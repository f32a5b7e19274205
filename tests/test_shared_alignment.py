"""Dynamic shared memory that kernels access 16 bytes at a time is declared
16-byte aligned: an array of a smaller type promises only that type's
alignment, and the accesses would then rest on where the toolchain happens to
place it.  Read from the sources; no device."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2503_13756_gb300", "csrc")


# the sources whose kernels take 16-byte accesses to dynamic shared memory
@pytest.mark.parametrize("name", ["sw_slice.cu", "sw_spectrum.cu", "sw_msw.cu", "sw_quantile.cu"])
def test_dynamic_shared_memory_is_16_byte_aligned(name):
    with open(os.path.join(CSRC, name)) as f:
        decls = re.findall(r"extern __shared__ ([^;]*);", f.read())
    assert decls
    short = [d for d in decls if "__align__(16)" not in d and not d.startswith("float4 ")
             and not d.startswith("float stg")]  # stg: 4-byte copies and loads only
    assert not short, short
