"""Registers of the persistent batch kernels: their claim loop sits on top of a
whole site update, so a block count that suits the single-lattice kernel can make
them spill.  At 164 bytes (E5, extended sums of level 1) a step took a fifth
longer; the limit is the largest spill that was measured to be harmless (112
bytes, E5 in BF16 storage) rounded up."""
import os
import re


def test_persistent_kernels_spill_little():
    from paper_1703_04605_gb300 import build as B
    B.build()
    log = open(os.path.join(B.BUILD, "ptxas.log")).read()
    found = re.findall(r"Compiling entry function '(\S*persist_kernel\S*)'.*?(\d+) bytes spill stores", log, re.S)
    assert len(found) == 16
    for name, spill in found:
        assert int(spill) <= 128, (name, spill)
