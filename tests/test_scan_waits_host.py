"""CPU check: the sort's kernels wait for no other CTA.

Bucket starts come from the scan in k_sort.cu, and the paint reads its particles between two
starts.  A look-back scan whose bounded wait ran out would leave starts that are not ordered, and
the paint's ranges would then reach beyond the arrays.  A scan that adds up the sums of an earlier
launch has nothing to wait for, so the source must hold no polling of global memory.
"""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_no_kernel_of_the_sort_polls_memory():
    text = open(os.path.join(ROOT, "paper_2007_13394_gb300", "csrc", "k_sort.cu")).read()
    code = re.sub(r"//[^\n]*", "", text)
    assert not re.findall(r"ld\.(?:relaxed|acquire|volatile)|\bvolatile\s+(?:uint|unsigned|int|long)|[Ss]pin", code)
    assert "__threadfence" not in code and "nanosleep" not in code
