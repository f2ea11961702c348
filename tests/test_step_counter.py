"""The step counter's one writer, from the source: the first kernel of a step advances
DevState::t with one thread while its other threads run, so no thread of it may read t."""

import os
import re

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2608_09231_gb300", "csrc",
                   "bag_api.cu")


def test_the_kernel_that_advances_the_step_reads_no_step():
    src = re.sub(r"//[^\n]*", "", open(SRC).read())
    bumps = re.findall(r"(\w+)\.bump = ", src)
    assert bumps == ["pe"]
    made = re.findall(r"Epi pe = base_epi\(ctx, ([^,]+), ([^)]+)\);", src)
    # an epilogue without state takes step 0 and no flag
    assert made == [("nullptr", "-1")]
