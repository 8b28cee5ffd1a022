"""A pass that decides from the store's count that all its work is known reads that
count after the atomic that told it so: the last block of the thread pass, and the
warp that completes the last unit of the persistent pass.  A load may be performed
before an atomic that precedes it unless a fence stands between them."""
import re
from pathlib import Path

import pytest

import paper_2008_10468_gb300

SRC = Path(paper_2008_10468_gb300.__file__).parent / "csrc" / "qed.cu"


@pytest.mark.parametrize("atomic,count", [
    (r"atomicAdd\(&ctl->cold_done, 1u\)", r"ctl->n1 = \(long long\)stored_rows\(P\)"),
    (r"sum \+ atomicAdd\(&ctl->finished, sum\)", r"units0 \+ \(stored_rows\(P\) - n1\)")])
def test_fence_between_completion_and_count(atomic, count):
    text = re.sub(r"//[^\n]*", "", SRC.read_text())
    between = re.search(atomic + r"(.{0,200}?)" + count, text, re.S)
    assert between and "__threadfence();" in between.group(1)
