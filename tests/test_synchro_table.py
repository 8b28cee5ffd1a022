"""The binary32 synchrotron table's envelope: exp(-x) multiplies the pieces from
one piece on and none before it, which the device code takes as one index."""
import re
from pathlib import Path

import paper_2008_10468_gb300


def test_exponential_envelope_starts_at_one_piece():
    text = (Path(paper_2008_10468_gb300.__file__).parent / "csrc" / "synchro_coeffs.h").read_text()
    body = re.search(r"qed_syn_table\[QED_SYN_NPIECE\]\[16\] = \{(.*?)\n\};", text, re.S).group(1)
    lam = [float(r.replace("f", "").split(",")[12]) for r in re.findall(r"\{(.*?)\}", body, re.S)]
    n = int(re.search(r"QED_SYN_NPIECE (\d+)", text).group(1))
    first = lam.index(1.0)
    assert len(lam) == n and lam == [0.0] * first + [1.0] * (n - first)
