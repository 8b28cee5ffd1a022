"""The push step draws a window of sub-steps against an upper bound of its
thresholds, which takes the tabulated envelope H of the emission bound at the
largest argument that the window can reach: H must not fall anywhere."""
import re
from pathlib import Path

import numpy as np

import paper_2008_10468_gb300


def test_emission_envelope_does_not_fall():
    text = (Path(paper_2008_10468_gb300.__file__).parent / "csrc" / "synchro_coeffs.h").read_text()
    body = re.search(r"qed_sqz_emission\[(\d+)\] = \{(.*?)\}", text, re.S)
    h = np.array([float.fromhex(t.rstrip("f")) if "0x" in t else float(t.rstrip("f"))
                  for t in re.findall(r"[-+0-9a-fA-Fxp.]+f?", body.group(2))])
    assert len(h) == int(body.group(1)) and (h > 0).all()
    assert (np.diff(h) >= 0).all()
