"""The fixed-point words that the binary64 synchrotron kernel reads
(synchro_coeffs64.h) and its arithmetic in integers (fit_synchrotron64.eval_fixed).
CPU: the words are those of the 60-digit fit, and the evaluation is within 5e-16 of
40-digit values at the edges of every piece and octave and between them (half a
unit in the last place, the rounding of the result, is 1.1e-16 of it; the rest is
the fit's and the words' share).  GPU: the kernel's results are the integers'
bit for bit."""
import os
import re

import numpy as np
import pytest

from paper_2008_10468_gb300 import fit_synchrotron64 as fit

HEADER = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                      "paper_2008_10468_gb300", "csrc", "synchro_coeffs64.h")


def _words():
    """(main, tail, exp2) by piece, as eval_fixed takes them."""
    with open(HEADER) as f:
        text = f.read()

    def pairs(name):
        body = re.search(name + r"\[[^=]*=\s*\{(.*?)\n\};", text, re.S).group(1)
        rows = [[(int(a), int(b)) for a, b in re.findall(r"\{(-?\d+)l*, (-?\d+)l*\}", line)]
                for line in body.strip().split("\n")]
        return [list(col) for col in zip(*rows)]

    exp2 = re.search(r"qed_syn64_exp2\[256\] = \{(.*?)\n\};", text, re.S).group(1)
    const = {n: int(v, 16) for n, v in re.findall(r"#define QED_SYN64_(LOG2E|LN2) (0x[0-9a-f]+)", text)}
    assert const == {"LOG2E": fit.LOG2E, "LN2": fit.LN2}
    return (pairs("qed_syn64_main"), pairs("qed_syn64_tail"),
            [int(v, 16) for v in re.findall(r"0x([0-9a-f]+)ull", exp2)])


def _points(octaves, per_piece, seed):
    """Edges of the octaves' pieces, their neighbours, and points between."""
    rng = np.random.default_rng(seed)
    x = []
    for k in octaves:
        for lo, hi in ((1.0, 1.25), (1.25, 1.5), (1.5, 2.0)):
            x += [lo * 2.0 ** k, float(np.nextafter(hi * 2.0 ** k, 0.0)),
                  float(np.nextafter(lo * 2.0 ** k, np.inf))]
            x += [float(v) for v in rng.uniform(lo, hi, per_piece) * 2.0 ** k]
    return x


def test_words_are_those_of_the_fit():
    mp = pytest.importorskip("mpmath")
    main, tail, exp2 = _words()
    assert len(main) == len(tail) == 3 * (fit.KMAX - fit.KMIN + 1) and len(exp2) == 256
    with mp.workdps(60):
        for i in range(256):
            assert exp2[i] == int(mp.nint(mp.power(2, 63 - mp.mpf(i) / 256)))
        assert fit.LOG2E == int(mp.nint(mp.power(2, 63) / mp.log(2)))
        assert fit.LN2 == int(mp.nint(mp.power(2, 64) * mp.log(2)))
    # the pieces up to x = 2 (the others take seconds each), word for word
    n = 3 * (1 - fit.KMIN)
    pieces = [fit.fit_piece(fit.KMIN + i // 3, i % 3) for i in range(n)]
    got = fit.fixed_tables(pieces)
    assert [list(map(tuple, p)) for p in got[0]] == main[:n]
    assert [list(map(tuple, p)) for p in got[1]] == tail[:n]


@pytest.mark.parametrize("octaves,per_piece", [(range(fit.KMIN, 0), 6), (range(0, 5), 6),
                                               (range(5, 7), 2), ([7], 0), ([8], 0)])
def test_evaluation_in_integers(octaves, per_piece):
    mp = pytest.importorskip("mpmath")
    from paper_2008_10468_gb300 import fit_synchrotron as fs
    words = _words()
    x = _points(octaves, per_piece, 5)
    if max(octaves) >= 7:
        x = x[::3]   # the 40-digit values take up to seconds each
    worst = 0.0
    for v in x:
        F, G = fit.eval_fixed(words, v)
        with mp.workdps(fs._dps_for(v)):
            worst = max(worst, abs(float(F / fs.F_mp(mp.mpf(v)) - 1)),
                        abs(float(G / fs.G_mp(mp.mpf(v)) - 1)))
    assert worst < 5e-16, worst


@pytest.mark.gpu
def test_kernel_is_the_integer_evaluation():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():  # pragma: no cover
        pytest.skip("no CUDA device")
    from paper_2008_10468_gb300 import qed
    words = _words()
    x = np.array(_points(range(fit.KMIN, fit.KMAX + 1), 200, 9))
    ref = np.array([fit.eval_fixed(words, float(v)) for v in x])
    y = torch.from_numpy(x).cuda()
    F, G = torch.empty_like(y), torch.empty_like(y)
    qed.synchrotron_F1F2_f64(y, F, G)
    np.testing.assert_array_equal(F.cpu().numpy(), ref[:, 0])
    np.testing.assert_array_equal(G.cpu().numpy(), ref[:, 1])
