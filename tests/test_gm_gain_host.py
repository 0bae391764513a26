"""The factor by which a generic window's line transform scales each frequency
(csrc/gm_gain.h, divided out of the propagator table), against the transforms
themselves: the passes' radix steps written out here as matrices in 64 bits, with
the constants that the kernels hold in FP32 rounded to FP32."""
import glob
import os
import re
import shutil
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2205_06327_gb300", "csrc")
SHAPES = sorted({tuple(int(v) for v in m) for f in glob.glob(os.path.join(CSRC, "chain_gm_*.cu"))
                 for m in re.findall(r"GmShape<(\d+), (\d+), (\d+),", open(f).read())}, key=np.prod)
SPLIT = {6: (2, 3), 8: (4, 2), 9: (3, 3), 12: (4, 3), 16: (4, 4)}


def _root(M, e):
    """exp(-2 pi i e / M) rounded to FP32 (the quarter turns exactly)."""
    w = np.exp(-2j * np.pi * (np.asarray(e) % M) / M)
    w = np.where(np.abs(w.real) < 1e-9, 0, w.real) + 1j * np.where(np.abs(w.imag) < 1e-9, 0, w.imag)
    return w.astype(np.complex64).astype(np.complex128)


def _radix(R):
    """The matrix of a radix-R step, as a product of its own steps."""
    if R == 1:
        return np.ones((1, 1), complex)
    if R in (2, 4):
        return np.round(np.exp(-2j * np.pi * np.outer(range(R), range(R)) / R))
    if R == 3:
        s = 1j * float(np.float32(0.86602540378443864676))
        return np.array([[1, 1, 1], [1, -0.5 - s, -0.5 + s], [1, -0.5 + s, -0.5 - s]])
    R1, R2 = SPLIT[R]
    x = np.eye(R, dtype=complex).reshape(R1, R2, R)            # [n1][n2] of n = R2 n1 + n2
    y = np.einsum("kn,nmr->kmr", _radix(R1), x)                # [k1][n2]
    y = y * _root(R, np.outer(range(R1), range(R2)))[:, :, None]
    y = np.einsum("lm,kmr->lkr", _radix(R2), y)                # [k2][k1] of k = k1 + R1 k2
    return y.reshape(R, R)


def _line(R1, R2, R3, inverse):
    """The whole line's transform as a matrix (inverse: of the frequencies)."""
    M, MI = R1 * R2 * R3, R2 * R3
    D1, D2, D3 = _radix(R1), _radix(R2), _radix(R3)
    tA = _root(M, np.outer(range(R1), range(MI)))              # [k1][j]
    tB = _root(M, R1 * np.outer(range(R2), range(R3))) if R2 > 1 else np.ones((1, R3))  # [k2][j2]
    n = np.arange(M).reshape(R1, MI)                           # element j + MI q
    k = (np.arange(R1)[:, None, None] + R1 * (np.arange(R2)[None, :, None] + R2 * np.arange(R3)[None, None, :]))
    if not inverse:
        x = np.zeros((R1, MI, M), complex)
        x[np.arange(R1)[:, None], np.arange(MI)[None, :], n] = 1
        x = np.einsum("kq,qjr->kjr", D1, x) * tA[:, :, None]
        x = x.reshape(R1, R2, R3, M)                           # j = j2 + R3 q2
        x = np.einsum("lq,kqjr->kljr", D2, x) * tB[None, :, :, None]
        x = np.einsum("mj,kljr->klmr", D3, x)                  # [k1][k2][k3]
        out = np.zeros((M, M), complex)
        out[k.reshape(-1)] = x.reshape(M, M)
        return out
    x = np.zeros((M, M), complex)
    x[np.arange(M), k.reshape(-1)] = 1
    x = x.reshape(R1, R2, R3, M)
    x = np.einsum("jm,klmr->kljr", D3.conj(), x) * tB.conj()[None, :, :, None]
    x = np.einsum("ql,kljr->kqjr", D2.conj(), x).reshape(R1, MI, M)
    x = x * tA.conj()[:, :, None]
    x = np.einsum("qk,kjr->qjr", D1.conj(), x)
    return x.reshape(M, M)


def test_every_instance_has_a_shape():
    assert len(SHAPES) == 18 and all(8 <= np.prod(s) <= 4096 for s in SHAPES)


@pytest.mark.parametrize("shape", [s for s in SHAPES if np.prod(s) <= 288], ids=lambda s: str(np.prod(s)))
def test_gain_is_that_of_the_transforms(tmp_path, shape):
    M = int(np.prod(shape))
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host compiler")
    src = tmp_path / "t.cpp"
    src.write_text('#include <cstdio>\n#include "gm_gain.h"\nint main() {\n'
                   f'  std::vector<double> g({M});\n  ptycho::gm_transform_gain({shape[0]}, {shape[1]}, {shape[2]}, '
                   'g.data());\n  for (double v : g) std::printf("%.17g\\n", v);\n}\n')
    subprocess.run([cxx, "-std=c++17", "-I", CSRC, str(src), "-o", str(tmp_path / "t")], check=True)
    gain = np.array(subprocess.run([str(tmp_path / "t")], check=True, capture_output=True, text=True).stdout.split(),
                    dtype=float)
    F, B = _line(*shape, inverse=False), _line(*shape, inverse=True)
    tones = np.exp(2j * np.pi * np.outer(np.arange(M), np.arange(M)) / M)  # [n][k]
    # both are the transforms, to the rounding of their constants
    exact = np.exp(-2j * np.pi * np.outer(np.arange(M), np.arange(M)) / M)
    assert np.abs(F - exact).max() < 1e-6 and np.abs(B - exact.conj()).max() < 1e-6
    want = np.abs(np.einsum("kn,nk->k", F, tones) * np.einsum("nk,nk->k", tones.conj(), B)) / M ** 2
    assert np.abs(gain - want).max() < 1e-13
    assert np.abs(gain - 1).max() < 1e-6 and (M == 16 or np.abs(gain - 1).max() > 1e-9)
