"""The FP32 Box-Muller normals in pairs of FP32 numbers, compiled for the host
from the library's header: against long double on random words and at every
edge (uniforms next to 0 and 1, angles at quadrants and table limits)."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_1808_02281_gb300 import build as B, synth

SRC = r"""
#define __host__
#define __device__
#include "gaussian.cuh"
static const lqcd::NormalTables tables{};
extern "C" void normals(const unsigned long long *w, float *out, long n)
{
    for (long i = 0; i < n; ++i) out[i] = lqcd::normal_of(w[2 * i], w[2 * i + 1], tables);
}
"""


@pytest.fixture(scope="module")
def normals(tmp_path_factory):
    d = tmp_path_factory.mktemp("normals")
    src, lib = d / "normals.cpp", d / "libnormals.so"
    src.write_text(SRC)
    subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-shared", "-fPIC", "-I", os.path.join(B.HERE, "csrc"),
                    "-o", str(lib), str(src)], check=True)
    fn = ctypes.CDLL(str(lib)).normals
    fn.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_long]

    def run(words):
        words = np.ascontiguousarray(words, dtype=np.uint64)
        out = np.empty(len(words), np.float32)
        fn(words.ctypes.data, out.ctypes.data, len(words))
        return out
    return run


def _exact(words):
    w = words.astype(np.float64).astype(np.longdouble)
    u1, u2 = (w[:, 0] + 1) * np.longdouble(2.0) ** -53, w[:, 1] * np.longdouble(2.0) ** -53
    pi = np.longdouble("3.14159265358979323846264338327950288")
    return np.sqrt(-2 * np.log(u1)) * np.cos(2 * pi * u2)


def test_normals(normals):
    top = 2 ** 53 - 1
    edge = [2 ** e - 1 for e in range(54)] + [top - 2 ** e for e in range(53)] + [0, 1, 2, 3, top - 1, top - 3]
    angle = [i * 2 ** 43 + d for i in range(1025) for d in (-2, -1, 0, 1, 2)]
    angle = [a for a in angle if 0 <= a <= top] + edge
    r = synth.words(11, 0, 2 * len(angle)) >> np.uint64(11)
    words = np.concatenate([
        (synth.words(7, 0, 400000) >> np.uint64(11)).reshape(-1, 2),
        np.stack([r[:len(angle)], np.array(angle, dtype=np.uint64)], 1),
        np.array([(a, b) for a in edge for b in edge[::3]], dtype=np.uint64)])
    y, want = normals(words).astype(np.longdouble), _exact(words)
    # rounded once: half a unit in the last place, and 2^-30 of the value for the pairs
    ulp = np.spacing(np.abs(want).astype(np.float32)).astype(np.longdouble)
    # (where long double has no better value, cos next to its zeros, 1e-18 of the radius)
    assert (np.abs(y - want) <= 0.5 * ulp + np.abs(want) * 2.0 ** -30 + 1e-18).all()
