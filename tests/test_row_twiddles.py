"""The twiddles of the pairing step of a row's real transform (row_tw in x_rows.cuh),
on the host: for rows of up to 512 reals every value that a thread uses has the
accuracy of a table entry (half a unit in the last place of 1, 2^-25 per
component), and the kernels choose such a form there."""

import subprocess

import numpy as np
import pytest


def table(k, M):
    t = np.pi * np.asarray(k, np.float64) / M
    return np.stack([np.cos(t), -np.sin(t)]).astype(np.float32)          # exp(-2 pi i k / (2 M)), rounded


def half(k, m, M, E):
    if m < E // 2:
        return table(k, M)
    c, s = table(k - M // 2, M)
    return np.stack([s, -c])                                             # times -i


def one(j, m, M, E):
    (c, s), f = table(j, M), np.float32
    t = np.pi * m / E
    a, b = f(np.cos(t)), f(-np.sin(t))
    return np.stack([c * a - s * b, c * b + s * a]).astype(f)


@pytest.mark.parametrize("M", [128, 256])
def test_half_table_form_has_table_accuracy(M):
    E, tl = 8, M // 8
    worst = {"half": 0.0, "one": 0.0}
    for m in range(E):
        j = np.arange(tl)
        k = j + tl * m
        t = np.pi * k / M
        exact = np.stack([np.cos(t), -np.sin(t)])
        worst["half"] = max(worst["half"], np.abs(half(k, m, M, E) - exact).max())
        worst["one"] = max(worst["one"], np.abs(one(j, m, M, E) - exact).max())
    assert worst["half"] <= 2.0 ** -25 * (1 + 1e-6)
    assert worst["one"] > 2.0 ** -25                                      # (why it is not used there)


def test_kernels_use_accurate_forms_up_to_512_reals(tmp_path):
    from paper_1408_4675_gb300 import build
    src = tmp_path / "t.cu"
    src.write_text('#include "x_rows.cuh"\nusing namespace kwgb;\n' +
                   "\n".join("static_assert(tw_form<%d>() != TW_ONE, \"accuracy\");" % (1 << n) for n in range(2, 9)) + "\n")
    subprocess.run([build._nvcc(), *build.ARCH, "-std=c++17", "-I", build.CSRC, "-I", build.INCLUDE, "-c", str(src), "-o",
                    str(tmp_path / "t.o")], check=True)
