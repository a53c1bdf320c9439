"""Kernels launched as dependents are resident while their predecessor still writes the planes they
will read, and the read-only path (``__ldg``, ``const __restrict__``) is specified for data that nobody
writes while a kernel runs: in such a kernel it may serve only the tables built with the plan."""
import pathlib
import re

import pytest

CSRC = pathlib.Path(__file__).resolve().parents[1] / "paper_2401_09961_gb300" / "csrc"
TABLES = {"tw", "tt", "lamN", "lamM"}   # twiddles and eigenvalues
# bodies and loaders that the dependent kernels call
HELPERS = ("k_direction_pap_body", "k_update_body", "ld4", "quad_stages", "stage_twiddles")


def functions(name):
    """(name, signature, body) of every function of a source file that begins at the margin."""
    src = re.sub(r"//[^\n]*", "", (CSRC / name).read_text())
    for m in re.finditer(r"(\w+)\(([^{};]*)\) \{\n(.*?)\n\}", src, re.S):
        yield m.groups()


@pytest.mark.parametrize("name", ["dct.cu", "dct_fft.cu", "irls_kernels.cu"])
def test_dependent_kernels_read_planes_with_ordinary_loads(name):
    seen = 0
    for fn, sig, body in functions(name):
        if "pdl_enter();" not in body and fn not in HELPERS:
            continue
        seen += 1
        for p in re.findall(r"const\s+\w+\s*\*\s*__restrict__\s+(\w+)", sig + body):
            assert p in TABLES, (fn, p)
        for arg in re.findall(r"__ldg\(([^()]*(?:\([^()]*\))?[^()]*)\)", body):
            base = re.sub(r"reinterpret_cast<[^>]*>\s*\(?|&", "", arg)
            ident = re.match(r"\s*(\w+)", base).group(1)
            if ident == "p" and fn == "quad_stages":   # an entry of tw, named just above
                assert "const float2* p = &tw[" in body
                continue
            assert ident in TABLES, (fn, arg)
    assert seen >= 3
