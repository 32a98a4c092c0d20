"""Kernels launched as dependent launches (their prologue runs while the
predecessor still writes), checked in the sources on the CPU: every one waits
for its predecessor, and none reads a predecessor's data by loads that the
compiler may make non-coherent (const __restrict__ parameters, __ldg)."""

import os
import re

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1602_04691_gb300", "csrc")
# complete before the first dependent launch of a call: the medium (host synchronisation in set_medium) and the
# caller's right-hand side (an event wait, which is a full dependency)
CONSTANT = {"S", "Sinv", "rhs"}


def read(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def kernels(src):
    """name -> (parameters, body up to its closing brace in column 0)"""
    out = {}
    for m in re.finditer(r"__global__ void\s+(?:__launch_bounds__\(.*?\)\)?\s*)?(k_\w+)(<float>)?\s*\(([^)]*)\)\s*\{", src,
                         re.S):
        end = src.index("\n}", m.end())
        out[m.group(1) + (m.group(2) or "")] = (m.group(3), src[m.end():end])
    return out


DEPENDENT = sorted(set(re.findall(r"launch_dep\((k_\w+)", read("ori_api.cu"))))


def test_the_solver_launches_vector_kernels_dependently():
    assert {"k_cocg_update", "k_cocg_init", "k_normalise_to_f32", "k_accumulate", "k_rhs", "k_read_heads"} <= set(DEPENDENT)


@pytest.mark.parametrize("name", DEPENDENT)
def test_vector_kernels_wait_and_read_coherently(name):
    ks = {k: v for k, v in kernels(read("vector_kernels.cuh")).items() if k.split("<")[0] == name}
    assert ks
    for params, body in ks.values():
        assert body.lstrip().startswith("dep_wait();")
        assert "__ldg" not in body and "ldgc(" not in body
        for p in params.split(","):
            if "const" in p and "__restrict__" in p:
                assert p.split()[-1] in CONSTANT, p.strip()


def test_passes_read_only_the_medium_and_the_spectrum_non_coherently():
    src = read("passes_impl.cuh")
    for m in re.finditer(r"\bldgc\(([^;]*);", src):
        assert re.match(r"(reinterpret_cast<const cpx<\w+>\*>\(a\.scale\)|gh |gp )", m.group(1)), m.group(0)
    assert "__ldg" not in src
    for m in re.finditer(r"const \w+(?:<\w+>)?\* __restrict__", src):
        pytest.fail(m.group(0))
