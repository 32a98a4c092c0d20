"""The blocked layout of the scratch cube T2 against the tensor maps, copies and
slices that read it (CPU): the maps' dimensions, strides and boxes, the copies'
coordinates and the rules by transform length are taken from the sources."""

import os
import re
import shutil
import subprocess

import numpy as np
import pytest
import test_mixed_lengths as mixed

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1602_04691_gb300", "csrc")
LENGTHS = [64, 128, 144, 200, 256, 288, 400, 512, 576, 800, 1024]
CB = 8


def read(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


API, IMPL = read("ori_api.cu"), read("passes_impl.cuh")


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    """yblk, zgroup, even_box, transform_length and the stage radices, compiled from the sources."""
    if shutil.which("g++") is None:
        pytest.skip("no g++")
    common, passes, dfft = read("common.cuh"), read("passes.cuh"), read("dfft.cuh")
    body = ["#include <cstdio>", "#include <initializer_list>", "constexpr bool is_pow2(int v) { return (v & (v - 1)) == 0; }",
            re.search(r"constexpr bool is_mixed_len.*?\n", common).group(0), "template <int L> struct MixRad;",
            *re.findall(r"template <> struct MixRad<.*?\n", common),
            re.search(r"template <int L, bool MIXED = is_mixed_len\(L\)>\nstruct SRad \{.*?\n\};", dfft, re.S).group(0),
            re.search(r"template <int L>\nstruct SRad<L, true> \{.*?\n\};", dfft, re.S).group(0),
            "constexpr int kZGroup = 16;",
            re.search(r"constexpr int zgroup\(.*?\n", passes).group(0),
            re.search(r"constexpr int transform_length\(.*?\n\}", passes, re.S).group(0),
            re.search(r"constexpr int yblk\(.*?\n\}", passes, re.S).group(0),
            re.search(r"constexpr int even_box\(.*?\n\}", passes, re.S).group(0)]
    main = "int main() {\n" + "".join(
        f'  std::printf("L {L} %d %d %d %d %d %d\\n", yblk({L}), zgroup({L}), even_box({L} / 2), even_box({L}), '
        f"SRad<{L}>::r2, SRad<{L}>::r3);\n" for L in LENGTHS + [2048])
    main += ('  for (int n = 2; n <= 1024; ++n) { int p = 4; while (p < 2 * n) p *= 2; '
             'std::printf("n %d %d\\n", n, transform_length(n, p)); }\n}\n')
    d = tmp_path_factory.mktemp("rules")
    (d / "r.cpp").write_text("\n".join(body) + "\n" + main)
    subprocess.run(["g++", "-std=c++17", "-o", str(d / "r"), str(d / "r.cpp")], check=True)
    out = subprocess.run([str(d / "r")], check=True, capture_output=True, text=True).stdout.split("\n")
    by_L = {int(w[1]): dict(zip(("B", "W", "half", "full", "r2", "r3"), map(int, w[2:]))) for w in map(str.split, out) if w and w[0] == "L"}
    by_n = {int(w[1]): int(w[2]) for w in map(str.split, out) if w and w[0] == "n"}
    return by_L, by_n


def test_the_restated_rules_are_the_sources(rules):
    """The Python copies in test_mixed_lengths.py."""
    by_L, by_n = rules
    for L, r in by_L.items():
        assert r["B"] == mixed.yblk(L) and r["half"] == mixed.even_box(L // 2) and r["full"] == mixed.even_box(L)
        assert (r["r2"], r["r3"]) == mixed.RADICES[L]
    assert all(m == mixed.transform_length(n) for n, m in by_n.items())


def array(name, env):
    """A dims / strides / box initialiser of a tensor map, evaluated."""
    body = re.search(r"const cuuint\w+ " + name + r"\[\d\] = \{(.*?)\};", API, re.S).group(1)
    body = re.sub(r"cuuint(?:64|32)_t", "", body).replace("/", "//").replace("p->n", "n").replace("std::", "")
    body = body.replace("t2_elems(p)", "(n * L * L)").replace("t1_elems(p)", "(n * n * L)")
    body = re.sub(r"(\w+ == \w+) \? (\w+) : (\w+)", r"(\2 if \1 else \3)", body)
    return list(eval("(" + body.replace("\n", " ") + ",)", {"min": min}, env))


def box_rows(dims, strides, box, at):
    """Element offsets of the rows of a box (None where the hardware fills in zeros), row-major over the box, x left out."""
    shape = box[1:][::-1]
    idx = np.indices(shape)[::-1]
    off = np.full(shape, at[0], dtype=np.int64)
    ok = np.ones(shape, dtype=bool)
    for d in range(len(shape)):
        c = at[1 + d] + idx[d]
        ok &= (c >= 0) & (c < dims[1 + d])
        off = off + c * strides[d] // CB
    return [int(o) if k else None for o, k in zip(off.ravel(), ok.ravel())]


@pytest.mark.parametrize("n", ["smallest", "odd", "largest"])
@pytest.mark.parametrize("L", LENGTHS)
def test_z_tiles_read_their_rows_and_nothing_else(L, n, rules):
    """Boxes of the Z map: row z of tile (ky, kx) is T2's, and the rows past n are not read."""
    r = rules[0][L]
    B = r["B"]
    n = {"smallest": L // 4 + 1, "odd": (3 * L // 8) | 1, "largest": L // 2}[n]
    plain, R = B == L, 2
    for w in sorted({r["W"]} if L & (L - 1) else {r["W"], 16}):       # mixed lengths: groups only
        rows = min(L // 2, 256) if w == 16 else r["half"]
        env = dict(L=L, B=B, n=n, R=R, es=CB, w=w, rows=rows, kZGroup=16, zbox=min(L // 2, 256), row=B * L * CB, rhs=n * L * L * CB)
        dims, strides = array("dims_p" if plain else "dims_b", env), array("str_p" if plain else "str_b", env)
        box = (array("box", env) if plain and w == 16 else array("box_b", env))[:len(dims)]
        assert box[0] == w and all(1 <= v <= 256 for v in box) and all(s % 16 == 0 and s < 1 << 40 for s in strides)
        assert dims[-1] == R and strides[-1] == n * L * L * CB
        nbox = -(-n // rows)
        assert nbox * rows <= L // 2 + 1
        for ky in (0, 1, B - 1, B % L, L // 2, L - 1):
            kb, kx, rhs = ky // B, 3 * w, 1
            got = []
            for q in range(nbox):
                at = [kx, ky, q * rows, rhs] if plain else [kx, ky - kb * B, q * rows, kb, rhs]
                got += box_rows(dims, strides, box, at)
            want = [rhs * n * L * L + kb * n * B * L + z * B * L + (ky % B) * L + kx for z in range(n)]
            assert got[:n] == want and got[n:] == [None] * (nbox * rows - n), (L, n, ky, w)
    src = IMPL[IMPL.index("void zpipe_tma_rows("):IMPL.index("void zpipe_tma_ghat(")]
    assert "tma_load_4d(S + q * a.zbox * C, &a.zrows, cb * C, ky, q * a.zbox, rhs, bar)" in src
    assert "tma_load_5d(S + q * a.zbox * C, &a.zrows, cb * C, ky - kb * yblk(L), q * a.zbox, kb, rhs, bar)" in src


@pytest.mark.parametrize("L", LENGTHS)
def test_y_inverse_boxes_are_the_rows_in_order(L, rules):
    r = rules[0][L]
    B, n, R = r["B"], L // 4 + 1, 2
    nblk = L // B
    nb = max(q for q in range(1, nblk + 1) if nblk % q == 0 and (q * B <= 256 or q == 1))
    bi = r["full"] if B == L else nb * B
    env = dict(L=L, B=B, n=n, R=R, es=CB, nblk=nblk, nb=nb, bi=bi, kZGroup=16, min=min)
    dims, strides, box = array("dims_i", env), array("str_i", env), array("box_i", env)
    assert box[0] == 16 and all(1 <= v <= 256 for v in box) and L % bi == 0
    z, kx, rhs = n - 1, 16, 1
    got = []
    for q in range(L // bi):
        got += box_rows(dims, strides, box, [kx, q * bi if B == L else 0, 0 if B == L else q * (bi // B), z, rhs])
    assert got == [rhs * n * L * L + (ky // B) * n * B * L + z * B * L + (ky % B) * L + kx for ky in range(L)]
    src = IMPL[IMPL.index("void yinv_tma_rows("):]
    assert re.search(r"tma_load_5d\(S \+ q \* a\.zbox \* C, &a\.zrows, cb \* C, BK == L \? q \* a\.zbox : 0, "
                     r"BK == L \? 0 : q \* \(a\.zbox / BK\), outer,\s+rhs, bar\);", src)


@pytest.mark.parametrize("C,L1", [(16, 32), (8, 32), (16, 64)])
def test_spectrum_slices_of_the_1024_point_variants(C, L1):
    """The spectrum lies in groups of W = 8 columns at 1024 points: the slice of a
    16-column tile is two runs, one after another in the cube and in the buffer,
    and every product reads the entry of its own frequency."""
    L, W = 1024, 8
    H, L2 = L // 2 + 1, L // L1
    my, cb = 5, 7
    gz = lambda kx, mz: ((my * (L // W) + kx // W) * H + mz) * W + kx % W          # noqa: E731  (k_build_ghatZ)
    base = (my * (L // W) + cb * (C // W)) * H * W                                  # zpipe_tma_ghat
    c2, k1, k2 = np.meshgrid(np.arange(C), np.arange(L1), np.arange(L2), indexing="ij")
    kz = k1 + L1 * k2
    run = (c2 // W) * H * W + c2 % W
    at = np.where(k2 < L2 // 2, run + k1 * W + k2 * L1 * W, run + (L - k1) * W - k2 * L1 * W)
    assert at.min() >= 0 and at.max() < H * C
    assert np.array_equal(base + at, gz(cb * C + c2, np.minimum(kz, L - kz)))
    for line in ("const cpx<T>* run = S + (c2 / W) * (L / 2 + 1) * W + c2 % W;", "const cpx<T>* lo = run + k1 * W;",
                 "const cpx<T>* hi = run + (L - k1) * W;", "k2 < L2 / 2 ? lo[k2 * L1 * W] : hi[-k2 * L1 * W]",
                 "((long long)my * (L / W) + cb * (C / W)) * run;"):
        assert line in IMPL, line
