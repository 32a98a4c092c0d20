"""Transform lengths between the powers of two (8 r2 r3 = L1 L2).

On the CPU: the index arithmetic of the kernels at these lengths (every
shared-memory index inside its buffer, the staged boxes, the exchange free of
bank conflicts), and the digit order and prime-factor maps restated in numpy
against numpy.fft.  On the GPU: every arithmetic's operator against the
oracle's direct sums at the smallest and largest grid of each length and at
odd sizes, solves, batches, and plans from saved spectra."""

import os

import numpy as np
import pytest

import oracle as O
from paper_1602_04691_gb300 import inputs

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1602_04691_gb300", "csrc")
SMEM_MAX = 227 * 1024
MIX = {144: (6, 3, 12), 200: (5, 5, 20), 288: (6, 6, 24), 400: (10, 5, 20), 576: (6, 12, 24), 800: (10, 10, 40)}


def transform_length(n):
    L = 4
    while L < 2 * n:
        L *= 2
    return next((m for m in MIX if 2 * n <= m < L and m > L // 2), L)


def grid(*r):
    return np.meshgrid(*[np.arange(v) for v in r], indexing="ij")


def even_box(rows):
    q = -(-rows // 256)
    while rows % q:
        q += 1
    return rows // q


def test_sources_define_the_restated_lengths():
    with open(os.path.join(CSRC, "common.cuh")) as f:
        src = f.read()
    for L, (r2, r3, L1) in MIX.items():
        assert f"struct MixRad<{L}> {{ static constexpr int r2 = {r2}, r3 = {r3}, L1 = {L1}; }};" in src
        assert 8 * r2 * r3 == L and L1 % (L // L1) == 0 and (L // L1) % 2 == 0


@pytest.mark.parametrize("L,C,G", [(L, 8, 1) for L in MIX] + [(1024, 8, 2)])
def test_zconv_group_indices(L, C, G):
    """Z pass in G groups of C columns per CTA (zconv_groups)."""
    L1 = MIX[L][2] if L in MIX else 32
    L2 = L // L1
    NT, NI = C * L2, L1 // L2
    r16 = lambda v: -(-v // 16) * 16                                    # noqa: E731
    mod = 4 if C == 8 else 8
    pitch = lambda v: v + (mod // 2 - v % mod + mod) % mod              # noqa: E731
    PK, PKI = L2 + 1, L1 + 1
    PC, PCI = pitch(L1 * PK), pitch(L2 * PKI)
    PT = L2 if L1 == L2 else L2 + 1
    E, S, TW = r16(C * max(PC, PCI)), r16((L // 2 + 1) * C), r16(L1 * PT)
    assert (TW + G * (E + S)) * 8 + 136 + 8 * G <= SMEM_MAX and L % (C * G) == 0
    assert G == 1 or NT % 32 == 0 and G < 16                            # whole warps; named barriers 1..G
    tid, j1 = grid(NT, L1 // 2)
    assert ((j1 * L2 + tid // C) * C + tid % C).max() < (L // 2) * C
    tid, k1 = grid(NT, L1)
    c, jl = tid % C, tid // C
    st = c * PC + k1 * PK + jl
    assert st.max() < E and len(np.unique(st)) == st.size and (k1 * PT + jl).max() < TW
    ld = c * PCI + jl * PKI + k1
    assert ld.max() < E
    s, j = grid(NT * NI, L2)
    c2, q1 = s % C, s // C
    assert q1.max() == L1 - 1
    assert np.array_equal(np.unique(c2 * PC + q1 * PK + j), np.unique(st))      # every stored value is read
    assert np.array_equal(np.unique(c2 * PCI + j * PKI + q1), np.unique(ld))
    assert (q1 * PT + j).max() < TW and (L1 != L2 or (j * PT + q1).max() < TW)
    rows = np.where(j < L2 // 2, q1 + j * L1, L - q1 - j * L1)
    assert rows.min() >= 0 and rows.max() <= L // 2
    kz = q1 + L1 * j
    assert np.array_equal(rows, np.minimum(kz, L - kz))
    box = even_box(L // 2)
    for n in range(1, L // 2 + 1):                                      # TMA boxes of rows
        nbox = -(-n // box)
        assert nbox * box * C <= S and nbox * box * C * 8 < 1 << 20
    assert box <= 256 and (box * C * 8) % 128 == 0 and (C * 8) % 16 == 0 and ((L // 2 + 1) * C * 8) % 16 == 0
    for acc in (lambda t, i: (t % C) * PC + i * PK + t // C, lambda t, i: (t % C) * PC + (t // C) * PK + i,
                lambda t, i: (t % C) * PCI + i * PKI + t // C, lambda t, i: (t % C) * PCI + (t // C) * PKI + i):
        for h in range(0, NT - 15, 16):                                  # a half warp: 16 different 8-byte banks
            assert len(np.unique(acc(np.arange(h, h + 16), 3) % 16)) == 16


@pytest.mark.parametrize("L", MIX)
def test_xy_pass_indices(L):
    L1 = MIX[L][2]
    L2 = L // L1
    PK, PKI = L2 + 1, L1 + 1
    PC, PCI = (L1 * PK) | 1, (L2 * PKI) | 1
    # Y passes: 16 columns by TMA up to L = 400, 8 columns beyond
    C = 16 if L % 16 == 0 and L <= 400 else 8
    E = C * max(PC, PCI)
    assert L % C == 0 and C * L2 <= 1024
    assert (E + (L // 2) * C + L) * 8 + 144 <= SMEM_MAX
    BUF = max(C * L, E)
    assert (BUF + L) * 8 + 144 <= SMEM_MAX
    for rows, room in ((L // 2, (L // 2) * C), (L, BUF)):
        box = even_box(rows)
        assert box <= 256 and rows % box == 0 and rows * C <= room and (box * 128) % 128 == 0
    assert C == 8 or (E * 8) % 128 == 0                                  # staged rows 128-byte aligned after E
    # X passes: whole warps
    C = next(m for m in range(1, 65) if (m * L2) % 32 == 0 and m * L2 >= 96)
    NT = C * L2
    E = C * max(PC, PCI)
    assert NT % 32 == 0 and (E + 3 * C * (L // 2) + L) * 8 <= SMEM_MAX and C % 2 == 0
    assert (max(C * L, E) + C * L) * 8 + 32 * 16 + 32 <= SMEM_MAX and max(C * L, E) % 2 == 0
    s, j = grid(NT * (L1 // L2), L2)
    assert ((s // L1) * PC + (s % L1) * PK + j).max() < E and (s // L1).max() == C - 1
    assert ((s // L1) * PCI + j * PKI + s % L1).max() < E


@pytest.mark.parametrize("L", MIX)
def test_digit_order_and_stages(L):
    """The shared-memory stages (8, r2, r3) leave frequency digit_rev(p) at position p."""
    r2, r3, _ = MIX[L]
    rng = np.random.default_rng(L)
    x = rng.standard_normal(L) + 1j * rng.standard_normal(L)
    v, M = x.copy(), L
    for R in (8, r2, r3):
        s = M // R
        w = v.reshape(L // M, R, s)
        t = np.fft.fft(w, axis=1)
        t = t * np.exp(-2j * np.pi * np.arange(R)[:, None] * np.arange(s)[None, :] / M)
        v, M = t.reshape(L), s
    p = np.arange(L)
    q = p // r3
    k = q // r2 + 8 * (q % r2 + r2 * (p - q * r3))
    assert np.allclose(v, np.fft.fft(x)[k])
    qk = k // 8
    assert np.array_equal((k % 8 * r2 + (qk - qk // r2 * r2)) * r3 + qk // r2, p)


RADICES = {64: (1, 8), 128: (1, 16), 256: (8, 4), 512: (8, 8), 1024: (8, 16), 2048: (16, 16),
           **{L: v[:2] for L, v in MIX.items()}}


@pytest.mark.parametrize("L", RADICES)
def test_line_tiles_of_the_shared_memory_x_passes(L):
    """A padded line (one element per L / 8 points): every point has its place, each
    stage addresses it by its own eighth, and the eight consecutive frequencies a
    quarter warp takes in the last stage lie on different 16-byte banks (two to a
    bank at L = 200)."""
    r2, r3 = RADICES[L]
    assert 8 * r2 * r3 == L
    j = np.arange(L)
    place = j + j // (L // 8)
    assert len(np.unique(place)) == L and place.max() < L + 8
    jj, t = grid(L // 8, 8)
    assert np.array_equal((jj + t * (L // 8)) // (L // 8), t)            # first stage
    if r2 > 1:
        M = L // 8
        s = M // r2
        bi, t = grid(8 * s, r2)
        assert np.array_equal((bi // s * M + bi % s + t * s) // (L // 8), bi // s)
    blk, t = grid(L // r3, r3)
    assert np.array_equal((blk * r3 + t) // (L // 8), blk // r2)         # last stage
    for k0 in range(0, L // r3 - 7, 8):
        k = np.arange(k0, k0 + 8)
        b = (k & 7) * r2 + (k >> 3)
        banks = (b * r3 + b // r2) % 8
        assert len(np.unique(banks)) >= (4 if L == 200 else 8)


@pytest.mark.parametrize("R", [3, 5, 6, 10, 12, 20])
def test_prime_factor_map(R):
    P = R & -R
    Q = R // P
    rng = np.random.default_rng(R)
    a = rng.standard_normal(R) + 1j * rng.standard_normal(R)
    n2, n1 = grid(Q, P)
    t = np.fft.fft(np.fft.fft(a[(Q * n1 + P * n2) % R], axis=1), axis=0)
    k = np.arange(R)
    assert np.allclose(t[k % Q, k % P], np.fft.fft(a))


def yblk(L):
    if L < 256:
        return L
    if L & (L - 1):
        return 40 if L == 800 else L
    return 64 if L == 256 else 32


@pytest.mark.parametrize("L", [64, 128, 144, 200, 256, 288, 400, 512, 576, 800, 1024, 2048])
def test_blocked_scratch_layout(L):
    """T2 in blocks of yblk(L) values of ky: every point has its own place, the
    steps of the kernels move the block and the place in it by constant amounts
    where they are whole blocks or divide one, and the boxes
    of the Y-inverse rows are whole blocks of at most 256 rows."""
    B, n = yblk(L), 3
    assert L % B == 0
    ky, z = grid(L, n)
    off = (ky // B) * n * B * L + z * B * L + (ky % B) * L
    assert len(np.unique(off)) == off.size and off.max() == (n * L - 1) * L
    if B == L:
        return
    lg = L.bit_length() - 1
    L1 = MIX[L][2] if L in MIX else 1 << ((lg + 1) // 2)
    assert L1 % B == 0 or B % L1 == 0
    for step in (L1, 2 * L1, L // 8, L // 4, L // 16):                  # blk_at
        if L % step or not (step % B == 0 or B % step == 0):
            continue
        k = np.arange(step)
        for t in range(L // step):
            kk = k + step * t
            move = t * (step // B) * 7919 if step % B == 0 else (step * t // B) * 7919 + step * t % B
            assert np.array_equal((kk // B) * 7919 + kk % B, (k // B) * 7919 + k % B + move)
    nb = max(q for q in range(1, L // B + 1) if (L // B) % q == 0 and (q * B <= 256 or q == 1))
    assert nb * B <= 256 and L % (nb * B) == 0


def test_transform_lengths():
    for n in range(2, 1025):
        m = transform_length(n)
        L = 4
        while L < 2 * n:
            L *= 2
        assert 2 * n <= m <= L


# ---------------------------------------------------------------------------- GPU


def to_dev(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).to("cuda:0")


def rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


@pytest.mark.gpu
@pytest.mark.parametrize("n", [65, 72, 73, 100, 129, 144, 145, 200, 257, 288, 289, 400])
def test_operators_match_the_oracle(n):
    """Bounds: 1e-5 for FP32 and 1e-12 for FP64 and paired FP32, the bars the other lengths are held to."""
    from paper_1602_04691_gb300 import Plan
    k = 3.0
    h, N = inputs.random_h_N(n, 400 + n)
    x = inputs.random_complex(n ** 3, 401 + n)
    plan = Plan(n, k, to_dev(h), to_dev(N))
    rng = np.random.default_rng(n)
    rows = np.unique(np.concatenate([[0, n - 1, n * n - 1, n ** 3 - 1, n ** 3 - n, (n // 2) * (n * n + n + 1)],
                                     rng.choice(n ** 3, 12, replace=False)]))
    S, G = O.sqrt_hN(h, N), O.kernel_octant(n, k)
    scale = O.C_S_SPHERE / n ** 3
    ref_a = x[rows] + scale * O.offdiag_sum_rows_octant(h * N * x, rows, n, k, octant=G)
    ref_b = x[rows] + S[rows] * scale * O.offdiag_sum_rows_octant(S * x, rows, n, k, octant=G)
    xd = to_dev(x)
    precs = [("fp32", 1e-5), ("df", 1e-12)] + ([("fp64", 1e-12)] if n <= 200 else [])
    for prec, bound in precs:
        for form, ref in (("A", ref_a), ("B", ref_b)):
            y = plan.matvec(xd, form=form, precision=prec).cpu().numpy()
            assert rel(y[rows], ref) < bound, (prec, form)
    x32 = to_dev(x.astype(np.complex64))
    for variant in (0, 1):                       # 1: the Z rows by cp.async instead of TMA
        plan.set_schedule(dict(plan.schedule(), zconv_variant=variant))
        y = plan.matvec32(x32, form="B").cpu().numpy()
        assert rel(y[rows], ref_b) < 1e-5, variant
    plan.close()


@pytest.mark.gpu
def test_solves_batches_and_saved_spectra():
    from paper_1602_04691_gb300 import Plan
    n, ks = 70, [2.0, 3.0]
    h, N = inputs.random_h_N(n, 500)
    hd, Nd = to_dev(h), to_dev(N)
    plan = Plan(n, ks, hd, Nd)
    pow2 = Plan(n, ks, hd, Nd, min_L=256)        # the same operators at the power-of-two length
    dirs = [(0.0, 0.0, 1.0), (0.6, 0.8, 0.0), (1.0, 0.0, 0.0)]
    for a, b in ((plan.solve_batch(dirs, tol=1e-10), pow2.solve_batch(dirs, tol=1e-10)),
                 (plan.solve_batch(dirs, tol=1e-11, precision="fp64"), pow2.solve_batch(dirs, tol=1e-11, precision="fp64"))):
        assert all(i["status"] == 0 for i in a[1])
        assert float((a[0] - b[0]).norm() / b[0].norm()) < 1e-9    # both meet tol; ||A^-1|| is of order 1
    saved, saved_pow2 = plan.save_spectrum(), pow2.save_spectrum()
    x = to_dev(inputs.random_complex(n ** 3, 501))
    for data, src in ((saved, plan), (saved_pow2, pow2)):          # each file runs at the length it was saved at
        q = Plan(n, 0.0, hd, Nd, spectrum=data, min_L=256 if src is pow2 else 0)
        for prec in ("fp32", "df", "fp64"):
            assert bool((q.matvec(x, "B", prec) == src.matvec(x, "B", prec)).all())
    q = Plan(n, 0.0, hd, Nd, spectrum=saved_pow2)                   # a power-of-two file without min_L
    assert bool((q.matvec(x, "B", "fp64") == pow2.matvec(x, "B", "fp64")).all())
