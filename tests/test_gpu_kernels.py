"""Single kernels at the sizes where their vector paths, tiles and splits meet
their edges, against exact integers or the oracle."""
import numpy as np
import pytest

import oracle
from paper_2101_01025_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    import paper_2101_01025_gb300 as aat
    return aat


@pytest.mark.parametrize("off", [0, 1, 2, 3])
@pytest.mark.parametrize("n,pad", [(1, 0), (2, 1), (3, 0), (4, 4), (5, 2), (33, 3), (64, 0), (257, 1)])
def test_zero_upper_clears_the_strict_upper_triangle_only(lib, n, pad, off):
    """Rows that start at every offset modulo 16 bytes; entries outside the
    n x n result and the lower triangle keep their values."""
    import torch
    p, k = 65521, 7
    A = synth.residues(11 + n, (n, k), p)
    ldc = n + pad
    buf = torch.full((off + n * ldc + 5,), -7, dtype=torch.int32, device="cuda")
    C = torch.as_strided(buf, (n, n), (ldc, 1), off)
    lib.aat_modp(torch.from_numpy(A).cuda(), p, C=C, flags=lib.AAT_ZERO_UPPER, levels=0)
    want = np.full(buf.shape, -7, dtype=np.int32)
    ref = oracle.aat_modp_low(A, p).astype(np.int64)
    for r in range(n):
        want[off + r * ldc:off + r * ldc + n] = 0
        want[off + r * ldc:off + r * ldc + r + 1] = ref[r, :r + 1]
    assert np.array_equal(buf.cpu().numpy(), want)


@pytest.mark.parametrize("p", [13, 65521, 1000003, 2**31 - 1])
@pytest.mark.parametrize("rows,cols,off", [(1, 1, 0), (3, 2, 1), (5, 3, 3), (9, 4, 0), (7, 4, 2),
                                           (8, 5, 0), (2, 127, 1), (3, 1024, 0), (2, 2051, 1)])
def test_split_of_ragged_and_unaligned_rows(lib, p, rows, cols, off):
    """Digits and pair sums of every entry, zeros in the row padding."""
    import torch
    from paper_2101_01025_gb300 import testing as T
    b, L, _, ns = T.digit_spec(p, with_sums=True)
    X = synth.residues(17 * rows + cols, (rows, cols), p, balanced=True)
    ld = cols + off
    buf = torch.zeros(off + rows * ld + 4, dtype=torch.int32, device="cuda")
    view = torch.as_strided(buf, (rows, cols), (ld, 1), off)
    view.copy_(torch.from_numpy(X))
    got = T.split(view, p).float().cpu().numpy().astype(np.int64)
    assert not got[:, :, cols:].any()
    d = got[:, :, :cols]
    assert np.array_equal(sum(d[i] << (b * i) for i in range(L)), X.astype(np.int64))
    pairs = [(i, j) for i in range(L) for j in range(i + 1, L)][:ns]
    for q, (i, j) in enumerate(pairs):
        assert np.array_equal(d[L + q], d[i] + d[j])


@pytest.mark.parametrize("lower", [False, True])
@pytest.mark.parametrize("p", [65521, 131071, 2**31 - 1])
@pytest.mark.parametrize("M,N,K", [(1, 1, 1), (128, 64, 64), (129, 65, 65), (127, 63, 63),
                                   (200, 191, 130), (260, 260, 1030)])
def test_narrow_leaf_tiles(lib, M, N, K, p, lower):
    """64-column tiles at their edges, stored and accumulated, with rows that
    are and are not 16-byte aligned."""
    import torch
    from paper_2101_01025_gb300 import testing as T
    if lower and M != N:
        N = M
    X = synth.residues(M + K, (M, K), p, balanced=True)
    Y = X if lower else synth.residues(N + 3 * K, (N, K), p, balanced=True)
    ref = (X.astype(object) @ Y.astype(object).T) % p
    Xd, Yd = torch.from_numpy(X).cuda(), torch.from_numpy(Y).cuda()
    for ld in (N, (N + 3) // 4 * 4):
        old = synth.residues(5, (M, ld), p)
        for acc in (False, True):
            C = torch.from_numpy(old.copy()).cuda()
            T.leaf(Xd, Xd if lower else Yd, p, C=C[:, :N], lower=lower, accumulate=acc)
            want = old.astype(object)
            new = (ref + (want[:, :N] if acc else 0)) % p
            mask = np.tril(np.ones((M, N), bool)) if lower else np.ones((M, N), bool)
            want[:, :N][mask] = new[mask]
            assert np.array_equal(C.cpu().numpy().astype(object), want)


@pytest.mark.parametrize("p", [65521, 131071, 2**31 - 1])
@pytest.mark.parametrize("n,k,pad", [(1, 1, 0), (33, 5, 0), (64, 132, 4), (130, 259, 1), (300, 96, 0)])
def test_quaternion_product_in_one_leaf_launch(lib, n, k, pad, p):
    """Operand planes straight from A, B, C, D (aligned and ragged rows), the
    six products' tiles in one launch, cleared upper triangles."""
    import torch
    parts = [synth.residues(7 * n + k + i, (n, k), p, balanced=bool(i & 1)) for i in range(4)]
    dev = []
    for x in parts:
        buf = torch.zeros((n, k + pad), dtype=torch.int32, device="cuda")
        buf[:, :k] = torch.from_numpy(x)
        dev.append(buf[:, :k])
    H = lib.aah_quat_modp(*dev, p, H=tuple(torch.full((n, n), -1, dtype=torch.int32, device="cuda")
                                           for _ in range(4)), flags=lib.AAT_ZERO_UPPER)
    ref = oracle.quat_aah_modp_low(*parts, p)
    for h, r in zip(H, ref):
        assert np.array_equal(h.cpu().numpy().astype(np.int64), np.tril(np.asarray(r, dtype=np.int64)))


def _row_relative(got, A, herm):
    """Largest |error| of a lower entry against |a_i| |a_j| (FP64)."""
    Z = A.astype(np.complex128)
    ref = Z @ (Z.conj() if herm else Z).T
    nrm = np.sqrt((np.abs(Z) ** 2).sum(1))
    scale = np.outer(nrm, nrm)
    scale[scale == 0] = 1
    err = np.abs(np.tril(np.where(scale < 1e37, got - ref, 0)) / scale)  # finite in FP32
    return err.max()


def _complex_rows(n, k, kind):
    rng = np.random.default_rng(n * 131 + k)
    A = rng.standard_normal((n, k)) + 1j * rng.standard_normal((n, k))
    if kind == "row_scales":    # one power of ten per row, 1e-15 .. 1e15
        A *= 10.0 ** rng.uniform(-15, 15, (n, 1))
    elif kind == "col_scales":  # every row spans 1e-6 .. 1e6
        A *= 10.0 ** rng.uniform(-6, 6, (1, k))
    elif kind == "zero_rows":
        A[::3] = 0
    elif kind == "huge_row":    # near the end of FP32's range
        A[0] *= 1e32
    return A.astype(np.complex64)


# FP32 class: pieces of 2^-23, dropped products of 2^-22, and FP32 sums of at
# most 512 products per drain, each a rounding of 2^-24 of a partial sum that
# stays below |a_i| |a_j|: (2 + 2 + 4) 2^-23 at the outside of their random
# sizes, 1e-6, taken twice
@pytest.mark.parametrize("kind", ["normal", "row_scales", "col_scales", "zero_rows", "huge_row"])
@pytest.mark.parametrize("n,k", [(1, 1), (5, 3), (33, 64), (130, 257), (300, 515)])
def test_complex_fp32_class_rows_of_any_scale(lib, n, k, kind):
    import torch
    A = _complex_rows(n, k, kind)
    Ad = torch.from_numpy(A).cuda()
    for fn, herm in ((lib.aah_complex, True), (lib.aat_complex, False), (lib.aat_complex_2m, False)):
        got = fn(Ad).cpu().numpy().astype(np.complex128)
        assert _row_relative(got, A, herm) <= 2e-6, fn.__name__


def test_complex_fp32_class_keeps_small_values_beside_an_outlier(lib):
    """Rows whose one large value meets zeros in the other rows: the product
    of their small values keeps FP32 accuracy (BF16 pieces)."""
    import torch
    n, k = 96, 200
    A = _complex_rows(n, k, "normal")
    A[: n // 2, 0] = 1e7
    A[n // 2:, 0] = 0
    for fn, conj in ((lib.aah_complex, True), (lib.aat_complex_2m, False)):
        got = fn(torch.from_numpy(A).cuda()).cpu().numpy().astype(np.complex128)[n // 2:, :n // 2]
        Z = A.astype(np.complex128)
        ref = Z[n // 2:] @ (Z.conj() if conj else Z)[:n // 2].T
        assert np.abs(got - ref).max() <= 1e-5 * k


def test_plan_of_complex_products_mixes_fp16_and_bf16_rows(lib):
    """Every problem of a plan chooses its own form, again on each execution."""
    import torch
    kinds = ["normal", "col_scales", "row_scales", "huge_row", "normal"]
    mats = [_complex_rows(40 + 37 * i, 30 + 61 * i, kd) for i, kd in enumerate(kinds)]
    xs = [torch.from_numpy(m).cuda() for m in mats]
    cs = [torch.zeros((x.shape[0],) * 2, dtype=torch.complex64, device="cuda") for x in xs]
    plan = lib.Plan([("aah", x, c, 0, lib.AAT_C_FP32) for x, c in zip(xs, cs)])
    for swap in (False, True):
        if swap:  # the forms change with the data
            for i, x in enumerate(xs):
                mats[i] = _complex_rows(*mats[i].shape, kinds[(i + 1) % len(kinds)])
                x.copy_(torch.from_numpy(mats[i]))
        plan.execute()
        torch.cuda.synchronize()
        for m, c in zip(mats, cs):
            assert _row_relative(c.cpu().numpy().astype(np.complex128), m, True) <= 2e-6
    plan.close()


@pytest.mark.parametrize("worst", [False, True])
@pytest.mark.parametrize("p", [3, 65521, 1000003, 2147483587, 2**31 - 1])
@pytest.mark.parametrize("n,k", [(1, 1), (15, 127), (16, 128), (17, 129), (33, 4), (96, 160), (50, 1024)])
def test_small_products_in_one_launch(lib, n, k, p, worst):
    """Low(A A^T) and X Y^T of small sizes, with entries at the ends of the
    range (the int64 sums at their largest), strided rows, cleared and kept
    upper triangles."""
    import torch
    if worst:  # squares all of one sign, and products of both signs
        A = np.full((n, k), (p - 1) // 2, dtype=np.int32)
        A[1::2] = -((p - 1) // 2)
        A[::3] = p - 1
    else:
        A = synth.residues(n + k, (n, k), p, balanced=True)
    buf = torch.zeros((n, k + 3), dtype=torch.int32, device="cuda")
    X = buf[:, :k]
    X.copy_(torch.from_numpy(A))
    ref = (A.astype(object) @ A.astype(object).T) % p
    for flags in (0, lib.AAT_ZERO_UPPER):
        C = torch.full((n, n + 1), -5, dtype=torch.int32, device="cuda")
        lib.aat_modp(X, p, C=C[:, :n], flags=flags)
        want = np.tril(ref) + (0 if flags else np.triu(np.full((n, n), -5, dtype=object), 1))
        got = C.cpu().numpy().astype(object)
        assert np.array_equal(got[:, :n], want) and (got[:, n] == -5).all()
    Y = torch.from_numpy(A[: max(1, n // 2)]).cuda()
    got = lib.aat_gemm_modp(X, Y, p).cpu().numpy().astype(object)
    assert np.array_equal(got, ref[:, : max(1, n // 2)])


@pytest.mark.parametrize("pad", [0, 1, 3])
@pytest.mark.parametrize("n,k", [(1030, 300), (1100, 2100), (2900, 40), (4100, 70), (4352, 64)])
def test_leaf_clears_the_upper_triangle(lib, n, k, pad):
    """The tensor-core leaf's own clearing (narrow tiles, wide tiles, CTA
    pairs; split products): every entry of C and nothing beside it."""
    import torch
    p = 65521
    A = synth.residues(n + k, (n, k), p)
    buf = torch.full((n, n + pad), -9, dtype=torch.int32, device="cuda")
    lib.aat_modp(torch.from_numpy(A).cuda(), p, C=buf[:, :n], flags=lib.AAT_ZERO_UPPER, levels=0)
    D = torch.from_numpy(A).cuda().double()     # products < 2^32, sums < 2^53
    ref = torch.remainder((D @ D.T).to(torch.int64), p).tril()
    assert torch.equal(buf[:, :n].to(torch.int64), ref)
    assert bool((buf[:, n:] == -9).all())


@pytest.mark.parametrize("p", [65521, 131071, 1000003, 2**31 - 1])
@pytest.mark.parametrize("M,N,K", [(130, 130, 2500), (700, 300, 4097), (64, 1500, 9000),
                                   (513, 513, 3001), (1001, 1001, 2100)])
def test_leaf_split_into_parts(lib, M, N, K, p):
    """Windows of the plane products and slices of K summed mod p: stored,
    accumulated (beta) and lower, aligned and ragged rows of C."""
    import torch
    from paper_2101_01025_gb300 import testing as T
    lower = M == N
    X = synth.residues(M + K, (M, K), p, balanced=True)
    Y = X if lower else synth.residues(N + 7 * K, (N, K), p, balanced=True)
    Xd, Yd = torch.from_numpy(X).cuda(), torch.from_numpy(Y).cuda()

    def dot(a, b):  # 16-bit halves: FP64 products and sums are exact integers
        return torch.remainder((a @ b.T).to(torch.int64), p)
    xl, yl = torch.remainder(Xd, 65536).double(), torch.remainder(Yd, 65536).double()
    xh = torch.div(Xd - xl.int(), 65536, rounding_mode="floor").double()
    yh = torch.div(Yd - yl.int(), 65536, rounding_mode="floor").double()
    ref = torch.remainder(dot(xh, yh) * ((1 << 32) % p) + dot(xl, yl)
                          + torch.remainder(dot(xl, yh) + dot(xh, yl), p) * 65536, p)
    for ld in (N, (N + 7) // 4 * 4):
        old = torch.from_numpy(synth.residues(3, (M, ld), p)).cuda()
        for acc in (False, True):
            C = old.clone()
            T.leaf(Xd, Xd if lower else Yd, p, C=C[:, :N], lower=lower, accumulate=acc)
            new = torch.remainder(ref + (old[:, :N].to(torch.int64) if acc else 0), p)
            want = old.to(torch.int64)
            want[:, :N] = torch.where(torch.ones_like(new).tril().bool(), new, want[:, :N]) if lower else new
            assert torch.equal(C.to(torch.int64), want)


def test_every_leaf_form_runs_after_the_allocation_free_entry_point(lib):
    """In a fresh process: the allocation-free product first, then products on
    the other one-CTA form and on CTA pairs."""
    import os
    import subprocess
    import sys
    code = """
import torch
import paper_2101_01025_gb300 as aat
from paper_2101_01025_gb300 import _native as nat
p = 65521
X = torch.randint(0, p, (300, 64), dtype=torch.int32, device="cuda")
C = torch.zeros((300, 300), dtype=torch.int32, device="cuda")
s = torch.cuda.current_stream().cuda_stream
nat.check(nat.lib().aat_gemm_modp_noalloc(X.data_ptr(), 64, X.data_ptr(), 64, 300, 300, 64, p,
                                          C.data_ptr(), 300, s))
for n, k in ((700, 700), (4000, 64), (2500, 640)):
    A = torch.randint(0, p, (n, k), dtype=torch.int32, device="cuda")
    D = A.double()
    assert torch.equal(aat.aat_gemm_modp(A, A, p).long(), torch.remainder((D @ D.T).long(), p))
print("ok")
"""
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", code], cwd=root, capture_output=True, text=True,
                       timeout=300)
    assert r.returncode == 0 and "ok" in r.stdout, r.stdout + r.stderr


@pytest.mark.parametrize("p", [65521, 131071, 2**31 - 1])
@pytest.mark.parametrize("M,N,K", [(2500, 4001, 130), (2304, 3970, 64), (2305, 3841, 65)])
def test_half_width_pair_tiles(lib, M, N, K, p):
    """256 x 128 tiles of CTA pairs at their edges (sampled rows, every column)."""
    import torch
    X = synth.residues(M + K, (M, K), p, balanced=True)
    Y = synth.residues(N + 5 * K, (N, K), p, balanced=True)
    got = lib.aat_gemm_modp(torch.from_numpy(X).cuda(), torch.from_numpy(Y).cuda(), p).cpu().numpy()
    rows = sorted({0, 1, 127, 128, 255, 256, 257, 2047, 2048, M - 2, M - 1})
    ref = (X[rows].astype(object) @ Y.astype(object).T) % p
    assert np.array_equal(got[rows].astype(object), ref)


@pytest.mark.parametrize("p", [65537, 65539, 131041, 131071])
@pytest.mark.parametrize("worst", [False, True])
@pytest.mark.parametrize("n,k", [(300, 2200), (1030, 600), (64, 5000)])
def test_two_digits_of_opposite_signs(lib, n, k, p, worst):
    """Primes whose two digits need opposite signs for their pair sum: random
    residues, and sums of one sign at the digits' ends over all of K."""
    import torch
    half = (p - 1) // 2
    if worst:
        ends = np.array([half, -half, half - 255, 65280 if half >= 65280 else half - 1, 1, -1])
        A = np.tile(ends[np.arange(n) % len(ends)][:, None], (1, k)).astype(np.int32)
    else:
        A = synth.residues(n + k, (n, k), p)
    D = torch.from_numpy(A).cuda()
    ref = torch.remainder((D.double() @ D.double().T).to(torch.int64), p)   # < 2^53
    assert torch.equal(lib.aat_gemm_modp(D, D, p).long(), ref)
    for levels in (0, 1, 2):
        got = lib.aat_modp(D, p, levels=levels, flags=lib.AAT_ZERO_UPPER)
        assert torch.equal(got.long(), ref.tril()), levels
    low = lib.aat_modp(D, p, levels=1, flags=lib.AAT_ZERO_UPPER | lib.AAT_LOW_MEMORY)
    assert torch.equal(low.long(), ref.tril())
    C = torch.zeros((n, n), dtype=torch.int32, device="cuda")
    plan = lib.Plan([("modp", D, C, p, 0)])
    plan.execute()
    assert torch.equal(C.long().tril(), ref.tril())
    plan.close()


@pytest.mark.parametrize("zero", [False, True])
@pytest.mark.parametrize("pinned", [False, True])
@pytest.mark.parametrize("p,n,k", [(2**31 - 1, 5000, 2600), (65521, 6200, 4100), (131071, 4700, 1999)])
def test_host_product_in_two_row_parts(lib, p, n, k, pinned, zero):
    """From host memory without recursion levels: both row parts, sampled rows
    against exact sums, cleared or untouched entries above the bands."""
    import torch
    A = torch.from_numpy(synth.residues(n + k, (n, k), p, balanced=True))
    C = torch.full((n, n), -3, dtype=torch.int32)
    if pinned:
        A, C = A.pin_memory(), C.pin_memory()
    for _ in range(2):  # a second call reuses every buffer and event
        C.fill_(-3)
        lib.aat_modp_host(A, p, C=C, flags=lib.AAT_ZERO_UPPER if zero else 0, levels=0)
        rows = sorted({0, 1, 511, 512, n // 2, n - 513, n - 512, n - 2, n - 1} | set(range(2048, n, 517)))
        X = A.numpy()
        for r in rows:
            lo, hi = X[r].astype(np.int64) & 0xffff, X[r].astype(np.int64) >> 16
            Y = X[: r + 1].astype(np.int64)
            ref = ((Y @ hi) % p * 65536 + Y @ lo) % p   # sums below 2^47 p's 2^31: exact in int64
            assert np.array_equal(C[r, : r + 1].numpy().astype(np.int64), ref), r
            if zero:
                assert not C[r, r + 1:].any()
            else:
                assert bool((C[r, (r // 512 + 1) * 512:] == -3).all())


@pytest.mark.parametrize("zero", [False, True])
@pytest.mark.parametrize("p", [65521, 131071, 2**31 - 1])
@pytest.mark.parametrize("n,k,pad", [(4, 8, 0), (66, 132, 0), (130, 64, 3), (512, 512, 0), (1300, 700, 1)])
def test_one_level_in_one_leaf_launch(lib, n, k, pad, p, zero):
    """The last level's five products in one launch and its closing kernel:
    tiles at their edges, cleared and kept surroundings."""
    import torch
    A = torch.from_numpy(synth.residues(n + k, (n, k), p, balanced=True)).cuda()
    buf = torch.full((n, n + pad), -4, dtype=torch.int32, device="cuda")
    lib.aat_modp(A, p, C=buf[:, :n], levels=1, flags=lib.AAT_ZERO_UPPER if zero else 0)
    ref = torch.tril(lib.aat_gemm_modp(A, A, p))   # the plain product (other tests' subject)
    got = buf[:, :n] if zero else torch.tril(buf[:, :n])
    assert torch.equal(got, ref)
    assert bool((buf[:, n:] == -4).all())


@pytest.mark.parametrize("off", [0, 1, 2, 3])
@pytest.mark.parametrize("cols", [1, 3, 4, 5, 125, 126, 127, 128, 129, 130, 131, 132, 509, 1029])
def test_split_reads_only_its_rows(lib, cols, off):
    """Every offset of a row from 16 bytes with the row's end at every offset:
    digits of the row itself, whatever stands before and behind it."""
    import torch
    from paper_2101_01025_gb300 import testing as T
    p, rows = 2**31 - 1, 7
    X = synth.residues(cols, (rows, cols), p, balanced=True)
    ld = cols + 1 + (cols + off) % 3        # rows at changing offsets
    buf = torch.full((off + rows * ld + 8,), 12345, dtype=torch.int32, device="cuda")
    view = torch.as_strided(buf, (rows, cols), (ld, 1), off)
    view.copy_(torch.from_numpy(X))
    b, L, _, _ = T.digit_spec(p, with_sums=True)
    got = T.split(view, p).float().cpu().numpy().astype(np.int64)
    assert np.array_equal(sum(got[i, :, :cols] << (b * i) for i in range(L)), X.astype(np.int64))
    assert not got[:, :, cols:].any()


@pytest.mark.parametrize("p", [131071, 2**31 - 1])
@pytest.mark.parametrize("k", [66000, 120000])
def test_split_parts_of_long_sums(lib, p, k):
    """Parts whose K segments fill the launch's group table."""
    import torch
    n = 200
    A = torch.from_numpy(synth.residues(k, (n, k), p, balanced=True)).cuda()
    got = torch.tril(lib.aat_gemm_modp(A, A, p))
    low = lib.aat_modp(A, p, levels=0, flags=lib.AAT_ZERO_UPPER)
    rows = [0, 1, 127, 128, n - 1]
    X = A.cpu().numpy()
    ref = (X[rows].astype(object) @ X.T.astype(object)) % p
    for i, r in enumerate(rows):
        want = ref[i, :r + 1].astype(np.int64)
        assert np.array_equal(got[r, :r + 1].cpu().numpy().astype(np.int64), want)
        assert np.array_equal(low[r, :r + 1].cpu().numpy().astype(np.int64), want)


# Each of G, H and H^T carries at most 8 2^-23 of its sum of magnitudes (the
# derivation above), and those are at most 2, 1 and 1 times sum |a_l| |b_l|:
# 4e-6.  A value alone in its row between 2^-28 and 2^-33 of the row's largest
# has 2^-17 of itself as FP16 pieces, in the same four sums.
@pytest.mark.parametrize("columns,depth", [(60, 13), (60, 26), (40, 34), (20, 60), (200, 27), (300, 28),
                                           (8, 29), (2, 33), (1, 28), (1, 33), (1, 34), (1, 60)])
def test_complex_fp32_class_entries_of_small_values_only(lib, columns, depth):
    """Rows with `columns` values 2^-depth of the rest (one real value where it
    is 1) against rows that are zero elsewhere: entries made of these alone."""
    import torch
    n, k, h = 96, 400, 48
    rng = np.random.default_rng(100 * columns + depth)
    part = [rng.uniform(1, 2, (n, k)) * rng.choice([-1, 1], (n, k)) for _ in range(2)]
    A = part[0] + 1j * part[1]
    A[:h, :columns] *= 2.0 ** -depth
    A[h:, columns:] = 0
    if columns == 1:
        A[:h, 0] = A[:h, 0].real
    A = np.ascontiguousarray(A[:, rng.permutation(k)].astype(np.complex64))
    Z = A.astype(np.complex128)
    tol = 4e-6 + (4 * 2.0 ** -17 if columns == 1 and 28 < depth <= 33 else 0)
    Ad = torch.from_numpy(A).cuda()
    Cp = torch.zeros((n, n), dtype=torch.complex64, device="cuda")
    plan = lib.Plan([("aah", Ad, Cp, 0, lib.AAT_C_FP32)])
    plan.execute()
    for got, conj in ((lib.aah_complex(Ad), True), (lib.aat_complex(Ad), False),
                      (lib.aat_complex_2m(Ad), False), (Cp, True)):
        ref = (Z @ (Z.conj() if conj else Z).T)[h:, :h]
        mag = (np.abs(Z) @ np.abs(Z).T)[h:, :h]
        err = np.abs(got.cpu().numpy().astype(np.complex128)[h:, :h] - ref) / mag
        assert err.max() <= tol
    plan.close()


@pytest.mark.parametrize("p", [65521, 131071, 2**31 - 1])
@pytest.mark.parametrize("n,k", [(600, 3001), (130, 5000), (3000, 700)])
def test_exact_bits_too_few_for_the_digits_is_an_error(lib, monkeypatch, n, k, p):
    """A bound on the partial sums that the digits cannot keep: no part of a
    split product and no plane pass is left out silently."""
    import torch
    A = torch.from_numpy(synth.residues(n + k, (n, k), p)).cuda()
    calls = [lambda: lib.aat_gemm_modp(A, A, p), lambda: lib.aat_modp(A, p, levels=0),
             lambda: lib.aat_modp(A, p, levels=0, flags=lib.AAT_LOW_MEMORY)]
    want = [c().tril() for c in calls]
    with monkeypatch.context() as m:
        m.setenv("AAT_EXACT_BITS", "20")
        for call in calls:
            with pytest.raises(lib.AatError):
                call()
    for call, w in zip(calls, want):
        assert torch.equal(call().tril(), w)


@pytest.mark.parametrize("pinned", [False, True])
@pytest.mark.parametrize("p", [65521, 131071])
@pytest.mark.parametrize("n,k,leaves", [(512, 300, 2), (2308, 140, 2), (2312, 140, 3), (4096, 516, 3)])
def test_host_product_with_a_level_sends_the_lower_rows_early(lib, n, k, leaves, p, pinned):
    """One level from host memory: P1 first, then the other products, P2 in a
    launch of its own (behind the event that lets the rows below n/2 go back)
    where those rows are many; every entry of the lower triangle."""
    import ctypes
    import torch
    from paper_2101_01025_gb300 import _native as nat
    A = torch.from_numpy(synth.residues(n + k, (n, k), p, balanced=True))
    C = torch.full((n, n), -3, dtype=torch.int32)
    if pinned:
        A, C = A.pin_memory(), C.pin_memory()
    D = A.cuda().double()                        # |sums| < 2^53
    ref = torch.remainder((D @ D.T).to(torch.int64), p).tril()
    prof = nat.Profile()
    for _ in range(2):
        C.fill_(-3)
        nat.check(nat.lib().aat_profile_begin())
        lib.aat_modp_host(A, p, C=C, levels=1)
        nat.check(nat.lib().aat_profile_end(ctypes.byref(prof)))
        assert torch.equal(C.cuda().to(torch.int64).tril(), ref)
        assert prof.launches[2] == leaves        # AAT_K_LEAF_TC


def test_paced_product_is_capturable_once_its_tiles_are_known(lib):
    """In a fresh process: a short product of CTA pairs makes every cache of its
    shape, then a longer one, whose pairs are paced, is captured and replayed."""
    import os
    import subprocess
    import sys
    code = """
import torch
import paper_2101_01025_gb300 as aat
from paper_2101_01025_gb300 import _native as nat
p = 65521
A = torch.randint(0, p, (6144, 33344), dtype=torch.int32, device="cuda")
C = torch.zeros((6144, 6144), dtype=torch.int32, device="cuda")
nat.check(nat.lib().aatx_workspace_reserve(1 << 31))
aat.aat_modp(A[:, :1024], p, C=C, levels=0)
torch.cuda.synchronize()
g = torch.cuda.CUDAGraph()
with torch.cuda.graph(g):
    aat.aat_modp(A, p, C=C, levels=0)
D = A.double()
ref = torch.remainder((D @ D.T).long(), p).tril()
for _ in range(3):
    C.zero_()
    g.replay()
    assert torch.equal(C.long().tril(), ref)
print("ok")
"""
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", code], cwd=root, capture_output=True, text=True,
                       timeout=300)
    assert r.returncode == 0 and "ok" in r.stdout, r.stdout + r.stderr


def test_paced_products_at_once(lib):
    """Two plans of paced products on two streams, more launches than there are
    counter arrays."""
    import torch
    p = 65521
    g = torch.Generator(device="cuda")
    g.manual_seed(5)
    mats = [torch.randint(0, p, (6144, 33344), dtype=torch.int32, device="cuda", generator=g)
            for _ in range(2)]
    outs = [[torch.zeros((6144, 6144), dtype=torch.int32, device="cuda") for _ in range(2)] for _ in mats]
    plans = [lib.Plan([("modp", A, C, p, lib.AAT_ZERO_UPPER) for C in cs]) for A, cs in zip(mats, outs)]
    streams = [torch.cuda.Stream() for _ in plans]
    torch.cuda.synchronize()
    for _ in range(5):
        for plan, s in zip(plans, streams):
            plan.execute(stream=s)
    torch.cuda.synchronize()
    for A, cs in zip(mats, outs):
        D = A.double()
        ref = torch.remainder((D @ D.T).to(torch.int64), p).tril()
        assert all(torch.equal(C.to(torch.int64), ref) for C in cs)
    for plan in plans:
        plan.close()


@pytest.mark.parametrize("p,n,k,launches", [(2**31 - 1, 2048, 8192, 1), (65521, 1024, 256, 1),
                                            (65521, 3000, 3000, 2), (2**31 - 1, 3000, 3000, 2)])
def test_host_row_parts_against_the_one_product_as_it_runs(lib, p, n, k, launches):
    """Two row parts only where the one product, itself in parts of plane
    products where its tiles are few, takes longer (leaf launches of a call)."""
    import ctypes
    import torch
    from paper_2101_01025_gb300 import _native as nat
    A = torch.from_numpy(synth.residues(n + k, (n, k), p, balanced=True)).pin_memory()
    C = torch.zeros((n, n), dtype=torch.int32).pin_memory()
    prof = nat.Profile()
    nat.check(nat.lib().aat_profile_begin())
    lib.aat_modp_host(A, p, C=C, flags=lib.AAT_ZERO_UPPER)
    nat.check(nat.lib().aat_profile_end(ctypes.byref(prof)))
    assert prof.launches[2] == launches          # AAT_K_LEAF_TC
    assert torch.equal(C, lib.aat_modp(A.cuda(), p, flags=lib.AAT_ZERO_UPPER).cpu())
    X = A.numpy().astype(np.int64)
    rows = [0, 1, 511, 512, n // 2, n - 1]
    ref = ((X @ (X[rows] >> 16).T) % p * 65536 + X @ (X[rows] & 0xffff).T) % p
    for i, r in enumerate(rows):
        assert np.array_equal(C[r, :r + 1].numpy().astype(np.int64), ref[:r + 1, i])


@pytest.mark.parametrize("off", [0, 1, 2, 3, 4])
@pytest.mark.parametrize("rows,cols", [(3, 8), (5, 13)])
def test_split_into_planes_at_any_offset(lib, rows, cols, off):
    """Planes whose first word lies `off` words of 16 bits from 16 bytes."""
    import torch
    from paper_2101_01025_gb300 import _native as nat
    from paper_2101_01025_gb300 import testing as T
    p = 2**31 - 1
    X = torch.from_numpy(synth.residues(rows, (rows, cols), p, balanced=True)).cuda()
    want = T.split(X, p).view(torch.int16).flatten()
    buf = torch.full((want.numel() + off + 8,), 77, dtype=torch.int16, device="cuda")
    nat.check(nat.lib().aatx_split(X.data_ptr(), rows, cols, X.stride(0), p,
                                   buf.data_ptr() + 2 * off, T._stream()))
    assert torch.equal(buf[off:off + want.numel()], want)
    assert bool((buf[:off] == 77).all()) and bool((buf[off + want.numel():] == 77).all())


@pytest.mark.parametrize("prec,tol", [("AAT_C_FP32", 1e-5), ("AAT_C_BF16X3", 1e-4)])
@pytest.mark.parametrize("n,k", [(2, 2), (64, 50), (34, 6), (130, 262), (40, 8)])
def test_complex_level_with_ragged_blocks(lib, n, k, prec, tol):
    """One level with halves of k that are and are not whole quads of columns,
    in the class's own bound (relative Frobenius error)."""
    import torch
    A = _complex_rows(n, k, "normal")
    got = lib.aat_complex(torch.from_numpy(A).cuda(), flags=getattr(lib, prec), levels=1).cpu().numpy()
    Z = A.astype(np.complex128)
    ref = np.tril(Z @ Z.T)
    assert np.linalg.norm(np.tril(got) - ref) <= tol * np.linalg.norm(ref)


@pytest.mark.parametrize("n,k,levels", [(300, 700, 0), (260, 132, 1), (1030, 600, 2)])
def test_scratch_limits_with_digits_of_opposite_signs(lib, n, k, levels):
    """Three planes, two planes and plane passes, by flag, limit and failed
    allocation: the same result."""
    import torch
    from paper_2101_01025_gb300 import _native as nat
    p = 131071
    A = torch.from_numpy(synth.residues(n + k, (n, k), p)).cuda()
    D = A.double()
    ref = torch.remainder((D @ D.T).to(torch.int64), p).tril()
    plain = lib.aat_workspace_size(n, k, p, lib.AAT_LEVELS(levels) | nat.AAT_DIGITS_PLAIN)
    fast = lib.aat_workspace_size(n, k, p, lib.AAT_LEVELS(levels))

    def same(flags=0):
        got = lib.aat_modp(A, p, levels=levels, flags=lib.AAT_ZERO_UPPER | flags)
        assert torch.equal(got.to(torch.int64), ref)
    same()
    same(lib.AAT_LOW_MEMORY)
    C = torch.zeros((n, n), dtype=torch.int32, device="cuda")
    lib.aat_syrk_modp(3, A, 0, C, p, flags=lib.AAT_LOW_MEMORY, levels=levels)
    assert torch.equal(C.to(torch.int64).tril(), torch.remainder(3 * ref, p))
    for limit in (max(fast, plain + 1) - 1, plain - 1):
        for flags in (0, lib.AAT_LOW_MEMORY):
            try:
                lib.aat_set_workspace_limit(limit)
                same(flags)
            finally:
                lib.aat_set_workspace_limit(None)
        lib.aat_shutdown()
        try:
            nat.lib().aatx_set_alloc_limit(limit)
            same()
        except lib.AatError as e:
            # no level: the passes need as much as two whole planes
            assert levels == 0 and limit < plain and e.code == nat.AAT_ENOMEM
        finally:
            nat.lib().aatx_set_alloc_limit(2**64 - 1)
