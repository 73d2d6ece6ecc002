"""Dense rows whose products are shared out over a block's warps: rows of B
around the lengths where a warp changes from steps over several rows to rounds
inside one (48 products left) and from a masked round to a whole one (128; 48
beyond one: 176), also as the only row of B that a row of A reads, so that the
warps' parts of it end on either side; rows of A around a batch of 32 entries,
entries without products, bitmap words and windows with a ragged end, zero
products of either sign. Values are held to |c - c*| <= tol * sum |a||b| (1e-5
float32, 1e-12 float64). An entry of C has at most 84 terms (as many
as B has rows; 35 in the tests with more rows), and a sum of m products in any order
is within m * 2^-24 of it: 5.0e-6; small integers, zeros among them, must be exact."""
import numpy as np
import pytest

from paper_2105_14156_gb300.rmat import Csr, csr_from_coo
from tests.gpu_util import assert_matches_oracle
from tests.helpers import random_csr

pytestmark = pytest.mark.gpu

LENS = [0, 1, 31, 32, 33, 47, 48, 49, 0, 64, 127, 128, 129, 160, 175, 176, 177, 255, 256, 257, 1000, 4096, 6000]
PER_WARP = [m * w for w in (8, 16, 32) for m in (47, 48, 49, 128, 176)]   # lengths of the parts of 8 to 32 warps


@pytest.fixture(scope="module")
def handle():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2105_14156_gb300 import build, smash
    build.build()
    h = smash.Handle(0)
    yield h
    h.close()


def values_of(rng, kind, n):
    if kind == "int":
        return rng.integers(-3, 4, n).astype(np.float64)
    return rng.uniform(-1, 1, n).astype(np.float32 if kind == "f32" else np.float64)


def operands(cols, kind, seed):
    rng = np.random.default_rng(seed)
    lens = [min(n, cols) for n in LENS * 3 + PER_WARP]
    k = len(lens)
    r = np.repeat(np.arange(k), lens)
    c = np.concatenate([rng.permutation(cols)[:n] for n in lens])
    rp, ci = csr_from_coo(k, cols, r, c)
    B = Csr(k, cols, rp, ci, values_of(rng, kind, ci.size))
    a_lens = [1, 2, 3, 31, 32, 33, k, 17, 5, 40] + [1] * len(PER_WARP)
    r = np.repeat(np.arange(len(a_lens)), a_lens)
    c = np.concatenate([rng.permutation(k)[:n] for n in a_lens[:10]] + [np.arange(k - len(PER_WARP), k)])
    rp, ci = csr_from_coo(len(a_lens), k, r, c)
    return Csr(len(a_lens), k, rp, ci, values_of(rng, kind, ci.size)), B


@pytest.mark.parametrize("kind", ["f32", "f64", "int"])
@pytest.mark.parametrize("cols", [7000, 12287, 12289, 40961, 131071])
def test_dense_row_shapes(handle, cols, kind):
    from paper_2105_14156_gb300 import smash
    A, B = operands(cols, kind, cols)
    handle.set_params(dense_ratio=1 << 20, sym_dense_ratio=1 << 20)
    try:
        dA, dB = smash.to_device(A), smash.to_device(B)
        assert_matches_oracle(handle.spgemm(dA, dB, check=True).to_host(), A, B, exact=kind == "int")
        C, _, owner = handle.spgemm_learned(dA, dB, None)
        assert_matches_oracle(C.to_host(), A, B, exact=kind == "int")
        owner.free()
    finally:
        handle.set_params(dense_ratio=4, sym_dense_ratio=64)


def test_dense_row_bad_columns_are_reported(handle):
    """A column of B past cols(B) in a dense row of either kind of pass: an error status, nothing out of range."""
    from paper_2105_14156_gb300 import smash
    A, B = operands(12289, "f32", 3)
    B.col_idx[int(B.row_ptr[15]) - 1] = 12289   # the last column of a long row
    handle.set_params(dense_ratio=1 << 20, sym_dense_ratio=1 << 20)
    try:
        dA, dB = smash.to_device(A), smash.to_device(B)
        with pytest.raises(smash.SmashError) as e:
            handle.symbolic(dA, dB)
        assert e.value.status == 1
        with pytest.raises(smash.SmashError) as e:
            handle.spgemm_learned(dA, dB, None)
        assert e.value.status == 1
    finally:
        handle.set_params(dense_ratio=4, sym_dense_ratio=64)


@pytest.mark.parametrize("cols", [8192, 12289])
@pytest.mark.parametrize("bad", ["cols", "cols + 1", "-1", "2**31 - 1"])
def test_dense_row_counts_after_a_bad_column(handle, cols, bad):
    """Columns out of range share the bit past the bitmap's last column (in a spare word where cols(B) fills the
    others): reported once, and not left in the counts of the next rows or products."""
    from paper_2105_14156_gb300 import smash
    A, B = operands(cols, "int", 5)
    good = B.col_idx.copy()
    B.col_idx[int(B.row_ptr[15]) - 1] = eval(bad, {"cols": cols})
    handle.set_params(sym_dense_ratio=1 << 20)
    try:
        with pytest.raises(smash.SmashError) as e:
            handle.symbolic(smash.to_device(A), smash.to_device(B))
        assert e.value.status == 1
        B.col_idx = good
        C = handle.spgemm(smash.to_device(A), smash.to_device(B), check=True).to_host()
        assert_matches_oracle(C, A, B, exact=True)
    finally:
        handle.set_params(sym_dense_ratio=64)


@pytest.mark.parametrize("kind", ["int", "f64"])
def test_dense_rows_counted_before_and_not(handle, kind):
    """The numeric count pass over rows that the symbolic bitmap counted (at least half the columns) and rows that it
    did not (a few products), in turn and many to a block: the sizes of both are checked, and match."""
    from paper_2105_14156_gb300 import smash
    cols, rng = 7000, np.random.default_rng(8)
    lens = [3600, 5, 3501, 1, 4097, 40, 3555, 3]   # rows of B
    r = np.repeat(np.arange(len(lens)), lens)
    c = np.concatenate([rng.permutation(cols)[:n] for n in lens])
    rp, ci = csr_from_coo(len(lens), cols, r, c)
    B = Csr(len(lens), cols, rp, ci, values_of(rng, kind, ci.size))
    pick = rng.integers(0, len(lens), 9000)   # one row of B each: several rows for each resident block
    rp, ci = csr_from_coo(pick.size, len(lens), np.arange(pick.size), pick)
    A = Csr(pick.size, len(lens), rp, ci, values_of(rng, kind, ci.size))
    handle.set_params(dense_ratio=1 << 20, sym_dense_ratio=2)
    try:
        assert_matches_oracle(handle.spgemm(smash.to_device(A), smash.to_device(B), check=True).to_host(), A, B,
                              exact=kind == "int")
    finally:
        handle.set_params(dense_ratio=4, sym_dense_ratio=64)


@pytest.mark.parametrize("kind", ["f32", "f64", "int"])
@pytest.mark.parametrize("per", [1, 3, 15, 17, 60, 130])
def test_dense_rows_of_short_rows_of_b(handle, per, kind):
    """Rows of B from one entry to more than a batch is worth: the warps of a block take whole batches of a row of A in
    turn below 16 products an entry, and up to 128 the rows with a batch for a fourth of the warps or for each."""
    from paper_2105_14156_gb300 import smash
    cols, k, rng = 9001, 1200, np.random.default_rng(per)
    lens = rng.integers(max(0, per - 2), per + 3, k)
    r = np.repeat(np.arange(k), lens)
    c = np.concatenate([rng.permutation(cols)[:n] for n in lens])
    rp, ci = csr_from_coo(k, cols, r, c)
    B = Csr(k, cols, rp, ci, values_of(rng, kind, ci.size))
    a_lens = [1, 31, 32, 33, 63, 64, 65, 127, 128, 129, 255, 256, 257, 511, 512, 513, 1024, 1025, k]
    r = np.repeat(np.arange(len(a_lens)), a_lens)
    c = np.concatenate([rng.permutation(k)[:n] for n in a_lens])
    rp, ci = csr_from_coo(len(a_lens), k, r, c)
    A = Csr(len(a_lens), k, rp, ci, values_of(rng, kind, ci.size))
    handle.set_params(dense_ratio=1 << 20, sym_dense_ratio=1 << 20)
    try:
        dA, dB = smash.to_device(A), smash.to_device(B)
        assert_matches_oracle(handle.spgemm(dA, dB, check=True).to_host(), A, B, exact=kind == "int")
        C, _, owner = handle.spgemm_learned(dA, dB, None)
        assert_matches_oracle(C.to_host(), A, B, exact=kind == "int")
        owner.free()
    finally:
        handle.set_params(dense_ratio=4, sym_dense_ratio=64)
