"""Rows whose products are stored as they come (no column repeats, by the kept
counts) when the counts do not hold: the call ends with an error status, stores
nothing outside C's arrays, and the handle works again afterwards. Row lengths
for a warp, for thread groups of 32 to 1024 threads, and at most 32 entries."""
import numpy as np
import pytest

from paper_2105_14156_gb300.rmat import Csr, csr_from_coo
from tests.gpu_util import assert_matches_oracle

pytestmark = pytest.mark.gpu

COLS = 300007
GUARD = 64
KERNELS = [{}, {"warp_rows": 0, "row_window": 0}, {"group_rows": 1}, {"bulk_copy": 1}, {"hash_kind": 2}]


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


def disjoint_pairs(n, dtype, rows=40):
    """A and B with `rows` rows of C, each of n entries from n products: two rows of B without a common column."""
    rng = np.random.default_rng(n)
    r, c = [], []
    for i in range(rows):
        cols = rng.permutation(COLS)[:n]
        for k, part in ((2 * i, cols[:n // 2]), (2 * i + 1, cols[n // 2:])):
            r.append(np.full(part.size, k))
            c.append(part)
    rp, ci = csr_from_coo(2 * rows, COLS, np.concatenate(r), np.concatenate(c))
    B = Csr(2 * rows, COLS, rp, ci, rng.uniform(-1, 1, ci.size).astype(dtype))
    arp, aci = csr_from_coo(rows, 2 * rows, np.repeat(np.arange(rows), 2), np.arange(2 * rows))
    return Csr(rows, 2 * rows, arp, aci, rng.uniform(-1, 1, aci.size).astype(dtype)), B


def guarded(A, B, c_rp, nnz):
    """C for numeric() between guard words, and a check that these are untouched."""
    import torch
    from paper_2105_14156_gb300 import smash
    ci = torch.full((nnz + 2 * GUARD,), -7, dtype=torch.int32, device="cuda")
    val = torch.full((nnz + 2 * GUARD,), -7, dtype=A.val.dtype, device="cuda")

    def check():
        for x in (ci, val):
            assert bool((x[:GUARD] == -7).all()) and bool((x[GUARD + nnz:] == -7).all())
    return smash.DeviceCsr(A.rows, B.cols, c_rp, ci[GUARD:GUARD + nnz], val[GUARD:GUARD + nnz]), check


def expect_refused(handle, dA, dB, c_rp, nnz):
    from paper_2105_14156_gb300 import smash
    C, check = guarded(dA, dB, c_rp, nnz)
    with pytest.raises(smash.SmashError) as e:
        handle.numeric(dA, dB, c_rp, nnz, out=C)
        handle.check()
    assert e.value.status == 1
    check()


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("params", KERNELS, ids=lambda p: "-".join(p) or "default")
@pytest.mark.parametrize("n", [24, 200, 700, 1500, 3000, 7000])
def test_columns_of_b_made_bad_after_the_counts(handle, n, params, dtype):
    from paper_2105_14156_gb300 import smash
    A, B = disjoint_pairs(n, dtype)
    dA, dB = smash.to_device(A), smash.to_device(B)
    base = {k: handle.params.as_dict()[k] for k in params}
    handle.set_params(**params)
    try:
        c_rp, nnz = handle.symbolic(dA, dB)
        good = dB.col_idx.clone()
        for bad in (COLS, -1, 2**31 - 1):
            dB.col_idx[n // 3] = bad                       # one product of the first row
            dB.col_idx[10 * n:10 * n + 2 * n // 3] = bad   # most of the 11th row's
            expect_refused(handle, dA, dB, c_rp, nnz)
            dB.col_idx.copy_(good)
            c_rp, nnz = handle.symbolic(dA, dB)            # (the failure dropped the kept counts)
        C = handle.numeric(dA, dB, c_rp, nnz)
        handle.check()
        assert_matches_oracle(C.to_host(), A, B)
    finally:
        handle.set_params(**base)


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("params", KERNELS, ids=lambda p: "-".join(p) or "default")
@pytest.mark.parametrize("n", [24, 200, 700, 3000])
def test_rows_of_b_emptied_after_the_counts(handle, n, params, dtype):
    """Fewer products than were counted, no bad column among them."""
    from paper_2105_14156_gb300 import smash
    A, B = disjoint_pairs(n, dtype)
    dA, dB = smash.to_device(A), smash.to_device(B)
    base = {k: handle.params.as_dict()[k] for k in params}
    handle.set_params(**params)
    try:
        c_rp, nnz = handle.symbolic(dA, dB)
        dA.col_idx[1] = 0
        dB.row_ptr[1] -= 1   # row 0 of B loses an entry, row 1 begins with it: A's first row reads row 0 twice
        expect_refused(handle, dA, dB, c_rp, nnz)
    finally:
        handle.set_params(**base)


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("params", KERNELS, ids=lambda p: "-".join(p) or "default")
@pytest.mark.parametrize("n", [24, 200, 700, 3000])
def test_bad_columns_in_rows_sized_by_their_bound(handle, n, params, dtype):
    """The one-pass product: rows whose products fit their room, some of them with a bad column."""
    from paper_2105_14156_gb300 import smash
    A, B = disjoint_pairs(n, dtype)
    dA, dB = smash.to_device(A), smash.to_device(B)
    good = dB.col_idx.clone()
    base = {k: handle.params.as_dict()[k] for k in params}
    handle.set_params(**params)
    try:
        for bad in (COLS, -1, 2**31 - 1):
            dB.col_idx[n // 3] = bad
            dB.col_idx[10 * n:10 * n + 2 * n // 3] = bad
            with pytest.raises(smash.SmashError) as e:
                handle.spgemm_learned(dA, dB, None)
            assert e.value.status == 1
            dB.col_idx.copy_(good)
        C, _, owner = handle.spgemm_learned(dA, dB, None)
        assert_matches_oracle(C.to_host(), A, B)
        owner.free()
    finally:
        handle.set_params(**base)


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("params", KERNELS, ids=lambda p: "-".join(p) or "default")
@pytest.mark.parametrize("n", [24, 200, 700, 1500, 3000])
def test_row_pointer_with_an_entry_for_every_product(handle, n, params, dtype):
    """A caller's row pointer that gives a row as many entries as products although one column repeats."""
    import torch
    A, B = disjoint_pairs(n, dtype)
    from paper_2105_14156_gb300 import smash
    B.col_idx[B.row_ptr[21]] = B.col_idx[B.row_ptr[20]]   # one column of the 11th row twice (rows of B may be unsorted)
    dA, dB = smash.to_device(A), smash.to_device(B)
    base = {k: handle.params.as_dict()[k] for k in params}
    handle.set_params(**params)
    try:
        c_rp, nnz = handle.symbolic(dA, dB)
        assert nnz == A.rows * n - 1
        all_products = torch.arange(A.rows + 1, dtype=torch.int64, device="cuda") * n
        expect_refused(handle, dA, dB, all_products, A.rows * n)
        C = handle.spgemm(dA, dB, check=True)
        assert_matches_oracle(C.to_host(), A, B)
    finally:
        handle.set_params(**base)
