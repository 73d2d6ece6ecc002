"""Products whose B is narrow enough for a warp's dense accumulator, at the
sizes where its lane groups, its unrolled steps and its choice of rows can go
wrong: mean row lengths of B on both sides of each group width, rows of B of
one to many steps, column counts around a multiple of 32 and around the widest
accumulator, rows of A for a chunk, a warp and a block, unsorted and repeated
columns. Values are held to |c - c*| <= tol * sum |a||b|, 1e-5 in float32 and 1e-12
in float64: a sum of m products in any order is within m * 2^-24 (2^-53) of it, which
stays below for the m <= 119 of these operands, except in the phases with one column,
where a row of 300 entries meets in one entry of C (m = 300, 1.8e-5: `terms`). Small
integers must be exact."""
import numpy as np
import pytest

from paper_2105_14156_gb300.rmat import Csr, csr_from_coo
from tests.gpu_util import assert_matches_oracle
from tests.helpers import random_csr

pytestmark = pytest.mark.gpu


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


def rows_of(lens, cols, values, seed):
    """A CSR matrix whose row r holds lens[r] distinct, ascending columns."""
    rng = np.random.default_rng(seed)
    r = np.repeat(np.arange(len(lens)), lens)
    c = np.concatenate([rng.permutation(cols)[:n] for n in lens]) if sum(lens) else np.zeros(0, np.int64)
    rp, ci = csr_from_coo(len(lens), cols, r, c)
    if values == "int":
        val = rng.integers(1, 5, ci.size).astype(np.float32)
    else:
        val = rng.uniform(-1, 1, ci.size).astype(np.float32 if values == "f32" else np.float64)
    return Csr(len(lens), cols, rp, ci, val)


def skewed_rows(n, k, values, seed, longest):
    """n rows of 0 .. ~10 entries, one of `longest` and one of all k."""
    rng = np.random.default_rng(seed)
    lens = rng.integers(0, min(k, 10) + 1, n)
    lens[n // 3] = min(k, longest)
    lens[n - 1] = k
    return rows_of(lens.tolist(), k, values, seed + 1)


# (cols, entries per row of B): every lane-group width, rows of one step, of
# two, and of more, and the widest accumulators
B_SHAPES = [(1, [1]), (31, [1, 2]), (32, [0, 4, 8]), (33, [6, 9, 16]), (100, [8, 17]), (256, [12, 16, 33]),
            (300, [15, 16, 17, 32, 33, 130]), (1000, [40, 64, 65, 129, 600]), (3072, [30, 700]), (3073, [30]),
            (6144, [30, 2000]), (6145, [30])]


def b_matrix(cols, lens, k, values, seed):
    return rows_of([min(lens[q % len(lens)], cols) for q in range(k)], cols, values, seed)


def run_batch_device(handle, pairs):
    Cs, _, owner = handle.spgemm_batched(pairs)
    host = [C.to_host() for C in Cs]
    owner.free()
    return host


def run_batch(handle, pairs):
    from paper_2105_14156_gb300 import smash
    return run_batch_device(handle, [(smash.to_device(A), smash.to_device(B)) for A, B in pairs])


@pytest.mark.parametrize("values", ["f32", "f64", "int"])
def test_batched_narrow_shapes(handle, values):
    pairs = [(skewed_rows(70 + 3 * q, 40, values, 11 * q, 37), b_matrix(cols, lens, 40, values, 7 * q + 1))
             for q, (cols, lens) in enumerate(B_SHAPES)]
    for (A, B), C in zip(pairs, run_batch(handle, pairs)):
        assert_matches_oracle(C, A, B, exact=values == "int")


@pytest.mark.parametrize("values", ["f32", "f64"])
def test_batched_narrow_row_sizes(handle, values):
    """Rows for a chunk (512 products or fewer), a warp and a block (above 8192), and their neighbours."""
    k = 700
    B = b_matrix(256, [16], k, values, 3)
    lens = [32, 33, 31, 511, 512, 513, 0, 1, 700, 699, 64, 65] + [5] * 50
    A = rows_of(lens, k, values, 4)
    for C in run_batch(handle, [(A, B), (A, B)]):
        assert_matches_oracle(C, A, B)


@pytest.mark.parametrize("values", ["f64", "int"])
def test_batched_narrow_unsorted_and_repeated(handle, values):
    """Unsorted or repeated columns in one B of a batch, next to a B that ascends and a wide one."""
    A = random_csr(90, 60, 0.2, 21, values=values)
    B = random_csr(60, 200, 0.1, 22, values=values, sort_cols=False, dup_frac=0.3)
    S = random_csr(60, 200, 0.1, 23, values=values)
    D = Csr(S.rows, S.cols, S.row_ptr, S.col_idx.copy(), S.val)
    s = int(S.row_ptr[7])
    assert S.row_ptr[8] - s >= 2
    D.col_idx[s + 1] = D.col_idx[s]   # one repeated column, else ascending
    W = random_csr(60, 20000, 0.002, 24, values=values)
    pairs = [(A, B), (A, S), (A, D), (A, W)]
    for (x, y), C in zip(pairs, run_batch(handle, pairs)):
        assert_matches_oracle(C, x, y, exact=values == "int")


@pytest.mark.parametrize("values", ["f32", "f64", "int"])
@pytest.mark.parametrize("cols,lens", B_SHAPES)
def test_narrow_phases(handle, cols, lens, values):
    """The two phases and the one-pass product on every shape, heavy rows (more than 256 entries) among them."""
    from paper_2105_14156_gb300 import smash
    k = 300
    B = b_matrix(cols, lens, k, values, 5)
    A = skewed_rows(150, k, values, 6, 257)
    dA, dB = smash.to_device(A), smash.to_device(B)
    terms = k if cols == 1 else 0
    assert_matches_oracle(handle.spgemm(dA, dB, check=True).to_host(), A, B, exact=values == "int", terms=terms)
    C, _, owner = handle.spgemm_learned(dA, dB, None)
    assert_matches_oracle(C.to_host(), A, B, exact=values == "int", terms=terms)
    owner.free()


@pytest.mark.parametrize("values", ["f64", "int"])
def test_narrow_phases_unsorted_and_repeated(handle, values):
    from paper_2105_14156_gb300 import smash
    A = random_csr(300, 400, 0.1, 31, values=values)
    B = random_csr(400, 900, 0.02, 32, values=values, sort_cols=False, dup_frac=0.3)
    C = handle.spgemm(smash.to_device(A), smash.to_device(B), check=True).to_host()
    assert_matches_oracle(C, A, B, exact=values == "int")


def test_narrow_wrong_sizes_are_reported(handle):
    """A row pointer of C that is not this product's: an error status, nothing written past a row's room."""
    import torch
    from paper_2105_14156_gb300 import smash
    A, B = random_csr(64, 50, 0.3, 41, values="f32"), random_csr(50, 300, 0.2, 42, values="f32")
    dA, dB = smash.to_device(A), smash.to_device(B)
    c_rp, nnz = handle.symbolic(dA, dB)
    short = torch.arange(65, dtype=torch.int64, device="cuda") * 70   # rows hold about 280 entries
    with pytest.raises(smash.SmashError) as e:
        handle.numeric(dA, dB, short, 64 * 70)
        handle.check()
    assert e.value.status == 1
    assert_matches_oracle(handle.spgemm(dA, dB, check=True).to_host(), A, B)


def test_bad_columns_by_the_million_are_reported(handle):
    """2**24 rows of B that ascend and end in a column past cols(B): still no plain adds, and an error status."""
    import torch
    from paper_2105_14156_gb300 import smash
    k, cols = 1 << 24, 256
    b_rp = torch.arange(k + 1, dtype=torch.int64, device="cuda") * 3
    b_ci = torch.tensor([3, 100, cols + 5], dtype=torch.int32, device="cuda").repeat(k)
    B = smash.DeviceCsr(k, cols, b_rp, b_ci, torch.ones(3 * k, device="cuda"))
    rows = 1024
    a_rp = torch.arange(rows + 1, dtype=torch.int64, device="cuda") * (k // rows)
    A = smash.DeviceCsr(rows, k, a_rp, torch.arange(k, dtype=torch.int32, device="cuda"), torch.ones(k, device="cuda"))
    with pytest.raises(smash.SmashError) as e:
        handle.spgemm_learned(A, B, None)
    assert e.value.status == 1
    with pytest.raises(smash.SmashError) as e:
        handle.spgemm_batched([(A, B)])
    assert e.value.status == 1


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
def test_rows_of_b_that_start_twice_at_one_place(handle, dtype):
    """A row of B whose end lies before its start, not read by A, so that two others begin at one place; the row after
    them has a repeated column. The row counts as no more than what A reads of it."""
    import torch
    from paper_2105_14156_gb300 import smash
    rng = np.random.default_rng(3)
    cols = 64
    first = np.sort(rng.permutation(cols)[:10])
    second = np.sort(rng.permutation(first[-1])[:10])      # begins below the first one's end
    third = np.sort(rng.permutation(cols)[:40])
    third[20] = third[21]
    ci = np.concatenate([first, second, third]).astype(np.int32)
    val = rng.uniform(-1, 1, 60).astype(dtype)
    rp = np.array([0, 10, 20, 10, 20, 60], np.int64)       # rows 1 and 3 are the same, row 2 has no extent
    n = 64
    reads = np.array([0, 1, 3, 4])
    a_val = rng.uniform(-1, 1, 4 * n).astype(dtype)
    B = smash.DeviceCsr(5, cols, *(torch.as_tensor(x, device="cuda") for x in (rp, ci, val)))
    A = smash.DeviceCsr(n, 5, *(torch.as_tensor(x, device="cuda") for x in
                                (np.arange(n + 1) * 4, np.tile(reads, n).astype(np.int32), a_val)))
    want, room = np.zeros((n, cols)), np.zeros((n, cols))
    for i in range(n):
        for q, r in enumerate(reads):
            np.add.at(want[i], ci[rp[r]:rp[r + 1]], float(a_val[4 * i + q]) * val[rp[r]:rp[r + 1]].astype(np.float64))
            np.add.at(room[i], ci[rp[r]:rp[r + 1]], abs(float(a_val[4 * i + q])) * abs(val[rp[r]:rp[r + 1]].astype(np.float64)))
    results = [handle.spgemm(A, B, check=True).to_host()]
    C, _, owner = handle.spgemm_learned(A, B, None)
    results.append(C.to_host())
    owner.free()
    results += run_batch_device(handle, [(A, B)])
    tol = 8 * np.finfo(dtype).eps   # at most five terms an entry: (m - 1 + 1) * u a term, u = eps / 2
    for C in results:
        got = np.zeros((n, cols))
        for i in range(n):
            got[i, C.col_idx[C.row_ptr[i]:C.row_ptr[i + 1]]] = C.val[C.row_ptr[i]:C.row_ptr[i + 1]]
            assert set(C.col_idx[C.row_ptr[i]:C.row_ptr[i + 1]]) == set(np.flatnonzero(room[i]))
        assert (abs(got - want) <= tol * room).all()


@pytest.mark.parametrize("values", ["f32", "f64", "int"])
def test_narrow_phases_of_long_rows_alike(handle, values):
    """Rows of A all longer than the least heavy row: a warp each where they are many, a block where they are few."""
    from paper_2105_14156_gb300 import smash
    for rows in (20, 6000):
        B = b_matrix(1000, [2, 3, 1], 400, values, 5)
        A = rows_of([147 + 3 * (q % 5) for q in range(rows)], 400, values, 6)
        dA, dB = smash.to_device(A), smash.to_device(B)
        assert_matches_oracle(handle.spgemm(dA, dB, check=True).to_host(), A, B, exact=values == "int")


@pytest.mark.parametrize("values", ["f32", "f64", "int"])
@pytest.mark.parametrize("cols", [64, 129, 256, 257, 2048])
@pytest.mark.parametrize("rows", [3, 4, 400])
def test_narrow_products_few_and_many(handle, rows, cols, values):
    """Fewer products than B has entries (added atomically) and more (with lane groups where copies fit)."""
    from paper_2105_14156_gb300 import smash
    pairs = []
    for q, per in enumerate((2, 6, 12, 40)):
        B = b_matrix(cols, [per, per + 1], 600, values, 7 + q)
        A = rows_of([150] * rows, 600, values, 8 + q)   # 600 entries of A and up: as many as B has rows
        pairs.append((A, B))
        C = handle.spgemm(smash.to_device(A), smash.to_device(B), check=True).to_host()
        assert_matches_oracle(C, A, B, exact=values == "int")
    for (A, B), C in zip(pairs, run_batch(handle, pairs)):
        assert_matches_oracle(C, A, B, exact=values == "int")


@pytest.mark.parametrize("values", ["f32", "f64", "int"])
@pytest.mark.parametrize("cols", [1024, 1025, 1536, 1537, 3072, 3073])
@pytest.mark.parametrize("per,entries", [(12, 60), (3, 240), (40, 250)])
def test_narrow_rows_or_windows(handle, cols, per, entries, values):
    """Columns around the sizes where a warp's accumulator gives way to tables and windows, with 3 and with 12 products
    an entry, about half the columns or more than twice as many (the widest: as many) products a row."""
    from paper_2105_14156_gb300 import smash
    B = b_matrix(cols, [per], 400, values, 3)
    A = rows_of([entries, max(1, entries // 3), max(1, entries // 9)] * 30, 400, values, 4)
    dA, dB = smash.to_device(A), smash.to_device(B)
    assert_matches_oracle(handle.spgemm(dA, dB, check=True).to_host(), A, B, exact=values == "int")
    C, _, owner = handle.spgemm_learned(dA, dB, None)
    assert_matches_oracle(C.to_host(), A, B, exact=values == "int")
    owner.free()


@pytest.mark.parametrize("values", ["f32", "f64", "int"])
@pytest.mark.parametrize("mix", ["sparse", "filled", "one wide", "half wide", "even", "skewed"])
def test_batched_accumulators_or_tables(handle, mix, values):
    """Wide-ish products whose rows are too empty for a warp's accumulator, or full enough; one of them among many
    narrow ones, which keep their shared memory, or enough of them to be worth it; rows in between, all alike or a few
    that outgrow a warp's table."""
    cols = 2900 if values == "f64" else 5800   # below the widest accumulator, above the default table's bytes

    def pair(n, a, c, b, seed):
        lens = [a] * n if isinstance(a, int) else [a[q % len(a)] for q in range(n)]
        return rows_of(lens, 60, values, seed), b_matrix(c, [b], 60, values, seed + 1)
    empty, full = (100, 2, cols, 5), (100, 40, cols, 40)
    small = [(80, 8, 256, 12)] * 12
    sizes = {"sparse": [empty] * 6, "filled": [full] * 6, "one wide": small + [full[:1] + (3,) + full[2:]],
             "half wide": small + [full] * 3, "even": [(100, 8, cols, 18)] * 6,
             "skewed": [(100, (2, 2, 60, 2, 2), cols, 18)] * 6}[mix]
    pairs = [pair(*s, 5 * q) for q, s in enumerate(sizes)]
    for (A, B), C in zip(pairs, run_batch(handle, pairs)):
        assert_matches_oracle(C, A, B, exact=values == "int")


@pytest.mark.parametrize("values", ["f32", "int"])
@pytest.mark.parametrize("cols", [2049, 3584, 3585])
@pytest.mark.parametrize("entries", [5, 8])
def test_batched_light_accumulators(handle, cols, entries, values):
    """Rows that fill more and less than a 32nd of B's columns, up to the last accumulator of which a block holds one
    for each of its warps, and one column more."""
    per = cols // (30 * 5)
    pairs = [(rows_of([entries] * 90, 60, values, 3 * q), b_matrix(cols, [per], 60, values, 3 * q + 1)) for q in range(5)]
    for (A, B), C in zip(pairs, run_batch(handle, pairs)):
        assert_matches_oracle(C, A, B, exact=values == "int")
