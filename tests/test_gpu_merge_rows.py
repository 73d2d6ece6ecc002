"""Rows that merge little: staged and merged after the sort up to a quarter more
products than entries, hashed above it. Each row of A selects two rows of B that
share d columns, so a row of C has n entries from n + d products: n around the
bins' ends, d at none, one, n // 4 and n // 4 + 1, in the exact phases (warp and
thread-group rows) and the one-pass product. Every entry has one or two terms:
float results are within 2^-23 (2^-52) of |a||b| sums, far inside the checked
1e-5 (1e-12); small integers must be exact."""
import numpy as np
import pytest

from paper_2105_14156_gb300.rmat import Csr, csr_from_coo
from tests.gpu_util import assert_matches_oracle

pytestmark = pytest.mark.gpu

SIZES = [4, 32, 33, 63, 64, 65, 127, 128, 129, 205, 255, 256, 257, 409, 410, 511, 512, 513, 1023, 1024, 1025, 2047, 2049,
         4095, 4097]


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


def overlapping_pairs(kind, cols=300007, seed=5):
    rng = np.random.default_rng(seed)
    rows, cs, ar, ac = [], [], [], []
    k = 0
    for n in SIZES:
        for d in sorted({0, 1, n // 4, n // 4 + 1}):
            c = rng.permutation(cols)[:n]
            half = (n - d) // 2 + d   # first row: `half` columns, the last d of them in the second row too
            for part in (c[:half], c[half - d:]):
                rows.append(np.full(part.size, k))
                cs.append(part)
                ac.append(k)
                k += 1
            ar += [len(ac) // 2 - 1] * 2
    rp, ci = csr_from_coo(k, cols, np.concatenate(rows), np.concatenate(cs))
    arp, aci = csr_from_coo(len(ac) // 2, k, np.array(ar), np.array(ac))

    def values(m):
        if kind == "int":
            return rng.integers(1, 5, m).astype(np.float32)
        return rng.uniform(-1, 1, m).astype(np.float32 if kind == "f32" else np.float64)
    return Csr(len(ac) // 2, k, arp, aci, values(aci.size)), Csr(k, cols, rp, ci, values(ci.size))


@pytest.mark.parametrize("kind", ["f32", "f64", "int"])
def test_rows_that_merge_little(handle, kind):
    from paper_2105_14156_gb300 import smash
    A, B = overlapping_pairs(kind)
    dA, dB = smash.to_device(A), smash.to_device(B)
    assert_matches_oracle(handle.spgemm(dA, dB, check=True).to_host(), A, B, exact=kind == "int")
    C, _, owner = handle.spgemm_learned(dA, dB, None)
    assert_matches_oracle(C.to_host(), A, B, exact=kind == "int")
    owner.free()


@pytest.mark.parametrize("params", [{"bulk_copy": 1}, {"hash_kind": 2}, {"bulk_copy": 1, "hash_kind": 2}],
                         ids=lambda p: "-".join(p))
@pytest.mark.parametrize("kind", ["f32", "f64", "int"])
def test_rows_that_merge_little_with_either_write_out(handle, kind, params):
    """The same with the bulk copy-out and the order-preserving hash, which one kernel serves in both modes."""
    from paper_2105_14156_gb300 import smash
    A, B = overlapping_pairs(kind)
    dA, dB = smash.to_device(A), smash.to_device(B)
    handle.set_params(**params)
    try:
        assert_matches_oracle(handle.spgemm(dA, dB, check=True).to_host(), A, B, exact=kind == "int")
        C, _, owner = handle.spgemm_learned(dA, dB, None)
        assert_matches_oracle(C.to_host(), A, B, exact=kind == "int")
        owner.free()
    finally:
        handle.set_params(bulk_copy=0, hash_kind=1)


@pytest.mark.parametrize("kind,cols", [("f32", c) for c in (338200, 338304, 338320, 338368, 338369)]
                         + [("f64", c) for c in (59700, 59776, 59800, 59840, 59841)])
def test_bitmaps_that_fill_shared_memory(handle, kind, cols):
    """Rows of the largest tables (4097 to 8192 entries) where the column bitmap beside the table takes all of a
    block's 227 KB but the last few words, or one more than there is."""
    from paper_2105_14156_gb300 import smash
    rng = np.random.default_rng(cols)
    lens = [4097, 5000, 3000, 8192]
    r = np.repeat(np.arange(len(lens)), lens)
    rp, ci = csr_from_coo(len(lens), cols, r, np.concatenate([rng.permutation(cols)[:n] for n in lens]))
    dtype = np.float32 if kind == "f32" else np.float64
    B = Csr(len(lens), cols, rp, ci, rng.uniform(-1, 1, ci.size).astype(dtype))
    ac = [0, 1, 2, 3, 0, 2, 1, 2]   # one row of B each, then pairs
    rp, ci = csr_from_coo(6, len(lens), np.array([0, 1, 2, 3, 4, 4, 5, 5]), np.array(ac))
    A = Csr(6, len(lens), rp, ci, rng.uniform(-1, 1, ci.size).astype(dtype))
    dA, dB = smash.to_device(A), smash.to_device(B)
    assert_matches_oracle(handle.spgemm(dA, dB, check=True).to_host(), A, B)
    C, _, owner = handle.spgemm_learned(dA, dB, None)
    assert_matches_oracle(C.to_host(), A, B)
    owner.free()
