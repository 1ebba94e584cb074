"""How many rows a cluster of the decode merge takes: a host function of the batch, the heads and the clusters that fit at once."""
import pytest

from tests.helpers import merge_variant


@pytest.fixture(scope="module")
def B():
    from paper_2603_04411_b200 import build
    build.build()
    from paper_2603_04411_b200 import binding
    return binding


@pytest.mark.parametrize("fit", [1, 18, 45, 52, 1000])
def test_fewest_rows_that_leave_all_clusters_resident(B, fit):
    """Heads of a slot are taken together before slots are; 32 rows only where sixteen are too few."""
    for rep in (1, 2, 4, 8):
        forms = [(1 << k, 1) for k in range(rep.bit_length())]
        forms += [(rep, n) for n in (2, 4, 8, 16) if rep * n <= 16]
        for hkv in range(1, 9):
            for n_seq in list(range(1, 70)) + [128, 500, 4096]:
                # (one slot more than half of the sequences already brings them all into one cluster per group of heads)
                fits = [hp * ns for hp, ns in forms if ns < 2 * n_seq and -(-n_seq // ns) * hkv * (rep // hp) <= fit]
                assert merge_variant(B, n_seq, hkv, rep, fit) == (fits[0] if fits else 32), (rep, hkv, n_seq, fit)
