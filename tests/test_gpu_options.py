"""Schedule options that a plan takes or refuses, on lengths of every route."""
import pytest

from paper_2005_00322_gb300._abi import PstdError

pytestmark = pytest.mark.gpu
DX = 1e-4
# folded compiled, folded run-time, convolution, convolution beyond the embeddings, dense
LENGTHS = [64, 70, 67, 1301, 37]


def plan(n, schedule):
    from paper_2005_00322_gb300 import Solver
    Solver((n, 6), DX, [("N", "D"), ("N", "N")], cfl=0.2, schedule=[schedule, None]).close()


@pytest.mark.parametrize("n", LENGTHS)
@pytest.mark.parametrize("variant", [None, 0])
@pytest.mark.parametrize("seqs", [0, 3, 512])
def test_line_pairs_that_are_no_power_of_two_are_refused(n, variant, seqs):
    with pytest.raises(PstdError, match="EINVAL"):
        plan(n, (variant, seqs))


@pytest.mark.parametrize("n", [67, 1301, 37, 75])
@pytest.mark.parametrize("variant", [1, 2, 3, 4, 5])
def test_variants_without_a_register_schedule_are_refused(n, variant):
    with pytest.raises(PstdError, match="EINVAL"):
        plan(n, (variant, 1))


# (on 64 a register schedule checks the pairs against its lanes)
@pytest.mark.parametrize("n", LENGTHS[1:])
@pytest.mark.parametrize("schedule", [(None, None), (None, 2), (0, None), (0, 1)])
def test_automatic_and_first_variant_are_taken(n, schedule):
    plan(n, schedule)
