"""What a batch refuses, and with which reason."""
import pytest

pytestmark = pytest.mark.gpu

ISING, POTTS = 0, 1


@pytest.fixture(scope="module")
def muca():
    import paper_1212_3975_gb300 as m
    from paper_1212_3975_gb300 import build
    build.build()
    return m


@pytest.mark.parametrize("job", [(ISING, 6, 2, 8, 1), (ISING, 18, 2, 8, 1), (ISING, 90, 2, 8, 1), (POTTS, 5, 8, 8, 1),
                                 (POTTS, 30, 8, 8, 1), (POTTS, 255, 8, 8, 1)])
def test_ragged_side_names_the_reason(muca, job):
    with pytest.raises(muca.MucaError) as ei:
        muca.MucaBatch([(ISING, 8, 2, 8, 1), job])
    assert ei.value.code == muca._muca.MUCA_ERR_ARG
    assert "L % 4 == 0 (job 1)" in str(ei.value)
