"""What a batch refuses, and with which reason; batches beside each other."""
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


def test_a_smaller_batch_leaves_a_larger_one_its_shared_memory(muca):
    large = muca.MucaBatch([(ISING, 64, 2, 8, 1)])
    small = muca.MucaBatch([(ISING, 8, 2, 8, 1)])
    large.iterate(1, 2)
    small.iterate(1, 2)
    assert int(large.job(0).get_histogram().sum()) == 2 * 8 * 64 * 64
    assert int(small.job(0).get_histogram().sum()) == 2 * 8 * 8 * 8
    small.close()
    large.close()
