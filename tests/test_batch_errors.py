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


@pytest.mark.parametrize("model,L,fits", [(ISING, 64, True), (ISING, 160, True), (ISING, 164, False),
                                          (ISING, 224, True), (ISING, 256, False), (POTTS, 68, True),
                                          (POTTS, 80, False), (POTTS, 128, False)])
def test_batches_stage_what_single_contexts_stage(muca, model, L, fits):
    """Lattices in shared memory: a batch and a context of its own take and refuse the same."""
    q = 2 if model == ISING else 8
    with muca.Muca(model, L, q, 3, 1, staging=1) as g:
        if fits:
            want = g.iterate(1)
        else:
            with pytest.raises(muca.MucaError):
                g.iterate(1)
    if not fits:
        with pytest.raises(muca.MucaError) as ei:
            muca.MucaBatch([(model, L, q, 3, 1)], staging=1)
        assert ei.value.code == muca._muca.MUCA_ERR_ARG and "shared memory" in str(ei.value)
        return
    b = muca.MucaBatch([(model, L, q, 3, 1)], staging=1)
    b.iterate(1, 1)
    assert (b.job(0).get_histogram() == want).all()
    b.close()


@pytest.mark.parametrize("job", [(ISING, 132, 2, 5, 2), (ISING, 224, 2, 3, 2), (ISING, 240, 2, 9, 2), (ISING, 256, 2, 6, 2),
                                 (ISING, 260, 2, 5, 2), (ISING, 292, 2, 2, 2), (POTTS, 132, 8, 5, 2), (POTTS, 160, 8, 3, 2)])
def test_long_rows_in_a_batch(muca, job):
    """Rows of several passes and every histogram of theirs (32-bit and 16-bit counts in shared
    memory, global): a batch and a context of its own agree bit for bit."""
    b = muca.MucaBatch([job, (ISING, 8, 2, 8, 1)])
    b.iterate(2, 2)
    with muca.Muca(*job) as g:
        for _ in range(2):
            H = g.iterate(2)
            g.update_weights()
        v = b.job(0)
        assert (v.get_histogram() == H).all() and (v.get_lnw() == g.get_lnw()).all()
        assert (v.get_spins() == g.get_spins()).all()
    b.close()
