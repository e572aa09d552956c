"""Checkpoint files hold the lattices word by word for the p chains, whatever their order
on the device: written by hand from the spins, and with no memory for a device buffer."""
import os
import subprocess
import sys

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
ISING, POTTS = 0, 1


def lattice_words(model, L, spins):
    """[p, V] spins to the file's [words, p] 32-bit words."""
    p = len(spins)
    per, bits = (32, 1) if model == ISING else (4, 8)
    rw = (L + per - 1) // per
    s = np.zeros((p, L, rw * per), dtype=np.uint64)
    s[:, :, :L] = (spins.reshape(p, L, L) > 0) if model == ISING else spins.reshape(p, L, L)
    w = (s.reshape(p, L, rw, per) << (bits * np.arange(per, dtype=np.uint64))).sum(axis=3)
    return np.ascontiguousarray(w.reshape(p, L * rw).T.astype(np.uint32))


@pytest.mark.parametrize("model,L,p", [(ISING, 4, 1), (ISING, 34, 33), (ISING, 64, 70), (POTTS, 5, 40), (POTTS, 33, 31),
                                       (POTTS, 32, 64)])
def test_file_holds_words_by_chain(tmp_path, model, L, p):
    import paper_1212_3975_gb300 as muca
    path = str(tmp_path / "a.ckpt")
    with muca.Muca(model, L, 2 if model == ISING else 8, p, 8) as g:
        g.iterate(2)
        g.save(path)
        spins = g.get_spins()
    want = lattice_words(model, L, spins).tobytes()
    data = open(path, "rb").read()
    assert data.count(want) == 1 and data.index(want) < 512
    h = muca.Muca.load(path)
    assert np.array_equal(h.get_spins(), spins)
    h.iterate(1)
    h.close()


_CHILD = """
import sys
sys.path.insert(0, %r)
import paper_1212_3975_gb300 as m
try:
    h = m.Muca.load(sys.argv[1])
    h.save(sys.argv[2])
    print("saved")
except m.MucaError as e:
    print(e)
"""


@pytest.mark.parametrize("fail", [17, 18])
def test_no_memory_for_the_buffer(tmp_path, fail):
    """Allocations 1 to 16 are the context's; the next are the buffers of the load and of the
    save, without which the host does the work."""
    import paper_1212_3975_gb300 as muca
    a, b = str(tmp_path / "a.ckpt"), str(tmp_path / "b.ckpt")
    with muca.Muca(POTTS, 33, 8, 31, 8) as g:
        g.iterate(2)
        g.save(a)
    out = subprocess.run([sys.executable, "-c", _CHILD % ROOT, a, b], env=dict(os.environ, MUCA_TEST_FAIL_ALLOC=str(fail)),
                         capture_output=True, text=True, timeout=120)
    assert "saved" in out.stdout, out.stdout + out.stderr
    assert open(a, "rb").read() == open(b, "rb").read()
