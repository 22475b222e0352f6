"""Neighbour lists on every route of the build against the oracle's brute
force, bit for bit: found-neighbour columns with 1, 2 and 4 threads per atom,
columns that run over (clusters far denser than the box), cells thinner than
the search (several images of one atom), rows longer than the ordering buffer,
open axes, unwrapped positions, one atom, and lists rebuilt in place."""
import numpy as np
import pytest

import synth
from oracle import mtp as O
from tests.test_gpu_parity import gpu_pot

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def P():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_00193_gb300 import build as B
    B.build()
    import paper_2510_00193_gb300 as P
    return P


def box(kind):
    g = np.random.default_rng(11)
    if kind == "one":
        return np.array([[0.3, 0.2, 0.1]]), np.diag([9.0, 8.0, 7.0]), (1, 1, 1)
    if kind == "sheared":
        st = synth.crystal("bcc", (5, 4, 7), 3.16, 0.1, 1, 1)
        return st.x, st.cell + np.array([[0, 0, 0], [2.1, 0, 0], [-1.7, 3.3, 0]]), (1, 1, 1)
    if kind == "cluster":      # 300 atoms in a corner of a large box: most columns run over
        return g.uniform(0.0, 7.0, (300, 3)), np.diag([60.0, 50.0, 40.0]), (1, 1, 1)
    if kind == "open":
        return g.uniform(-20.0, 20.0, (400, 3)), np.diag([40.0, 13.0, 11.0]), (0, 1, 0)
    if kind == "thin":         # thinner than the cutoff along two axes
        return g.uniform(0.0, 4.0, (23, 3)), np.array([[3.1, 0, 0], [0.4, 4.2, 0], [0.2, -0.6, 25.0]]), (1, 1, 1)
    if kind == "dense":        # about 1,700 neighbours per atom
        st = synth.crystal("bcc", (3, 3, 3), 0.85, 0.02, 1, 1)
        return st.x, st.cell, (1, 1, 1)
    st = synth.crystal("bcc", (6, 6, 6), 3.16, 0.1, 1, 1)   # unwrapped: whole cells added per atom
    return st.x + g.integers(-2, 3, (st.n, 3)) @ st.cell, st.cell, (1, 1, 1)


def check(P, nl, x, cell, pbc, r_cut, sample=40):
    off, j, img = (t.cpu().numpy() for t in nl.to_tensors())
    q = np.unique(np.linspace(0, len(x) - 1, min(sample, len(x))).astype(int))
    i, jo, no = O.neighbor_list(x, cell, pbc, r_cut, query=q)
    for k in q:
        rows = i == k
        assert off[k + 1] - off[k] == rows.sum()
        assert np.array_equal(j[off[k]:off[k + 1]], jo[rows])
        assert np.array_equal(img[off[k]:off[k + 1]], no[rows])
    return off[-1]


@pytest.mark.parametrize("kind", ["one", "sheared", "cluster", "open", "thin", "dense", "unwrapped"])
def test_list_routes(P, kind):
    x, cell, pbc = box(kind)
    pot = gpu_pot(P, "bcc-l8-s1")
    xd = torch.tensor(x, device="cuda")
    nl = P.mtp_build_neighbors(pot, xd, cell, pbc)
    check(P, nl, x, cell, pbc, pot.r_cut, 6 if kind in ("dense", "unwrapped") else 40)
    first = [t.clone() for t in nl.to_tensors()]
    P.mtp_build_neighbors(pot, xd, cell, pbc, nlist=nl)     # in place, with room for the rows
    assert all(torch.equal(a, b) for a, b in zip(first, nl.to_tensors()))


@pytest.mark.parametrize("cells", [(24, 24, 24), (32, 33, 31), (40, 47, 41)])
def test_threads_per_atom(P, cells):
    """27,648, 65,472 and 154,160 atoms: 4, 2 and 1 threads per atom; built over a list of another size."""
    st = synth.crystal("bcc", cells, 3.16, 0.1, 1, 1)
    pot = gpu_pot(P, "bcc-l8-s1")
    small = synth.crystal("bcc", (4, 4, 4), 3.16, 0.1, 1, 1)
    nl = P.mtp_build_neighbors(pot, torch.tensor(small.x, device="cuda"), small.cell, small.pbc)
    P.mtp_build_neighbors(pot, torch.tensor(st.x, device="cuda"), st.cell, st.pbc, nlist=nl)
    total = check(P, nl, st.x, st.cell, st.pbc, pot.r_cut, 12)
    off, j, _ = (t.cpu().numpy() for t in nl.to_tensors())
    assert total == len(j)
    # a full list holds every pair from both sides
    deg = np.bincount(j, minlength=st.n)
    assert np.array_equal(deg, np.diff(off))
    P.mtp_build_neighbors(pot, torch.tensor(small.x, device="cuda"), small.cell, small.pbc, nlist=nl)
    check(P, nl, small.x, small.cell, small.pbc, pot.r_cut)
