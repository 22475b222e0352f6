"""A neighbour-list build in place that fails leaves the list as it was: same
offsets and rows, usable for the atoms it was built for."""
import numpy as np
import pytest

import synth
from tests.helpers import pot_dict
from tests.test_gpu_nlist_paths import box

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


def dev(a):
    return torch.tensor(np.asarray(a), dtype=torch.float64, device="cuda")


def failing(x, cell, how):
    """Positions (and cell) of a build that must fail, and its status code."""
    if how == "nan":
        x = x.copy()
        x[len(x) // 2, 1] = np.nan
        return x, cell, -5
    if how == "more atoms":          # the new offsets do not fit in the list's buffer
        x = np.concatenate([x, x + 0.5, [[np.nan, 0.0, 0.0]]])
        return x, cell, -5
    if how == "fewer atoms":
        x = x[: max(1, len(x) // 3)].copy()
        x[0, 0] = np.inf
        return x, cell, -5
    return np.array([[1.0, 1.0, 0.001], [4.0, 2.0, 0.003]]), np.diag([12.0, 12.0, 0.004]), -4   # images beyond +-511


@pytest.mark.parametrize("kind", ["sheared", "cluster", "open", "thin"])   # columns, second search, open axes, images
@pytest.mark.parametrize("how", ["nan", "more atoms", "fewer atoms", "thin cell"])
def test_list_survives_a_failed_build(P, kind, how):
    x, cell, pbc = box(kind)
    pot = P.Potential.from_dict(pot_dict("bcc-l8-s1"))
    nl = P.mtp_build_neighbors(pot, dev(x), cell, pbc)
    before = [t.clone() for t in nl.to_tensors()]
    info = nl.info()
    bad, bad_cell, code = failing(x, cell, how)
    for _ in range(2):
        with pytest.raises(P.MtpError) as e:
            P.mtp_build_neighbors(pot, dev(bad), bad_cell, (1, 1, 1) if how == "thin cell" else pbc, nlist=nl)
        assert e.value.code == code
    assert nl.info() == info
    assert all(torch.equal(a, b) for a, b in zip(before, nl.to_tensors()))
    P.mtp_build_neighbors(pot, dev(x), cell, pbc, nlist=nl)
    assert all(torch.equal(a, b) for a, b in zip(before, nl.to_tensors()))


def test_empty_rows_are_published(P):
    """A list rebuilt to no pairs at all, and back."""
    pot = P.Potential.from_dict(pot_dict("bcc-l8-s1"))
    st = synth.crystal("bcc", (4, 4, 4), 3.16, 0.1, 1, 1)
    far = np.diag([20.0, 20.0, 20.0])
    nl = P.mtp_build_neighbors(pot, dev(st.x[:2] * [1, 1, 0] + [[0, 0, 0], [9.0, 9.0, 9.0]]), far, (1, 1, 1))
    assert nl.info() == (2, 0) and not nl.to_tensors()[0].any()
    P.mtp_build_neighbors(pot, dev(st.x), st.cell, st.pbc, nlist=nl)
    ref = P.mtp_build_neighbors(pot, dev(st.x), st.cell, st.pbc)
    assert all(torch.equal(a, b) for a, b in zip(ref.to_tensors(), nl.to_tensors()))
    P.mtp_build_neighbors(pot, dev([[1.0, 1.0, 1.0]]), far, (1, 1, 1), nlist=nl)
    off, j, _ = nl.to_tensors()
    assert nl.info() == (1, 0) and off.tolist() == [0, 0] and j.numel() == 0
