"""Grade with rows in the order of their lengths and the re-check spread over
the blocks: 2,662 atoms (three groups of 1,024, the last one ragged) in two
chunks against the FP64 method, and basis rows against the same grades."""
import json
import os

import pytest

import synth
from tests.helpers import ROOT, pot_dict

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("tau_sel", [2.0, 0.01])   # 0.01: almost no row near a threshold
def test_tensor_method_against_fp64(tau_sel):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_00193_gb300 import build as B
    B.build()
    import paper_2510_00193_gb300 as P
    st = synth.crystal("bcc", (11, 11, 11), 3.16, 0.15, 1, 5)
    pot = P.Potential.from_dict(pot_dict("bcc-l16-s1"))
    with open(os.path.join(ROOT, "potentials", "bcc-l16-s1-active.json")) as fh:
        a_inv = torch.tensor(json.load(fh)["a_inv"], dtype=torch.float64, device="cuda").view(pot.m, pot.m)
    x, z = torch.tensor(st.x, device="cuda"), torch.tensor(st.z, device="cuda")
    nl = P.mtp_build_neighbors(pot, x, st.cell, st.pbc)
    kw = dict(a_inv=a_inv, tau_sel=tau_sel, tau_brk=10.0)
    ref = P.mtp_compute_grade(pot, nl, x, z, st.cell, method=P.MTP_GRADE_FP64, **kw)
    got = P.mtp_compute_grade(pot, nl, x, z, st.cell, method=P.MTP_GRADE_TENSOR, chunk_atoms=1500, **kw)
    # the products cancel by ~5e7: FP64 rounding alone reaches ~1e-8 relative
    assert torch.equal(got["flags"], ref["flags"])
    assert torch.all((got["gamma"] - ref["gamma"]).abs() <= 1e-7 * ref["gamma"].abs() + 1e-7)
    gamma = (P.mtp_compute_basis_rows(pot, nl, x, z, st.cell) @ a_inv).abs().max(1).values
    assert torch.all((gamma - ref["gamma"]).abs() <= 1e-6 * gamma + 1e-6)
