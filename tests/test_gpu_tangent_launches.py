"""Tangents of levels up to 16 where the launch changes form: a last, partial wave
launched by itself (FP64 and mixed), and the mixed level-16 kernel without its
staging area, against central differences of forces and dE/dtheta and FP64."""
import pytest

import synth
from tests.helpers import pot_dict

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


@pytest.mark.parametrize("name,kinds,cells", [
    ("bcc-l8-s1", 1, (29, 29, 31)),    # 52,142 atoms: 408 blocks, two per SM in FP64: 104 left over on 152 SMs
    ("bcc-l8-s1", 1, (35, 36, 36)),    # 90,720: 709 blocks, four per SM in FP32
    ("bcc-l16-s3", 3, (34, 34, 34)),   # 78,608: 615 blocks, no staging area in FP32
    ("bcc-l16-s3", 3, (12, 12, 12)),   # 3,456: one launch
])
def test_against_differences(P, name, kinds, cells):
    pot = P.Potential.from_dict(pot_dict(name))
    st = synth.crystal("bcc", cells, 3.16, 0.08, kinds, 2)
    x = torch.tensor(st.x, device="cuda")
    z = torch.tensor(st.z, dtype=torch.int32, device="cuda")
    g = torch.Generator(device="cuda").manual_seed(3)
    v = torch.randn(x.shape, generator=g, device="cuda", dtype=torch.float64)
    nl = P.mtp_build_neighbors(pot, x, st.cell, st.pbc)
    exact = P.mtp_compute_efv_tangent(pot, nl, x, z, st.cell, v, precision=P.MTP_FP64)
    mixed = P.mtp_compute_efv_tangent(pot, nl, x, z, st.cell, v, precision=P.MTP_MIXED)
    h = 1e-5
    hi, lo = (P.mtp_compute_efv(pot, nl, x + s * h * v, z, st.cell, precision=P.MTP_FP64, dtheta=True) for s in (1, -1))
    for k, f in (("dtheta_tan", "dtheta"), ("force_tan", "forces")):
        diff = (hi[f] - lo[f]) / (2 * h)
        # h^2 times third derivatives (some 10 to 100 times the first here) and 1e-15 / h of rounding
        assert float((exact[k] - diff).norm()) <= 1e-7 * float(diff.norm()), k
        # FP32 dual numbers: terms good to ~1e-6, sums that cancel by up to a few ten
        assert float((mixed[k] - exact[k]).norm()) <= 1e-4 * float(exact[k].norm()), k
    assert P.mtp_device_status(pot) == 0
