"""dE/dtheta of the mixed path at level 18: the sweeps' accumulators in columns
of shared memory (up to four species, n_q up to its largest), pairs straight
into the block's (five species), and basis values summed in groups of 32 (a
ragged last warp), below and above the size at which the contraction changes
kernels, against FP64."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("kinds,n_q", [(1, 3), (4, 16), (5, 8), (3, 10)])
@pytest.mark.parametrize("cells", [(3, 3, 3), (7, 12, 13)])   # 108 and 4,368 atoms
def test_mixed_gradient(kinds, n_q, cells):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_00193_gb300 import build as B
    B.build()
    import paper_2510_00193_gb300 as P
    info = P.mtp_basis_info(18)
    raw = synth.raw_potential(18, kinds, n_q, 2.0, 5.0, info["n_mu"], info["m"], 18)
    pot = P.Potential(18, kinds, n_q, 2.0, 5.0, raw.species_energy, 0.02 * raw.radial, raw.xi_raw)
    st = synth.crystal("fcc", cells, 3.6, 0.1, kinds, 6)
    x, z = torch.tensor(st.x, device="cuda"), torch.tensor(st.z, device="cuda")
    nl = P.mtp_build_neighbors(pot, x, st.cell, st.pbc)
    ref, got = (P.mtp_compute_efv(pot, nl, x, z, st.cell, precision=p, dtheta=True) for p in (P.MTP_FP64, P.MTP_MIXED))
    assert P.mtp_device_status(pot) == 0
    r, g = ref["dtheta"].cpu().numpy(), got["dtheta"].cpu().numpy()
    c = slice(kinds, kinds + info["n_mu"] * n_q * kinds * kinds)
    assert np.array_equal(r[:kinds], g[:kinds])            # atoms per species
    for part in (c, slice(c.stop, None)):                  # dE/dc, dE/dxi: FP32 sums of terms good to ~1e-6
        assert np.linalg.norm(g[part] - r[part]) <= 2e-5 * np.linalg.norm(r[part])
