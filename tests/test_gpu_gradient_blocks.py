"""Mixed dE/dtheta block by block, each against its own size: species energies
(whole numbers), dE/dc and dE/dxi, in the one-thread-per-atom kernel, the team
kernel and the batch kernel, against FP64."""
import numpy as np
import pytest

import synth

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


@pytest.mark.parametrize("level,kinds,n_q", [(8, 1, 8), (12, 3, 8), (12, 4, 5), (8, 5, 8), (16, 2, 8), (16, 4, 16)])
@pytest.mark.parametrize("cells", [(2, 3, 2), (5, 4, 7)])
def test_blocks(P, level, kinds, n_q, cells):
    info = P.mtp_basis_info(level)
    raw = synth.raw_potential(level, kinds, n_q, 2.0, 5.0, info["n_mu"], info["m"], 31)
    pot = P.Potential(level, kinds, n_q, 2.0, 5.0, raw.species_energy, 0.05 * raw.radial, raw.xi_raw)
    st = synth.crystal("bcc", cells, 3.16, 0.08, kinds, 4)
    x, z = torch.tensor(st.x, device="cuda"), torch.tensor(st.z, device="cuda")
    nl = P.mtp_build_neighbors(pot, x, st.cell, st.pbc)
    ref = P.mtp_compute_efv(pot, nl, x, z, st.cell, precision=P.MTP_FP64, dtheta=True)["dtheta"].cpu().numpy()
    got = []
    for variant in (1, 2):
        P.mtp_set_efv_variant(pot, variant)
        got.append(P.mtp_compute_efv(pot, nl, x, z, st.cell, dtheta=True)["dtheta"])
    batch = P.mtp_batch_create(pot, [0, st.n], st.cell[None], x)
    got.append(P.mtp_compute_batch(pot, batch, x, z, dtheta=True)["dtheta"].reshape(-1))
    c = slice(kinds, kinds + info["n_mu"] * n_q * kinds * kinds)
    for g in got:
        g = g.cpu().numpy()
        assert np.array_equal(g[:kinds], ref[:kinds])
        for part in (c, slice(c.stop, None)):   # FP32 sums of terms good to ~1e-6
            assert np.linalg.norm(g[part] - ref[part]) <= 2e-5 * np.linalg.norm(ref[part])
