"""Mixed dE/dtheta of levels 18 and 20 on more than 4,096 atoms for species
counts and radial basis sizes at which the coefficients alone fill 32 to 216 KB
of shared memory: the graph kernels against the tile program (smaller ranges of
the same box), and against FP64 where its coefficients fit."""
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


@pytest.mark.parametrize("level", [18, 20])
@pytest.mark.parametrize("kinds,n_q", [(8, 10), (9, 8), (6, 16), (16, 16)])
def test_many_species(P, level, kinds, n_q):
    info = P.mtp_basis_info(level)
    raw = synth.raw_potential(level, kinds, n_q, 2.0, 5.0, info["n_mu"], info["m"], 18)
    pot = P.Potential(level, kinds, n_q, 2.0, 5.0, raw.species_energy, 0.02 * raw.radial, raw.xi_raw)
    st = synth.crystal("fcc", (7, 12, 13), 3.6, 0.1, kinds, 6)   # 4,368 atoms
    x, z = torch.tensor(st.x, device="cuda"), torch.tensor(st.z, device="cuda")
    nl = P.mtp_build_neighbors(pot, x, st.cell, st.pbc)

    def run(precision, chunk=0):
        out = P.mtp_compute_efv(pot, nl, x, z, st.cell, precision=precision, dtheta=True, chunk_atoms=chunk)
        assert P.mtp_device_status(pot) == 0
        return out["dtheta"].cpu().numpy(), out["forces"].cpu().numpy()

    got = run(P.MTP_MIXED)
    refs = [run(P.MTP_MIXED, 1001)] + ([run(P.MTP_FP64)] if kinds < 16 else [])
    c = slice(kinds, kinds + info["n_mu"] * n_q * kinds * kinds)
    for dtheta, forces in refs:
        assert np.array_equal(dtheta[:kinds], got[0][:kinds])            # atoms per species
        for part in (c, slice(c.stop, None)):   # dE/dc, dE/dxi: FP32 sums of terms good to ~1e-6, on either side
            assert np.linalg.norm(got[0][part] - dtheta[part]) <= 2e-5 * np.linalg.norm(dtheta[part])
        assert np.linalg.norm(got[1] - forces) <= 2e-5 * np.linalg.norm(forces)
