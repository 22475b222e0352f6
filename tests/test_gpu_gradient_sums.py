"""dE/dtheta through every form of the lanes' sum: staged across the warp (up to
four species; n_q = 8 keeps the accumulators as 16-byte vectors), lane by lane
where the staging does not fit (level 12, four species, n_q = 16, 256-thread
batch blocks), and straight into the block's accumulators (five species).
Single configuration, batch and FP64 against one another."""
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


@pytest.mark.parametrize("level,kinds,n_q,threads", [(8, 1, 8, 32), (12, 3, 8, 64), (12, 4, 16, 256), (12, 4, 5, 128),
                                                     (8, 5, 8, 64), (16, 2, 8, 32)])
def test_parameter_gradient(P, level, kinds, n_q, threads):
    info = P.mtp_basis_info(level)
    raw = synth.raw_potential(level, kinds, n_q, 2.0, 5.0, info["n_mu"], info["m"], 31)
    pot = P.Potential(level, kinds, n_q, 2.0, 5.0, raw.species_energy, 0.05 * raw.radial, raw.xi_raw)
    sts = [synth.crystal("bcc", c, 3.16, 0.08, kinds, 4, k) for k, c in enumerate([(2, 3, 2), (3, 3, 2), (5, 4, 4)])]
    off = np.concatenate([[0], np.cumsum([s.n for s in sts])])
    x = torch.tensor(np.concatenate([s.x for s in sts]), device="cuda")
    z = torch.tensor(np.concatenate([s.z for s in sts]), device="cuda")
    batch = P.mtp_batch_create(pot, off, np.array([s.cell for s in sts]), x, atoms_per_block=threads)
    ref = []
    for k, st in enumerate(sts):
        xk, zk = x[off[k]:off[k + 1]].contiguous(), z[off[k]:off[k + 1]].contiguous()
        nl = P.mtp_build_neighbors(pot, xk, st.cell, st.pbc)
        for variant in (1, 2):
            P.mtp_set_efv_variant(pot, variant)
            o = [P.mtp_compute_efv(pot, nl, xk, zk, st.cell, precision=p, dtheta=True)["dtheta"].cpu().numpy()
                 for p in (P.MTP_FP64, P.MTP_MIXED)]
            scale = np.abs(o[0]).max()
            if variant == 1:
                ref.append(o[0])
            # FP64 sums of at most a few thousand terms; FP32 terms of about 1e-6 relative error
            assert np.abs(o[0] - ref[-1]).max() <= 1e-11 * scale
            assert np.abs(o[1] - ref[-1]).max() <= 1e-4 * scale
    ref = np.array(ref)
    scale = np.abs(ref).max(axis=1, keepdims=True)
    for p, tol in ((P.MTP_FP64, 1e-11), (P.MTP_MIXED, 1e-4)):
        got = P.mtp_compute_batch(pot, batch, x, z, precision=p, dtheta=True)["dtheta"].cpu().numpy()
        assert np.all(np.abs(got - ref) <= tol * scale)
