"""A call that the library refuses on the host leaves nothing behind that fails the next one."""
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


@pytest.mark.parametrize("call", ["efv", "batch"])
def test_valid_call_after_a_refused_one(P, call):
    """16 species with n_q = 16: the FP64 coefficients and dE/dc sums exceed a block's shared memory."""
    info = P.mtp_basis_info(20)
    raw = synth.raw_potential(20, 16, 16, 2.0, 5.0, info["n_mu"], info["m"], 18)
    pot = P.Potential(20, 16, 16, 2.0, 5.0, raw.species_energy, 0.02 * raw.radial, raw.xi_raw)
    st = synth.crystal("fcc", (3, 3, 3), 3.6, 0.1, 16, 6)
    x, z = torch.tensor(st.x, device="cuda"), torch.tensor(st.z, dtype=torch.int32, device="cuda")
    nl = P.mtp_build_neighbors(pot, x, st.cell, st.pbc)
    batch = P.mtp_batch_create(pot, [0, st.n], st.cell[None], x)
    with pytest.raises(P.MtpError) as e:
        if call == "efv":
            P.mtp_compute_efv(pot, nl, x, z, st.cell, precision=P.MTP_FP64, dtheta=True)
        else:
            P.mtp_compute_batch(pot, batch, x, z, precision=P.MTP_FP64, dtheta=True)
    assert e.value.code == -2
    P.mtp_build_neighbors(pot, x, st.cell, st.pbc, nlist=nl)
    a = P.mtp_compute_efv(pot, nl, x, z, st.cell, precision=P.MTP_FP64)["forces"]
    b = P.mtp_compute_batch(pot, batch, x, z, precision=P.MTP_FP64)["forces"]
    assert (a - b).abs().max() <= 1e-10 * a.abs().max()   # the same FP64 sums in another order
    assert P.mtp_device_status(pot) == 0
