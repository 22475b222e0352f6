"""Mixed forces with and without dE/dtheta on random gases with pairs closer
than R_min (whose second sweep differs between the two), as a batch and one
configuration at a time, against FP64."""
import numpy as np
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


@pytest.mark.parametrize("level", [8, 16, 20])
def test_close_pairs(P, level):
    if level == 16:
        pot = P.Potential.from_dict(pot_dict("gas-l16-s2"))
    else:
        info = P.mtp_basis_info(level)
        raw = synth.raw_potential(level, 2, 8, 2.0, 5.0, info["n_mu"], info["m"], 18)
        pot = P.Potential(level, 2, 8, 2.0, 5.0, raw.species_energy, 0.02 * raw.radial, raw.xi_raw)
    sts = synth.random_gas_batch(12, 8, 256, 0.085, 1.9, 2, 4, workers=1)
    off = np.concatenate([[0], np.cumsum([s.n for s in sts])]).astype(np.int64)
    x = torch.tensor(np.concatenate([s.x for s in sts]), device="cuda")
    z = torch.tensor(np.concatenate([s.z for s in sts]), dtype=torch.int32, device="cuda")
    batch = P.mtp_batch_create(pot, off, np.array([s.cell for s in sts]), x)

    def one_by_one(precision, dtheta):
        f = []
        for k, st in enumerate(sts):
            xk, zk = x[off[k]:off[k + 1]].contiguous(), z[off[k]:off[k + 1]].contiguous()
            nl = P.mtp_build_neighbors(pot, xk, st.cell, st.pbc)
            o, j, img = nl.to_tensors()
            i = torch.repeat_interleave(torch.arange(st.n, device="cuda"), o.diff())
            d = xk[j.long()] + img.double() @ torch.tensor(st.cell, device="cuda") - xk[i]
            close.append(int((d.norm(dim=1) < 2.0).sum()))
            f.append(P.mtp_compute_efv(pot, nl, xk, zk, st.cell, precision=precision, dtheta=dtheta)["forces"])
        return torch.cat(f)

    close = []
    exact = one_by_one(P.MTP_FP64, False)
    assert sum(close) > 20
    scale = float(exact.abs().max())

    def rms(f):
        return float((f - exact).square().mean().sqrt())

    batched = [rms(P.mtp_compute_batch(pot, batch, x, z, precision=P.MTP_MIXED, dtheta=d)["forces"]) for d in (False, True)]
    single = [rms(one_by_one(P.MTP_MIXED, d)) for d in (False, True)]
    assert P.mtp_device_status(pot) == 0
    # roundings of one size on either side, a few close pairs dominating both
    for plain, with_dtheta in (batched, single):
        assert plain <= 1e-4 * scale
        assert with_dtheta <= 4 * plain + 1e-6 * scale
