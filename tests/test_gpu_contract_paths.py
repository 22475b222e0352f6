"""Mixed-precision contraction of levels 18 and 20: the straight-line graph
kernels (ranges of 4,096 atoms and more) against the tile program (smaller
ranges, reached by chunking the same box) and against FP64, with dE/dtheta and
ragged ends; and the tile program at one atom, one tile and its neighbours."""
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


def potential(P, level):
    if level == 20:
        return P.Potential.from_dict(pot_dict("fcc-l20-s4")), 4
    info = P.mtp_basis_info(level)
    raw = synth.raw_potential(level, 2, 7, 2.0, 5.0, info["n_mu"], info["m"], 18)
    # radial functions of O(1) moments, basis terms of comparable size (levels grow by powers of the moments)
    return P.Potential(level, 2, 7, 2.0, 5.0, raw.species_energy, 0.02 * raw.radial, raw.xi_raw), 2


def run(P, pot, st, precision, chunk=0):
    x, z = torch.tensor(st.x, device="cuda"), torch.tensor(st.z, device="cuda")
    nl = P.mtp_build_neighbors(pot, x, st.cell, st.pbc)
    out = P.mtp_compute_efv(pot, nl, x, z, st.cell, precision=precision, dtheta=True, chunk_atoms=chunk)
    assert P.mtp_device_status(pot) == 0
    return {k: v.cpu().numpy() for k, v in out.items()}


def off(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


@pytest.mark.parametrize("level", [18, 20])
@pytest.mark.parametrize("cells", [(8, 16, 8), (11, 10, 13)])   # 4,096 and 5,720 atoms
def test_graph_kernels_against_tiles_and_fp64(P, level, cells):
    pot, kinds = potential(P, level)
    st = synth.crystal("fcc", cells, 3.6, 0.1, kinds, 3)
    ref = run(P, pot, st, P.MTP_FP64)
    graphs, tiles = run(P, pot, st, P.MTP_MIXED), run(P, pot, st, P.MTP_MIXED, chunk=1001)
    ragged = run(P, pot, st, P.MTP_MIXED, chunk=4097)
    for k in ("e_atom", "forces", "dtheta"):
        own = off(tiles[k], ref[k])
        # both round in FP32; errors of one path are taken as the scale for the other
        assert own <= 2e-5
        for o in (graphs, ragged):
            assert off(o[k], ref[k]) <= 4 * own + 1e-6


@pytest.mark.parametrize("n", [1, 2, 7, 8, 9, 129])
def test_tile_edges(P, n):
    """n atoms of a random gas: FP64 against the same atoms in chunks of one (one atom per tile)."""
    pot, kinds = potential(P, 20)
    st = synth.random_gas(n, 0.085, 1.9, kinds, synth.rng(3, 300 + n))
    a = run(P, pot, st, P.MTP_FP64)
    b = run(P, pot, st, P.MTP_FP64, chunk=1)
    m = run(P, pot, st, P.MTP_MIXED)
    for k in ("e_atom", "forces", "dtheta"):
        if np.linalg.norm(b[k]) > 0:
            scale = np.abs(b[k]).max()
            assert np.abs(a[k] - b[k]).max() <= 1e-10 * max(1.0, scale)
            assert np.abs(m[k] - b[k]).max() <= 2e-3 * max(1.0, scale)


@pytest.mark.parametrize("cells", [(1, 1, 1), (3, 3, 3), (6, 5, 5), (7, 7, 7), (10, 10, 10), (17, 16, 16)])
def test_team_lanes_per_atom(P, cells):
    """2 to 8,704 atoms: 16 to 1 lanes per atom in the team kernel, against one thread per atom (level 16)."""
    pot = P.Potential.from_dict(pot_dict("bcc-l16-s3"))
    st = synth.crystal("bcc", cells, 3.16, 0.08, 3, 2)
    P.mtp_set_efv_variant(pot, 1)
    ref, mixed_ref = run(P, pot, st, P.MTP_FP64), run(P, pot, st, P.MTP_MIXED)
    P.mtp_set_efv_variant(pot, 2)
    got, mixed = run(P, pot, st, P.MTP_FP64), run(P, pot, st, P.MTP_MIXED)
    for k in ("e_atom", "forces", "virial", "dtheta"):
        scale = max(1.0, np.abs(ref[k]).max())
        assert np.abs(got[k] - ref[k]).max() <= 1e-11 * scale
        assert np.abs(mixed[k] - ref[k]).max() <= 4 * np.abs(mixed_ref[k] - ref[k]).max() + 1e-6 * scale
