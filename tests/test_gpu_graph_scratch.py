"""A captured evaluation replayed after a larger call has outgrown the handle's
scratch: the graph's own scratch is still there and the results are the same."""
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


@pytest.mark.parametrize("precision", [0, 1])   # FP64, mixed
@pytest.mark.parametrize("name,lattice,a,kinds", [("fcc-l20-s4", "fcc", 3.6, 4), ("bcc-l16-s3", "bcc", 3.16, 3)])
def test_replay_after_growth(P, precision, name, lattice, a, kinds):
    pot = P.Potential.from_dict(pot_dict(name))

    def made(cells):
        st = synth.crystal(lattice, cells, a, 0.08, kinds, 11)
        x = torch.tensor(st.x, device="cuda")
        return st, x, torch.tensor(st.z, dtype=torch.int32, device="cuda"), P.mtp_build_neighbors(pot, x, st.cell, st.pbc)

    st, x, z, nl = made((5, 5, 5))
    ref = P.mtp_compute_efv(pot, nl, x, z, st.cell, precision=precision)
    ref = {k: v.clone() for k, v in ref.items() if torch.is_tensor(v)}
    graphs = []
    for cells in ((9, 9, 9), (12, 12, 12)):
        out = {k: torch.zeros_like(v) for k, v in ref.items()}
        out["dtheta"] = None
        graph = torch.cuda.CUDAGraph()
        torch.cuda.synchronize()
        with torch.cuda.graph(graph):
            P.mtp_compute_efv(pot, nl, x, z, st.cell, precision=precision, out=out)
        graphs.append((graph, out))
        big, xb, zb, nb = made(cells)
        other = P.Potential.from_dict(pot_dict(name))
        for p in (pot, other):   # outgrows the scratch; the second handle takes what the first would have freed
            P.mtp_compute_efv(p, nb, xb, zb, big.cell, precision=precision)
    for graph, out in graphs:
        graph.replay()
        torch.cuda.synchronize()
        for k, r in ref.items():
            # the same sums in another order: FP64 1e-11; FP32 forces, about 100 additions of 6e-8 on partial
            # sums a few times the largest force
            tol = 1e-11 if precision == 0 or k == "e_atom" else 2e-5
            assert (out[k] - r).abs().max() <= tol * r.abs().max(), k
    assert P.mtp_device_status(pot) == 0


def test_capture_with_room_for_the_tile_program_only(P):
    """4,200 atoms at level 20, mixed, captured when earlier calls have sized the scratch for the moments but
    not for the graph values: the tile program runs on them, against the graph kernels of an ordinary call."""
    st = synth.crystal("fcc", (7, 10, 15), 3.6, 0.1, 4, 11)
    assert st.n == 4200
    x, z = torch.tensor(st.x, device="cuda"), torch.tensor(st.z, dtype=torch.int32, device="cuda")
    pot, other = (P.Potential.from_dict(pot_dict("fcc-l20-s4")) for _ in range(2))
    nl = P.mtp_build_neighbors(pot, x, st.cell, st.pbc)
    ref = P.mtp_compute_efv(other, nl, x, z, st.cell, dtheta=True)
    exact = P.mtp_compute_efv(other, nl, x, z, st.cell, precision=P.MTP_FP64, dtheta=True)
    out = {k: torch.zeros_like(v) for k, v in ref.items()}
    P.mtp_compute_efv(pot, nl, x, z, st.cell, chunk_atoms=1000)                           # the mixed path's own scratch
    P.mtp_compute_efv(pot, nl, x, z, st.cell, precision=P.MTP_FP64, chunk_atoms=2520)     # between the two sizes
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        P.mtp_compute_efv(pot, nl, x, z, st.cell, dtheta=True, out=out)
    graph.replay()
    torch.cuda.synchronize()
    for k in ("e_atom", "forces", "virial", "dtheta"):
        r = exact[k]
        off = [float((o[k] - r).norm() / r.norm()) for o in (out, ref)]
        assert off[0] <= 2e-5 and off[1] <= 2e-5, (k, off)   # FP32 sums of terms good to ~1e-6
    assert P.mtp_device_status(pot) == 0
