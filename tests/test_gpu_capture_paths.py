"""FP64 energies and forces captured into a CUDA graph as the first call of a
handle: no scratch of the handle may be allocated then (the row order at
level 16, the split kernels' moments at level 20)."""
import pytest

import synth
from tests.helpers import pot_dict

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("name,lattice,cells,a,species", [
    ("bcc-l16-s3", "bcc", (18, 18, 18), 3.16, 3),      # 11,664 atoms: one thread per atom
    ("bcc-l16-s3", "bcc", (5, 5, 5), 3.16, 3),         # 250: warps share atoms
    ("fcc-l20-s4", "fcc", (5, 5, 5), 3.6, 4),          # 500
])
def test_first_call_is_captured(name, lattice, cells, a, species):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_00193_gb300 import build as B
    B.build()
    import paper_2510_00193_gb300 as P
    st = synth.crystal(lattice, cells, a, 0.08, species, 11)
    x = torch.tensor(st.x, device="cuda")
    z = torch.tensor(st.z, dtype=torch.int32, device="cuda")
    warm, fresh = (P.Potential.from_dict(pot_dict(name)) for _ in range(2))
    nl = P.mtp_build_neighbors(warm, x, st.cell, st.pbc)
    ref = P.mtp_compute_efv(warm, nl, x, z, st.cell, precision=P.MTP_FP64)
    out = {k: torch.zeros_like(v) if torch.is_tensor(v) else v for k, v in ref.items()}
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        P.mtp_compute_efv(fresh, nl, x, z, st.cell, precision=P.MTP_FP64, out=out)
    graph.replay()
    torch.cuda.synchronize()
    for k in ("e_atom", "forces", "virial"):
        # the same FP64 sums in another order: a few thousand roundings of 1.1e-16
        assert (out[k] - ref[k]).abs().max() <= 1e-11 * ref[k].abs().max(), k
