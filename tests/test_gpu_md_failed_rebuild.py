"""An MD run that stops because its list build fails: the exact list stays the
one of the last completed step, the handle's status word stays clear, and the
run can be taken up again from good positions."""
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


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("steps_before", [0, 3])
def test_list_after_a_failed_rebuild(P, precision, steps_before):
    pot = P.Potential.from_dict(pot_dict("bcc-l16-s3"))
    st = synth.crystal("bcc", (6, 5, 7), 3.16, 0.08, 3, 2)
    masses, dt = [183.84, 95.95, 50.94], 1e-3
    x = torch.tensor(st.x, device="cuda")
    z = torch.tensor(st.z, dtype=torch.int32, device="cuda")
    v = torch.zeros_like(x)
    md = P.MD(pot, x, st.cell, st.pbc, skin=0.4)
    f = P.mtp_compute_efv(pot, md.nlist(), x, z, st.cell, precision=precision)["forces"]
    if steps_before:
        md.run(x, v, z, masses, dt, steps_before, f, rebuild_every=-1, precision=precision)
    rows = [t.clone() for t in md.nlist().to_tensors()]
    good_x, good_v, good_f = x.clone(), v.clone(), f.clone()
    builds = md.rebuilds()
    v[17, 2] = float("nan")
    with pytest.raises(P.MtpError) as e:
        md.run(x, v, z, masses, dt, 2, f, rebuild_every=-1, precision=precision)
    assert e.value.code == -5
    assert all(torch.equal(a, b) for a, b in zip(rows, md.nlist().to_tensors()))
    assert P.mtp_device_status(pot) == 0
    # from the last good state: the flag of the failed step has the list built again
    for t, g in ((x, good_x), (v, good_v), (f, good_f)):
        t.copy_(g)
    md.run(x, v, z, masses, dt, 2, f, rebuild_every=-1, precision=precision)
    assert P.mtp_device_status(pot) == 0
    ref = P.mtp_build_neighbors(pot, x, st.cell, st.pbc)
    assert all(torch.equal(a, b) for a, b in zip(ref.to_tensors(), md.nlist().to_tensors()))
    assert md.rebuilds() == builds + 1


def test_errors_of_checked_steps_are_reported(P):
    """The status of an evaluation queued before the displacement flag is read reaches the handle."""
    pot = P.Potential.from_dict(pot_dict("bcc-l16-s3"))
    st = synth.crystal("bcc", (4, 4, 4), 3.16, 0.08, 3, 2)
    x = torch.tensor(st.x, device="cuda")
    z = torch.tensor(st.z, dtype=torch.int32, device="cuda")
    md = P.MD(pot, x, st.cell, st.pbc, skin=0.4)
    f = P.mtp_compute_efv(pot, md.nlist(), x, z, st.cell)["forces"]
    z[5] = 7   # out of range: read as species 0 and reported
    md.run(x, torch.zeros_like(x), z, [183.84, 95.95, 50.94], 1e-3, 1, f, rebuild_every=-1)
    with pytest.raises(P.MtpError) as e:
        P.mtp_device_status(pot)
    assert e.value.code == -1
    assert P.mtp_device_status(pot) == 0
