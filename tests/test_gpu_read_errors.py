"""sph_read_fields with a requested field that has no destination: an argument error, with the fields
before it complete and no copy in flight."""
import ctypes as C

import numpy as np
import pytest

from paper_2511_22852_gb300 import binding as Bd
from paper_2511_22852_gb300 import inputs as I

pytestmark = pytest.mark.gpu

# name, attribute, rows, of the fields before the missing one
CASES = [("SIGMA_STAR", [("S", "S", 1), ("U", "u", 2)]), ("STATUS", [("S", "S", 1), ("T", "T", 1), ("PI_BULK", "Pi", 1)]),
         ("CELL", [("X", "x", 2), ("MU", "mu", 3), ("PI_BULK", "Pi", 1), ("NNB", "nnb", 1)])]


@pytest.mark.parametrize("missing,given", CASES)
@pytest.mark.parametrize("device", [False, True])
def test_fields_before_a_missing_destination_are_complete(missing, given, device):
    torch = pytest.importorskip("torch")
    g = Bd.GpuEvent(I.viscous_bsq_2p1(n_target=3000, R=3.0, n_hot=20))
    want = g.read([k for k, _, _ in given])
    bufs, mask, keep = Bd.FieldBufs(), Bd.F[missing], {}
    bufs.on_device = int(device)
    for name, attr, rows in given:
        t = torch.full((rows, g.n), -7, dtype=torch.int32 if name == "NNB" else torch.float64, device="cuda" if device else "cpu")
        keep[name] = t
        setattr(bufs, attr, t.data_ptr())
        mask |= Bd.F[name]
    if device:
        torch.cuda.synchronize()
    rc = Bd.lib().sph_read_fields(g.h, C.c_uint64(mask), C.byref(bufs), None)
    assert rc == Bd.SPH_ERR_ARG
    assert "null destination" in Bd.lib().sph_last_error().decode()
    for name, t in keep.items():
        assert np.array_equal(t.cpu().numpy().reshape(np.asarray(want[name]).shape), want[name]), name
    g.free()
