"""The size up to which the plain 3+1D form keeps pair lists: as many entries as a quarter of the free
device memory holds at 40 bytes each.  (The memory is reserved, not touched: the event is small.)"""
import pytest

from paper_2511_22852_gb300 import binding as Bd
from paper_2511_22852_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bytes_each,lists", [(45, True), (42, True), (40.5, True), (39.5, False)])
def test_lists_up_to_a_quarter_at_40_bytes_an_entry(bytes_each, lists, monkeypatch):
    torch = pytest.importorskip("torch")
    g = Bd.GpuEvent(I.smooth_blob_3d(half_widths=(0.5, 0.5, 0.4), with_table=False))
    free = torch.cuda.mem_get_info()[0]
    total = int(free / 4 / bytes_each)
    monkeypatch.setenv("SPH_PAIR_TOTAL", str(total))
    g.step(1, sync=True)
    taken = free - torch.cuda.mem_get_info()[0]
    g.free()
    assert (taken > 36 * total) == lists
