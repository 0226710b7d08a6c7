"""The tensor-core spreading's share of a plan's workspace: its records are made in passes of bounded
size, so what grows with the images is the placed points only (at most 9 bytes a point more than
the ids of the bank-class form, which alone W = 8 plans have)."""
import pytest

GIB = 1 << 30


@pytest.mark.parametrize("flags", [0, 2])
@pytest.mark.parametrize("M", [14000, 50000, 334000])
def test_workspace_stays_near_the_bank_class_form(M, flags):
    import __graft_entry__ as g
    g.build()
    from paper_1307_5824_gb300 import _lib as L
    size = lambda W: L.firm_workspace_size(L.make_params(128, M, 20, W, img_dtype=L.FIRM_IMG_BF16, flags=flags))
    points = M * 6434                                   # half disc at N = 128
    assert size(6) - size(8) <= 9 * points + 1.6 * GIB
    assert size(7) - size(8) <= 9 * points + 1.6 * GIB
