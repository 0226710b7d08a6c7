"""The data term in FP64: images and volume scaled by a power of two scale both sums by its square
(exactly so in FP64; 1e-6 for the FP32 transforms of subnormal neighbours), also where that square
leaves FP32's range, and zero images give zero."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("power", [80, -80])
def test_data_term_beyond_the_range_of_fp32(power):
    import __graft_entry__ as g
    g.build()
    import paper_1307_5824_gb300 as F
    N, M = 16, 24
    inp = synth.config_inputs("C2", M=M, N=N)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    rec = F.Reconstructor(N, M, groups=inp["groups"], lam=1e-3)
    R, gid, sh = dev(inp["R"].reshape(M, 9)), dev(inp["group_id"]), dev(inp["shifts"])
    V = np.random.default_rng(3).standard_normal((N, N, N)).astype(np.float32)
    s = np.float32(2.0 ** power)
    res, b2 = rec.data_residual(dev(V), dev(inp["images"]), sh, R, gid)
    got, got_b = rec.data_residual(dev(V * s), dev(inp["images"] * s), sh, R, gid)
    scale = 2.0 ** (2 * power)
    print(f"2^{power}: {got / scale / res - 1:.1e} {got_b / scale / b2 - 1:.1e}")
    assert abs(got / scale - res) <= 1e-6 * res and abs(got_b / scale - b2) <= 1e-6 * b2
    zero = dev(np.zeros_like(inp["images"]))
    assert rec.data_residual(dev(np.zeros_like(V)), zero, sh, R, gid) == (0.0, 0.0)
    rec.close()
