"""Tensor-core spreading without a bias.  The tensor core's FP32 additions truncate, so a group of
16 points goes through at most three of them (each at most 2^-24 of the sum short, 1.8e-7
together) before a rounded add: Ker and A*b may be 3e-7 of their value too small or large, measured
as the part of the error along the oracle's sums with the same window (sums of 128 points
through the tensor core come out 5e-7 to 7e-7 too small)."""
import numpy as np
import pytest

import oracle as O
from oracle import gridding as GR
import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.fixture(scope="module")
def F():
    import __graft_entry__ as g
    g.build()
    import paper_1307_5824_gb300 as F
    return F


@pytest.mark.parametrize("N,M,cfg,W", [(16, 6001, "C3", 6), (32, 3301, "C5", 6), (16, 1641, "C5", 7), (16, 6001, "C3", 7)])
def test_sums_are_not_biased(F, N, M, cfg, W):
    inp = synth.config_inputs(cfg, M=M, N=N)
    K = O.disc(N)
    kw = dict(W=W, window="kb", beta=GR.kb_beta(W))
    Ker = GR.kernel_gridded(inp["R"], inp["groups"], inp["group_id"], K, N, **kw).real[1:, 1:, N:]
    rhs_o = GR.backproject_gridded(inp["images"], inp["shifts"], inp["R"], inp["groups"], inp["group_id"], K, sigma=2, **kw)
    rec = F.Reconstructor(N, M, groups=inp["groups"], W=W, lam=1e-3)
    R, gid = dev(inp["R"].reshape(M, 9)), dev(inp["group_id"])
    ker, rhs = torch.empty(rec.half_shape(), device="cuda"), torch.empty((N, N, N), device="cuda")
    rec.kernel(R, gid)
    rec.backproject(dev(inp["images"]), dev(inp["shifts"]), R, gid, rhs_out=rhs)
    rec.copy_out(F._lib.FIRM_OUT_KER, ker)
    for name, got, want in (("Ker", ker.cpu().numpy()[1:, 1:, :N], Ker), ("A*b", rhs.cpu().numpy(), rhs_o)):
        along = float(((got - want) * want).sum() / (want * want).sum())
        print(f"N={N} M={M} {cfg} W={W} {name}: {along:.2e}")
        assert abs(along) <= 3e-7
    rec.close()


@pytest.mark.parametrize("W", [6, 7])
def test_undamped_volume_of_a_dense_set(F, W):
    """300 noiseless Haar views at N = 32, lambda = 0, 10 iterations: A*b in the tensor-core form
    (447 points a brick).  The FP64 CG mode shows what Ker and A*b alone do to the volume;
    1e-4 is the volume target."""
    inp = synth.config_inputs("C1", M=300)
    N, M = inp["N"], inp["M"]
    K = O.disc(N)
    h = np.ones((M, K.shape[0]))
    Ker = O.kernel(inp["R"], h, K, N).real
    b = O.backproject(inp["images"].astype(np.float64), inp["shifts"], inp["R"], h, K)
    want, _, _ = O.cg(lambda v: O.toeplitz_apply(O.khat(Ker), v).real, b, 10)
    rec = F.Reconstructor(N, M, W=W, lam=0.0, flags=F._lib.FIRM_FLAG_FP64_CG)
    R = dev(inp["R"].reshape(M, 9))
    rec.kernel(R)
    rec.backproject(dev(inp["images"].astype(np.float32)), dev(inp["shifts"]), R)
    x = torch.empty((N, N, N), device="cuda")
    rec.cg_solve(x, 10)
    err = float(np.linalg.norm(x.cpu().numpy() - want) / np.linalg.norm(want))
    print(f"W={W}: {err:.2e}")
    assert err <= 1e-4
    rec.close()
