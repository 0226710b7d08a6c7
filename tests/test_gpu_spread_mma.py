"""The tensor-core spreading (dense bricks, W = 6 and 7) against the FP64 gridding oracle with the
same Kaiser-Bessel window (eq. kernel, eq. backprojection), which leaves the arithmetic's
own error: the sizes run from just above the rule's threshold, where most classes of a
brick hold less than one group of points, to bricks of several work items.

Tolerance 3e-6: taps and weights carry 22 bits and the window polynomials 2e-7; a cell's
sum over at most 4096 points is rounded to 2^-18 of the largest weight about ten times,
which is 1e-6 of a cell's sum of weights of rms a third of the largest."""
import numpy as np
import pytest

import oracle as O
from oracle import gridding as GR
import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


@pytest.mark.parametrize("N,M,cfg,fused,W", [
    (16, 141, "C2", False, 6), (16, 1641, "C5", False, 6), (16, 6001, "C3", False, 6), (32, 3301, "C5", False, 6),
    (16, 641, "C3", True, 6), (16, 2003, "C5", True, 6), (32, 1301, "C2", True, 6),
    (16, 1641, "C5", False, 7), (16, 6001, "C3", False, 7), (32, 1001, "C2", False, 7)])
def test_tensor_core_spreading_matches_oracle(N, M, cfg, fused, W):
    import __graft_entry__ as g
    g.build()
    import paper_1307_5824_gb300 as F
    inp = synth.config_inputs(cfg, M=M, N=N)
    K = O.disc(N)
    kw = dict(W=W, window="kb", beta=GR.kb_beta(W))
    Ker = GR.kernel_gridded(inp["R"], inp["groups"], inp["group_id"], K, N, **kw).real
    rhs_o = GR.backproject_gridded(inp["images"], inp["shifts"], inp["R"], inp["groups"], inp["group_id"], K,
                                   sigma=4 if fused else 2, **kw)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    rec = F.Reconstructor(N, M, groups=inp["groups"], W=W, lam=1e-3, fused=fused)
    R, gid = dev(inp["R"].reshape(M, 9)), dev(inp["group_id"])
    ker = torch.empty(rec.half_shape(), device="cuda")
    rhs = torch.empty((N, N, N), device="cuda")
    if fused:
        rec.kernel_backproject(dev(inp["images"]), dev(inp["shifts"]), R, gid, rhs_out=rhs)
    else:
        rec.kernel(R, gid)
        rec.backproject(dev(inp["images"]), dev(inp["shifts"]), R, gid, rhs_out=rhs)
    rec.copy_out(F._lib.FIRM_OUT_KER, ker)
    assert rec.lambda_eff() > 0.0                    # waits for the stream and the device's error flag
    e_k = rel(ker.cpu().numpy()[1:, 1:, :N], Ker[1:, 1:, N:])
    e_r = rel(rhs.cpu().numpy(), rhs_o)
    print(f"N={N} M={M} {cfg} W={W} fused={fused}: Ker {e_k:.2e} A*b {e_r:.2e}")
    assert e_k <= 3e-6 and e_r <= 3e-6
    rec.close()


@pytest.mark.parametrize("N,scale", [(16, 2.8), (48, 2.5), (64, 1.5), (80, 1.5), (96, 1.3)])
def test_scaled_matrices_wrap_the_grid(N, scale):
    """Matrices longer than a rotation put samples past the grid's edge, where they wrap:
    Ker against its direct sum at 300 lags.  KB W = 6 is within 2e-5 of the sum of |weights|
    there; a lag's own sum is at least a tenth of their root mean square, so 1e-3 of the
    lags' norm, against 1 for samples in wrong cells."""
    import __graft_entry__ as g
    g.build()
    import paper_1307_5824_gb300 as F
    inp = synth.config_inputs("C2", M=5, N=N)
    K = O.disc(N)
    Rs = inp["R"] * scale
    rng = np.random.default_rng(N)
    lags = rng.integers([0, -N + 1, -N + 1], N, size=(300, 3))
    h = O.ctf_weights(N, K, inp["groups"], inp["group_id"])
    want = O.kernel_at(Rs, h, K, N, lags).real
    rec = F.Reconstructor(N, 5, groups=inp["groups"], lam=1e-3)
    rec.kernel(torch.from_numpy(Rs.reshape(5, 9)).cuda(), torch.from_numpy(inp["group_id"]).cuda())
    ker = torch.empty(rec.half_shape(), device="cuda")
    rec.copy_out(F._lib.FIRM_OUT_KER, ker)
    got = ker.cpu().numpy()[lags[:, 2] + N, lags[:, 1] + N, lags[:, 0]]
    print(f"N={N} x{scale}: {rel(got, want):.2e}")
    assert rel(got, want) <= 1e-3
    rec.close()
