"""Matrices beyond rotations: columns (R_1d, R_2d) of length below 3 put samples past the grid's
edge, where they wrap; longer or NaN ones are reported and leave the plan usable."""
import numpy as np
import pytest

import oracle as O
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


@pytest.mark.parametrize("N", [16, 32, 48, 64, 80, 96, 128])
def test_matrices_below_the_limit_wrap_the_grid(F, N):
    """Ker against its direct sum at 300 lags, the scaled columns at most 2.95 long.  KB W = 6
    is within 2e-5 of the sum of |weights| there; a lag's own sum is at least a tenth of
    their root mean square, so 1e-3 of the lags' norm, against 1 for samples in wrong cells."""
    inp = synth.config_inputs("C2", M=5, N=N)
    K = O.disc(N)
    Rs = inp["R"] * 2.95 / np.sqrt((inp["R"][:, :2] ** 2).sum(1)).max()
    rng = np.random.default_rng(N)
    lags = rng.integers([0, -N + 1, -N + 1], N, size=(300, 3))
    h = O.ctf_weights(N, K, inp["groups"], inp["group_id"])
    want = O.kernel_at(Rs, h, K, N, lags).real
    rec = F.Reconstructor(N, 5, groups=inp["groups"], lam=1e-3)
    rec.kernel(dev(Rs.reshape(5, 9)), dev(inp["group_id"]))
    ker = torch.empty(rec.half_shape(), device="cuda")
    rec.copy_out(F._lib.FIRM_OUT_KER, ker)
    got = ker.cpu().numpy()[lags[:, 2] + N, lags[:, 1] + N, lags[:, 0]]
    err = float(np.linalg.norm(got - want) / np.linalg.norm(want))
    print(f"N={N}: {err:.2e}")
    assert err <= 1e-3
    rec.close()


@pytest.mark.parametrize("bad", [3.01, np.nan, np.inf])
def test_matrices_beyond_the_limit_are_reported(F, bad):
    N, M = 16, 7
    inp = synth.config_inputs("C2", M=M, N=N)
    rec = F.Reconstructor(N, M, groups=inp["groups"], lam=1e-3)
    R, gid = inp["R"].reshape(M, 9).copy(), dev(inp["group_id"])
    rec.kernel(dev(R), gid)
    good = rec.lambda_eff()
    R[3, 0] = bad
    rec.kernel(dev(R), gid)
    with pytest.raises(F._lib.FirmError) as e:
        rec.lambda_eff()
    assert e.value.code == F._lib.FIRM_EINVAL
    rec.kernel(dev(inp["R"].reshape(M, 9)), gid)
    assert rec.lambda_eff() == pytest.approx(good, rel=1e-5)
    rec.close()
