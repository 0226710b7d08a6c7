"""A*b of images far from unit size in the tensor-core spreading, alone and with Ker in one pass."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

DENSE = [(1641, False), (2003, True)]


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.fixture(scope="module")
def F():
    import __graft_entry__ as g
    g.build()
    import paper_1307_5824_gb300 as F
    return F


def setup(F, M, fused, N=16):
    inp = synth.config_inputs("C5", M=M, N=N)
    rec = F.Reconstructor(N, M, groups=inp["groups"], lam=1e-3, fused=fused)
    R, gid, shifts = dev(inp["R"].reshape(M, 9)), dev(inp["group_id"]), dev(inp["shifts"])

    def rhs(images):
        out = torch.empty((N, N, N), device="cuda")
        if fused:
            rec.kernel_backproject(dev(images), shifts, R, gid, rhs_out=out)
        else:
            rec.kernel(R, gid)
            rec.backproject(dev(images), shifts, R, gid, rhs_out=out)
        rec.lambda_eff()                             # waits, and reports the device's flag
        return out.cpu().numpy().astype(np.float64)

    return rec, inp["images"].astype(np.float32), rhs


@pytest.mark.parametrize("M,fused", DENSE)
def test_small_images_scale(F, M, fused):
    """Images scaled by a power of two so that the largest |h b| is near 2^-104: the fixed-point
    units follow it, so A*b is the unscaled one times that power to the rounding of the FP32
    transforms (1e-6)."""
    rec, images, rhs = setup(F, M, fused)
    top = np.abs(np.fft.fft2(images.astype(np.float64))).max()
    scale = 2.0 ** (-104 - int(np.ceil(np.log2(top))))
    want = rhs(images)
    got = rhs((images * np.float32(scale)).astype(np.float32)) / scale
    err = float(np.linalg.norm(got - want) / np.linalg.norm(want))
    print(f"M={M} fused={fused}: {err:.2e}")
    assert err <= 1e-6
    rec.close()


@pytest.mark.parametrize("M,fused", DENSE)
@pytest.mark.parametrize("value", [np.nan, np.inf])
def test_non_finite_images_are_reported(F, M, fused, value):
    """One bad pixel spoils the sums of every class of cells its image crosses: reported by the
    next call that waits, and the plan takes the next images."""
    rec, images, rhs = setup(F, M, fused)
    want = rhs(images)
    bad = images.copy()
    bad[M // 2, 3, 5] = value
    with pytest.raises(F._lib.FirmError) as e:
        rhs(bad)
    assert e.value.code == F._lib.FIRM_EINVAL
    got = rhs(images)
    assert np.linalg.norm(got - want) <= 1e-6 * np.linalg.norm(want)
    rec.close()


@pytest.mark.parametrize("M,fused", DENSE)
def test_host_images(F, M, fused):
    """Host images, copied in stream order into the memory the points take afterwards, and staged
    ahead, against the same images on the device (1e-6: the order of the sums)."""
    N = 16
    inp = synth.config_inputs("C5", M=M, N=N)
    rec = F.Reconstructor(N, M, groups=inp["groups"], lam=1e-3, fused=fused)
    R, gid, shifts = dev(inp["R"].reshape(M, 9)), dev(inp["group_id"]), dev(inp["shifts"])
    host = torch.from_numpy(inp["images"].astype(np.float32)).pin_memory()
    got = []
    for images, stage in ((host.cuda(), False), (host, False), (host, True)):
        out = torch.empty((N, N, N), device="cuda")
        if stage:
            rec.stage_images(images)
        if fused:
            rec.kernel_backproject(images, shifts, R, gid, rhs_out=out)
        else:
            rec.kernel(R, gid)
            rec.backproject(images, shifts, R, gid, rhs_out=out)
        rec.lambda_eff()
        got.append(out.cpu().numpy().astype(np.float64))
    for other in got[1:]:
        assert np.linalg.norm(other - got[0]) <= 1e-6 * np.linalg.norm(got[0])
    rec.close()
