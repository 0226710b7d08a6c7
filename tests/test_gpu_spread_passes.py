"""Tensor-core spreading in several passes (more record slots than one pass holds).  Ker is a sum over
the images, so a large set equals the sum of its parts, each of one pass: 1e-6, two roundings of
each part's FP32 sums (3e-7 against 64 bits, measured bias included).  A*b is A's adjoint, so
<A*b, A*b> = <b, A A*b>: 2e-5, the windows' errors (6e-6 each at W = 6).  A pass left out is half of either."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


N, M = 32, 200000                                       # 8e7 points


def dense_set():
    gen = torch.Generator(device="cuda").manual_seed(4)
    q = torch.randn((M, 4), generator=gen, device="cuda", dtype=torch.float64)
    w, x, y, z = (q / q.norm(dim=1, keepdim=True)).T
    R = torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - z * w), 2 * (x * z + y * w), 2 * (x * y + z * w),
                     1 - 2 * (x * x + z * z), 2 * (y * z - x * w), 2 * (x * z - y * w), 2 * (y * z + x * w),
                     1 - 2 * (x * x + y * y)], dim=1).contiguous()
    images = torch.randn((M, N, N), generator=gen, device="cuda")
    shifts = torch.rand((M, 2), generator=gen, device="cuda", dtype=torch.float64)
    return R, images, shifts


@pytest.mark.parametrize("W,fused", [(6, False), (6, True), (7, False)])
def test_passes_cover_a_large_set(W, fused):
    import __graft_entry__ as g
    g.build()
    import paper_1307_5824_gb300 as F
    R, images, shifts = dense_set()
    rec = F.Reconstructor(N, M, W=W, lam=1e-3, fused=fused)

    def sums(a, b):
        ker, rhs = torch.empty(rec.half_shape(), device="cuda"), torch.empty((N, N, N), device="cuda")
        if fused:
            rec.kernel_backproject(images[a:b], shifts[a:b], R[a:b], None, M=b - a, rhs_out=rhs)
        else:
            rec.kernel(R[a:b], M=b - a)
            rec.backproject(images[a:b], shifts[a:b], R[a:b], None, M=b - a, rhs_out=rhs)
        rec.copy_out(F._lib.FIRM_OUT_KER, ker)
        rec.lambda_eff()                                # waits, and reports the device's flag
        return ker.double(), rhs.double()

    cuts = [0, 66000, 131000, M]
    part = sum(sums(a, b)[0] for a, b in zip(cuts, cuts[1:]))
    ker, rhs = sums(0, M)
    err = float((ker - part).norm() / part.norm())
    b = torch.empty((M, (F._lib.disc_size(N) + 1) // 2, 2), device="cuda")
    rec.copy_out(F._lib.FIRM_OUT_SAMPLES, b)            # the origin's halved: every other one stands for two
    AV = rec.forward(rhs.float(), R)
    dot = 2.0 * sum(float((x.double() * y.double()).sum()) for x, y in zip(b.split(20000), AV.split(20000)))
    adj = dot / float((rhs * rhs).sum()) - 1.0
    print(f"W={W} fused={fused}: Ker {err:.2e} adjoint {adj:.2e}")
    assert err <= 1e-6 and abs(adj) <= 2e-5
    rec.close()


def test_several_passes_in_a_batch():
    """A reconstruction of several passes among ones of one pass and of bank classes: each volume equals
    the single plan's after 5 damped iterations (2e-5: the order of FP64 sums and the ids' dither)."""
    import __graft_entry__ as g
    g.build()
    import paper_1307_5824_gb300 as F
    R, images, shifts = dense_set()
    Ms = [M, 4000, 100]
    recs = [F.Reconstructor(N, m, lam=1e-2) for m in Ms]
    xs = [torch.zeros((N, N, N), device="cuda") for _ in Ms]
    want = []
    for rec, m in zip(recs, Ms):
        rec.kernel(R, M=m)
        rec.backproject(images, shifts, R, None, M=m)
        x = torch.empty((N, N, N), device="cuda")
        rec.cg_solve(x, 5)
        want.append(x.double())
    B = F.BatchReconstructor(recs, n_streams=2)
    B.set_items([dict(M=m, R=R, group=None, images=images, shifts=shifts, x=x) for m, x in zip(Ms, xs)])
    for graph in (False, True, True):
        for x in xs:
            x.zero_()
        B.run(5, graph=graph, persistent=True)
        st, sts, _ = B.wait()
        assert st == 0 and (sts == 0).all()
        errs = [float((x.double() - w).norm() / w.norm()) for x, w in zip(xs, want)]
        print(graph, ["%.1e" % e for e in errs])
        assert max(errs) <= 2e-5
    B.close()
    for rec in recs:
        rec.close()
