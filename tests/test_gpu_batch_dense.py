"""Batches whose reconstructions spread in different forms: dense members on the tensor cores, sparse
ones in bank classes, in one persistent launch each; plans made for more images than they are
given, on both sides of the rule.  Every volume equals the single plan's after 5 damped
iterations (2e-5: the order of FP64 sums and the dither of the ids)."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

ITERS = 5
# (N, images the plan is made for, images of the first run, of the second).  N = 16: both channels on
# the tensor cores from 1,625 images, A*b from 136; N = 32: from 3,225 and 269.
SPECS = [(16, 2500, 2100, 60), (32, 3400, 1000, 3300), (16, 2500, 60, 1700), (32, 3400, 3300, 90), (48, 150, 150, 40)]


@pytest.mark.parametrize("W", [6, 7])
def test_mixed_forms_match_single_plans(W):
    import __graft_entry__ as g
    g.build()
    import paper_1307_5824_gb300 as F
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    probs = []
    for k, (N, cap, _, _) in enumerate(SPECS):
        inp = synth.config_inputs("C2", M=cap, N=N)
        gid = np.random.default_rng(k).integers(0, inp["groups"].shape[0], cap).astype(np.int32)
        probs.append(dict(N=N, groups=inp["groups"], R=dev(inp["R"].reshape(-1, 9)), group=dev(gid),
                          images=dev(inp["images"]), shifts=dev(inp["shifts"])))

    def single(p, M):
        rec = F.Reconstructor(p["N"], M, groups=p["groups"], W=W, lam=1e-2)
        rec.kernel(p["R"], p["group"], M=M)
        rec.backproject(p["images"], p["shifts"], p["R"], p["group"], M=M)
        x = torch.empty((p["N"],) * 3, device="cuda")
        rec.cg_solve(x, ITERS)
        out = x.cpu().numpy().astype(np.float64)
        rec.close()
        return out

    recs = [F.Reconstructor(p["N"], s[1], groups=p["groups"], W=W, lam=1e-2) for p, s in zip(probs, SPECS)]
    xs = [torch.zeros((p["N"],) * 3, device="cuda") for p in probs]
    B = F.BatchReconstructor(recs, n_streams=3)
    for run in (2, 3):
        want = [single(p, s[run]) for p, s in zip(probs, SPECS)]
        B.set_items([dict(M=s[run], R=p["R"], group=p["group"], images=p["images"], shifts=p["shifts"], x=x)
                     for p, s, x in zip(probs, SPECS, xs)])
        for graph, persistent in ((False, False), (False, True), (True, True), (True, True)):
            for x in xs:
                x.zero_()
            B.run(ITERS, graph=graph, persistent=persistent)
            st, sts, _ = B.wait()
            assert st == 0 and (sts == 0).all()
            errs = [float(np.linalg.norm(x.cpu().numpy() - w) / np.linalg.norm(w)) for x, w in zip(xs, want)]
            print(W, run, graph, persistent, ["%.1e" % e for e in errs])
            assert max(errs) <= 2e-5
    B.close()
    for r in recs:
        r.close()
