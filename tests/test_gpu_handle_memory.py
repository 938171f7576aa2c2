"""Device memory of the hierarchies a program keeps: what only a setup uses is not theirs."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rsd():
    from paper_1210_6266_gb300 import build
    build.build()
    import paper_1210_6266_gb300 as m
    return m


# 13^3 nodes in 64 leaves: factors, Schur contributions and indices of under 20 MB; the scratch of
# the TF32 leaves' diagonal blocks is 150 MB, the digits of the FP64 fronts' panels 100 MB (LU: 200)
@pytest.mark.parametrize("prec,lu", [("FP64", False), ("FP64", True), ("TF32", False), ("FP16", False)])
def test_kept_hierarchies_hold_no_setup_workspace(rsd, prec, lu):
    n = 13
    prob = rsd.grid_problem(n, 2, np.exp(synth.normal(87, (n - 1) ** 3)), synth.uniform(88, (n - 2) ** 3))
    p = getattr(rsd, "RSD_PREC_" + prec)

    def setup():
        return rsd.RSD.setup(prob["rowptr"], prob["col"], prob["val"], prob["dof_node"], prob["parent"],
                             prec_leaf=p, prec_mid=p, prec_root=p, nonsymmetric=lu)
    hs = [setup()]
    assert hs[0].info()["device_bytes"] <= 40 << 20
    z_ref = hs[0].apply(prob["b"])
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    hs += [setup() for _ in range(4)]
    torch.cuda.synchronize()
    # each: its arena, for TF32 and 16-bit levels the split-K buffers (80 MB), pages of the allocator
    assert free - torch.cuda.mem_get_info()[0] <= 4 * ((40 << 20) + (0 if prec == "FP64" else 84 << 20) + (4 << 20))
    for h in hs:
        assert torch.equal(h.apply(prob["b"]), z_ref)
        h.close()


def test_setups_of_several_threads_at_once(rsd):
    """Each setup has a workspace of its own while it runs, whichever block it got."""
    import threading
    n = 17
    probs = [rsd.grid_problem(n, 2, np.exp(synth.normal(90 + q, (n - 1) ** 3)), synth.uniform(95 + q, (n - 2) ** 3))
             for q in range(3)]
    precs = [rsd.RSD_PREC_FP64, rsd.RSD_PREC_TF32, rsd.RSD_PREC_FP64]

    def one(q):
        p = precs[q]
        h = rsd.RSD.setup(probs[q]["rowptr"], probs[q]["col"], probs[q]["val"], probs[q]["dof_node"], probs[q]["parent"],
                          prec_leaf=p, prec_mid=p, prec_root=p)
        z = h.apply(probs[q]["b"])
        h.check()
        h.close()
        return z
    want = [one(q) for q in range(3)]
    torch.cuda.synchronize()
    bad = []

    def run(q):
        with torch.cuda.stream(torch.cuda.Stream()):
            for _ in range(6):
                z = one(q)
                torch.cuda.current_stream().synchronize()
                if not torch.equal(z, want[q]):
                    bad.append(q)
    ts = [threading.Thread(target=run, args=(q,)) for q in range(3)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert bad == []
