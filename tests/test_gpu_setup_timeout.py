"""Waits of the factorisation's tensor-core GEMMs that give up (rsd_inject_setup_timeout):
the kernels finish, rsd_setup returns RSD_ERR_TIMEOUT and no handle, and the CUDA context
stays usable."""
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


# FP64: the digit products; TF32: single-tile and persistent GEMMs; FP16: persistent, 16-bit operands
@pytest.mark.parametrize("prec,n,depth,lu", [("FP64", 17, 2, False), ("FP64", 17, 1, True), ("TF32", 25, 1, False),
                                             ("FP16", 25, 1, False)])
def test_waits_of_the_factorisation_that_give_up(rsd, prec, n, depth, lu):
    from paper_1210_6266_gb300 import _lib
    lib = _lib.load()
    prob = rsd.grid_problem(n, depth, np.exp(synth.normal(85, (n - 1) ** 3)), synth.uniform(86, (n - 2) ** 3))
    p = getattr(rsd, "RSD_PREC_" + prec)

    def setup():
        return rsd.RSD.setup(prob["rowptr"], prob["col"], prob["val"], prob["dof_node"], prob["parent"],
                             prec_leaf=p, prec_mid=p, prec_root=p, nonsymmetric=lu)
    h = setup()
    z_ref = h.apply(prob["b"]).clone()
    h.close()
    assert lib.rsd_inject_setup_timeout() == 0
    with pytest.raises(rsd.RSDError) as e:
        setup()
    assert e.value.code == _lib.RSD_ERR_TIMEOUT
    torch.cuda.synchronize()                               # the kernels finished
    h = setup()
    assert torch.equal(h.apply(prob["b"]), z_ref)
    h.check()
    h.close()
