"""Setups without room for all of the factorisation's workspace (rsd_inject_workspace_limit):
FP64 fronts on the FP64 pipe at the tolerances of the tensor-core form, in smaller groups
with the same results, and TF32 / FP16 levels with scratch of their own."""
import numpy as np
import pytest

import synth
import test_gpu_fp64_fronts as fronts

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rsd():
    from paper_1210_6266_gb300 import build
    build.build()
    import paper_1210_6266_gb300 as m
    return m


class _Limited:
    """The package with every RSD.setup under a workspace limit."""
    def __init__(self, rsd, limit):
        from paper_1210_6266_gb300 import _lib

        class RSD(rsd.RSD):
            @classmethod
            def setup(cls, *a, **kw):
                assert _lib.load().rsd_inject_workspace_limit(limit) == 0
                return super().setup(*a, **kw)
        self._rsd, self.RSD = rsd, RSD

    def __getattr__(self, name):
        return getattr(self._rsd, name)


@pytest.mark.parametrize("count,edge,s_root", [(1, 1, 3), (2, 128, 31), (3, 130, 200), (1, 1030, 140), (80, 131, 33)])
def test_fp64_pipe_factor_of_arrow_fronts(rsd, count, edge, s_root):
    fronts.test_fp64_factor_of_arrow_fronts(_Limited(rsd, 0), count, edge, s_root)


@pytest.mark.parametrize("count,edge,s_root", [(1, 1, 3), (2, 128, 31), (3, 130, 200), (1, 1030, 140)])
def test_fp64_pipe_lu_of_arrow_fronts(rsd, count, edge, s_root):
    fronts.test_fp64_lu_of_arrow_fronts(_Limited(rsd, 0), count, edge, s_root)


# 64 leaves of up to 125 rows + couplings: about 1.7 MB of digits each (3.4 MB for LU), the root's
# front over 1000 rows 11 MB (22)
@pytest.mark.parametrize("prec,lu,limit,simt", [("FP64", False, 0, True), ("FP64", False, 24 << 20, False),
                                                ("FP64", True, 48 << 20, False), ("TF32", False, 0, False),
                                                ("FP16", False, 0, False)])
def test_limited_workspace_gives_the_same_application(rsd, prec, lu, limit, simt):
    n = 21
    prob = rsd.grid_problem(n, 2, np.exp(synth.normal(97, (n - 1) ** 3)), synth.uniform(98, (n - 2) ** 3))
    p = getattr(rsd, "RSD_PREC_" + prec)

    def apply(m):
        h = m.RSD.setup(prob["rowptr"], prob["col"], prob["val"], prob["dof_node"], prob["parent"], profile=True,
                        prec_leaf=p, prec_mid=p, prec_root=p, nonsymmetric=lu)
        used = h.profile()["gemm_simt"]["launches"] > 0
        z = h.apply(prob["b"])
        h.close()
        return z, used
    want, _ = apply(rsd)
    got, used = apply(_Limited(rsd, limit))
    assert used == simt
    if simt:
        assert float((got - want).abs().max()) <= 1e-12 * float(want.abs().max())
    else:
        assert torch.equal(got, want)
