"""Paper mode with gamma inner iterations on levels of many interfaces, where the inner
GMRES takes fewer CTAs per interface (two from 77 interfaces on, one from 153 on), against
the oracle's recursive Algorithm 2."""
import numpy as np
import pytest

import synth
from oracle import fem2d, partition
from oracle.rsd_paper import PaperRSD

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,P,gamma", [(7, 256, 3), (5, 512, 2)])
def test_gamma_apply_with_many_interfaces_on_a_level(N, P, gamma):
    from paper_1210_6266_gb300 import build
    build.build()
    import paper_1210_6266_gb300 as rsd
    A, coords = fem2d.strip_poisson(N, P)
    owner = fem2d.binary_owner(N, P, coords)
    parent = fem2d.binary_parent(int(np.log2(P)))
    R = PaperRSD(A, partition.Symbolic(A, owner, parent), gamma)
    h = rsd.RSD.setup(torch.as_tensor(A.indptr.astype(np.int64)), torch.as_tensor(A.indices.astype(np.int32)),
                      torch.as_tensor(A.data.astype(np.float64)), torch.as_tensor(owner.astype(np.int32)), parent,
                      prec_leaf=rsd.RSD_PREC_FP64, prec_mid=rsd.RSD_PREC_FP64, prec_root=rsd.RSD_PREC_FP64,
                      mode=rsd.RSD_MODE_PAPER, gamma=gamma)
    for seed in (97, 98):
        r = synth.uniform(seed, A.shape[0])
        z = h.apply(torch.as_tensor(r, device="cuda")).cpu().numpy()
        zr = R.apply_recursive(r)
        # the bound of the same comparison on the octree levels
        assert np.abs(z - zr).max() <= 1e-10 * np.abs(zr).max(), (seed, np.abs(z - zr).max() / np.abs(zr).max())
    h.check()
    h.close()
