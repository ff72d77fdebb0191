"""Device memory of FP64 plans under a cap on the intermediates.  A cap cuts sigma into
chunks with plans of their own, whose partial sums share one buffer: at L = 24, D = 512 the
intermediates fill their default gigabyte, and a cap of 256 or 64 MB gives back at least
half of it (with a buffer for each of the 184 and 778 plans it gave back 96 and 320 MB)."""
import gc

import pytest
import torch

from paper_2501_18263_gb300 import binding as B
from paper_2501_18263_gb300 import inputs as I
from gpu_util import rel, stream, to_dev

pytestmark = pytest.mark.gpu


def test_a_cap_on_intermediates_saves_memory():
    L, na, nb, D, bond = 24, 12, 12, 512, 11
    t, v = I.synthetic_integrals(L, 3)
    bp = I.bond_problem(L, na, nb, D, bond, seed=4)
    psi = to_dev(B.pack_psi(bp.psi))
    out, used = [], []
    for cap in (0, 256 << 20, 64 << 20):
        gc.collect()
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        free = torch.cuda.mem_get_info()[0]
        d = B.Dmrg(t, v, na, nb, D=D, mem_cap=cap, stream=stream())
        d.load_bond_problem(bp)
        d.prepare(bond)
        x = torch.empty_like(psi)
        d.sigma(bond, psi.data_ptr(), x.data_ptr())
        torch.cuda.synchronize()
        used.append(free - torch.cuda.mem_get_info()[0])
        out.append(x.cpu().numpy())
        d.close()
        assert rel(out[-1], out[0]) < 1e-13
    assert max(used[1:]) <= used[0] - (512 << 20), used
