"""Results that no other path in the library repeats, pinned bit for bit: the costs and
controls of split-precision steps of up to 512 points, whose sums have an order of their
own (a cluster of CTAs once held the factor: every 64-column slice its stages in the
order of that CTA), and Step 2's covariance.  The words in golden/former_bits.txt are
those rollouts' on this GPU, before the rollout went query by query."""
import os

import numpy as np
import pytest

import scenarios as S
from parity import make_ctrl

pytestmark = pytest.mark.gpu

GOLDEN = os.path.join(os.path.dirname(__file__), "golden", "former_bits.txt")

# each side of the slices' and the shares' edges
SIZES = [1, 64, 65, 128, 129, 192, 193, 256, 257, 320, 321, 384, 385, 448, 449, 512]
CASES = [(f"step-N{N}-p{p}", dict(N=N, precision=p)) for N in SIZES for p in (1, 2)]
CASES += [(f"nominal-N{N}", dict(N=N, precision=0, variance_mode=1)) for N in (1, 45, 300, 700)]


def words(lib, name, kw):
    """The words of two steps' controls and costs, and of the carried covariance."""
    import torch
    sc = S.scenario("small", K=40, T=6, O=5, **kw)
    _, ctrl = make_ctrl(lib, sc)
    U = torch.tensor(sc.U0, dtype=torch.float32, device="cuda")
    out = []
    for it in (3, 4):
        lib.mppi_set_iteration(ctrl, it)
        Un, w, c = torch.empty_like(U), torch.empty(40, device="cuda"), torch.empty(40, device="cuda")
        lib.mppi_step(ctrl, sc.x0.astype(np.float32), U, Un, w, c)
        out += [Un, c]
        if sc.params.variance_mode:
            out.append(torch.empty(6, 3, device="cuda"))
            lib.mppi_nominal_sxy(ctrl, out[-1])
        U = Un
    return np.concatenate([x.cpu().numpy().ravel().view(np.uint32) for x in out])


@pytest.mark.parametrize("name,kw", CASES, ids=[c[0] for c in CASES])
def test_former_bits(lib, name, kw):
    want = dict(line.split(" ", 1) for line in open(GOLDEN) if line.strip())[name]
    assert " ".join("%08x" % w for w in words(lib, name, kw)) == want.strip()
