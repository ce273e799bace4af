"""A handle's kernel shape variant decides the row grouping of the reference tables of its own evolve alone: the
general batch kernel and the general adjoint kernel read two-row groups whatever variant their handles have set."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import mtp_synth as S
import paper_1906_11029_gb300 as mtp
from _oracle_bridge import rel_l2

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _random_state(mesh, seed):
    return torch.randn(mesh.state_shape, generator=torch.Generator().manual_seed(seed), dtype=torch.float64).to(DEV, mesh.torch_dtype())


@pytest.mark.parametrize("degrees,variants", [((5, 3), (2, 0)), ((5, 3), (0, 4)), ((5, 2), (2, 2))])
def test_batch_with_p5_ignores_variants(degrees, variants):
    """p = 5 has 35 rows in the first factor of the volume term, p = 3 has 10 and p = 2 has 4; odd counts group differently."""
    v, e = S.cube_mesh(1)
    one = np.ones(len(e))
    tents, states, want = [], [], []
    for i, (p, variant) in enumerate(zip(degrees, variants)):
        mesh = mtp.Mesh(3, v, e, one, one, p=p, precision=mtp.MTP_FP32)
        t = mesh.pitch(0.05, 0.5)
        states.append(_random_state(mesh, i))
        want.append(states[-1].clone())
        t.evolve(want[-1])
        t.set_variant(variant)
        tents.append(t)
    mtp.Batch(tents).evolve(states)
    for got, ref in zip(states, want):
        assert rel_l2(got.cpu().numpy(), ref.cpu().numpy()) <= 1e-5


@pytest.mark.parametrize("p", [1, 2, 3, 4, 5])
def test_gradient_ignores_variants(p):
    """2D FP32: the same gradients with every variant (the forward kernels differ in rounding only)."""
    v, e = S.square_mesh(2)
    one = np.ones(len(e))
    mesh = mtp.Mesh(2, v, e, one, one, p=p, precision=mtp.MTP_FP32)
    t = mesh.pitch(0.1, 0.5)
    Y, lam = _random_state(mesh, 1), _random_state(mesh, 2)
    out = []
    for variant in (0, 1, 2):
        t.set_variant(variant)
        l0, ge, gm = torch.empty_like(Y), *(torch.empty(len(e), dtype=torch.float64, device=DEV) for _ in range(2))
        mtp.mtp_adjoint(t.h, Y, lam, l0, ge, gm, 0)
        out.append([x.cpu().numpy() for x in (l0, ge, gm)])
    for got in out[1:]:
        assert all(rel_l2(g, r) <= 1e-5 for g, r in zip(got, out[0]))
