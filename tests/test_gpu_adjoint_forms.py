"""Gradients in the forms of the adjoint kernel that need small patches (FP64 at p = 3, FP32 at p = 4 in 3D), and with
several right-hand sides."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import mtp_synth as S
import paper_1906_11029_gb300 as mtp

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _gradients(mesh, tents, Y, lam, every):
    l0 = torch.empty_like(Y)
    ge, gm = (torch.empty(mesh.info["n_elems"], dtype=torch.float64, device=DEV) for _ in range(2))
    mtp.mtp_adjoint(tents.h, Y, lam, l0, ge, gm, every)
    return l0, ge, gm


@pytest.mark.parametrize("name", ["one_tet", "cube1"])
@pytest.mark.parametrize("prec,p,tol", [(mtp.MTP_FP64, 3, 1e-8), (mtp.MTP_FP32, 4, 1e-5), (mtp.MTP_FP32, 3, 1e-5)])
def test_small_patch_gradients_match_directional_differences(name, prec, p, tol):
    """Along one direction each in the initial state, eps and mu, against central differences of FP64 evolves (h = 1e-6:
    about 1e-9 of rounding and h^2 of truncation; FP32 gradients to the 1e-5 of that mode)."""
    v, e = S.cube_mesh(1)
    v = v + 0.1 * np.random.default_rng(5).uniform(-1, 1, v.shape)
    e = e[:1] if name == "one_tet" else e
    if name == "one_tet":
        used = np.unique(e)
        v, e = v[used], np.searchsorted(used, e).astype(np.int32)
    rng = np.random.default_rng(p)
    eps, mu = rng.uniform(1, 2, len(e)), rng.uniform(1, 2, len(e))
    ws, T = np.ones(len(e)), 0.05
    ref = mtp.Mesh(3, v, e, eps, mu, p=p)
    Y0, dY = (torch.tensor(rng.standard_normal(ref.state_shape), device=DEV) for _ in range(2))
    de, dm = rng.standard_normal(len(e)), rng.standard_normal(len(e))

    def J(h, which):
        m = mtp.Mesh(3, v, e, eps + (h * de if which == 1 else 0), mu + (h * dm if which == 2 else 0), p=p)
        Y = Y0 + h * dY if which == 0 else Y0.clone()
        m.pitch(T, 0.5, wavespeed=ws).evolve(Y)
        return 0.5 * Y.square().sum().item()

    want = [(J(1e-6, k) - J(-1e-6, k)) / 2e-6 for k in range(3)]
    mesh = mtp.Mesh(3, v, e, eps, mu, p=p, precision=prec)
    tents = mesh.pitch(T, 0.5, wavespeed=ws)
    for every in (0, 3):
        Y = Y0.to(mesh.torch_dtype(), copy=True)
        YT = Y.clone()
        tents.evolve(YT)
        l0, ge, gm = _gradients(mesh, tents, Y, YT, every)
        got = [(l0.double() * dY).sum().item(), (ge.cpu().numpy() * de).sum(), (gm.cpu().numpy() * dm).sum()]
        for a, b in zip(got, want):
            assert abs(a - b) <= tol * Y0.square().sum().item(), (every, got, want)


@pytest.mark.parametrize("dim,p", [(2, 2), (3, 2)])
@pytest.mark.parametrize("every", [0, 2])
def test_several_right_hand_sides(dim, p, every):
    """Three right-hand sides at once: each state gradient has the bits of a call of its own (one CTA a tent and
    right-hand side), the material gradients are the sum of the three (sums by atomics, FP64: 1e-12 of the norm)."""
    v, e = S.square_mesh(3) if dim == 2 else S.cube_mesh(2)
    eps, mu = np.random.default_rng(1).uniform(1, 2, (2, len(e)))
    one, many = (mtp.Mesh(dim, v, e, eps, mu, p=p, n_rhs=n) for n in (1, 3))
    t1, t3 = (m.pitch(0.1, 0.5) for m in (one, many))
    Y, lam = (torch.tensor(np.random.default_rng(s).standard_normal(many.state_shape), device=DEV) for s in (2, 3))
    l0, ge, gm = _gradients(many, t3, Y, lam, every)
    parts = [_gradients(one, t1, Y[r:r + 1].contiguous(), lam[r:r + 1].contiguous(), every) for r in range(3)]
    for r in range(3):
        assert torch.equal(l0[r:r + 1], parts[r][0])
    for i, g in ((1, ge), (2, gm)):
        total = sum(q[i] for q in parts)
        assert (g - total).norm().item() <= 1e-12 * total.norm().item()
