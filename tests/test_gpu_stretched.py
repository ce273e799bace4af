"""Stretched meshes (longest edge over smallest height of an element above 12, or 7.5 in the root mean square) run
the general kernels, whose rounding error does not grow with the stretch: evolve, batches and gradients against
the oracle or FP64 at the tolerances of the precision contract (FP64 1e-11, FP32 1e-5)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import mtp_synth as S
import paper_1906_11029_gb300 as mtp
from _oracle_bridge import max_rel, rel_l2
from test_gpu_apex import TOL, _oracle, _problem

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _stretch(v, how, s):
    return v * np.array({"z*": [1, 1, s], "z/": [1, 1, 1 / s], "xy*": [1, s, s], "y*": [1, s], "y/": [1, 1 / s]}[how])


_CASES = [("cube2", how, s, p) for how, s in (("z*", 1000.0), ("z/", 1000.0), ("xy*", 100.0), ("z*", 5.0), ("z*", 6.0))
          for p in (1, 2, 3, 4)]
_CASES += [("square3", how, s, p) for how, s in (("y*", 1000.0), ("y/", 1000.0), ("y*", 7.0), ("y*", 8.0)) for p in (1, 2, 3, 4, 5)]


@pytest.mark.parametrize("name,how,s,p", _CASES)
def test_evolve_on_stretched_mesh(name, how, s, p):
    v, e, eps, mu = _problem(name)
    v = _stretch(v, how, s)
    dim, T = v.shape[1], 0.04 / (s if "/" in how else 1.0)
    nf, nb = (3, (p + 1) * (p + 2) // 2) if dim == 2 else (6, (p + 1) * (p + 2) * (p + 3) // 6)
    vals = np.random.default_rng(p).standard_normal((len(e), nb, nf))
    ref = _oracle(v, e, eps, mu, p, T, vals)
    for prec in (mtp.MTP_FP64, mtp.MTP_FP32):
        mesh = mtp.Mesh(dim, v, e, eps, mu, p=p, precision=prec)
        tents = mesh.pitch(T, 0.5)
        for variant in (0, 1, 2) if prec == mtp.MTP_FP32 else (0,):
            tents.set_variant(variant)
            st = mesh.state_from_lattice(torch.tensor(vals[None], device=DEV))
            tents.evolve(st)
            got = mesh.state_to_lattice(st).cpu().numpy()[0]
            assert rel_l2(got, ref) <= TOL[prec] and max_rel(got, ref) <= TOL[prec], (variant, rel_l2(got, ref))


def test_large_patches_in_fp64_keep_the_apex_kernel():
    """32 tetrahedra at p = 4 in FP64 do not fit the general kernel's shared memory."""
    v, e, eps, mu = _problem("ball32")
    v = _stretch(v, "z*", 20.0)
    vals = np.random.default_rng(0).standard_normal((len(e), 35, 6))
    ref = _oracle(v, e, eps, mu, 4, 0.06, vals)
    mesh = mtp.Mesh(3, v, e, eps, mu, p=4)
    tents = mesh.pitch(0.06, 0.5)
    states = [mesh.state_from_lattice(torch.tensor(vals[None], device=DEV)) for _ in range(2)]
    tents.evolve(states[0])
    mtp.Batch([tents]).evolve(states[1:])
    for st in states:
        assert rel_l2(mesh.state_to_lattice(st).cpu().numpy()[0], ref) <= 1e-11


@pytest.mark.parametrize("dim", [2, 3])
def test_batch_with_a_stretched_mesh(dim):
    """A regular and a stretched instance together equal their own evolves (the regular one's in the apex kernel)."""
    for prec, tol in ((mtp.MTP_FP64, 1e-13), (mtp.MTP_FP32, 1e-5)):
        tents, states, want = [], [], []
        for i, s in enumerate((1.0, 50.0)):
            v, e, eps, mu = _problem("square3" if dim == 2 else "cube2")
            mesh = mtp.Mesh(dim, _stretch(v, "y*" if dim == 2 else "z*", s), e, eps, mu, p=2 + i, precision=prec)
            tents.append(mesh.pitch(0.04, 0.5))
            st = torch.randn(mesh.state_shape, generator=torch.Generator().manual_seed(i), dtype=torch.float64)
            states.append(st.to(DEV, mesh.torch_dtype()))
            want.append(states[-1].clone())
            tents[-1].evolve(want[-1])
        mtp.Batch(tents).evolve(states)
        for got, ref in zip(states, want):
            assert rel_l2(got.cpu().numpy(), ref.cpu().numpy()) <= tol


@pytest.mark.parametrize("dim,precision", [(2, mtp.MTP_FP32), (3, mtp.MTP_FP32), (3, mtp.MTP_TF32X3)])
def test_gradient_on_stretched_mesh(dim, precision):
    """FP32 gradients against FP64 ones at a stretch of 100 (p = 2)."""
    v, e = S.square_mesh(2) if dim == 2 else S.cube_mesh(2)
    v = _stretch(v, "y*" if dim == 2 else "z*", 100.0)
    one, out = np.ones(len(e)), []
    for prec in (mtp.MTP_FP64, precision):
        mesh = mtp.Mesh(dim, v, e, one, one, p=2, precision=prec)
        t = mesh.pitch(0.1, 0.5)
        Y = torch.tensor(np.random.default_rng(1).standard_normal(mesh.state_shape), device=DEV)
        Y = Y.to(mesh.torch_dtype()).requires_grad_(True)
        pe, pm = (torch.ones(len(e), dtype=torch.float64, device=DEV, requires_grad=True) for _ in range(2))
        YT = mtp.mtp_evolve_autograd(Y, pe, pm, t)
        out.append([g.double().cpu().numpy() for g in torch.autograd.grad(0.5 * YT.square().sum(), (Y, pe, pm))])
    for ref, got in zip(*out):
        assert rel_l2(got, ref) <= 1e-5
