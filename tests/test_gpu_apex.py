"""Apex tent kernel (3D, p = 1..4), its many-instance form, and the lattice / energy kernels at the
sizes where they can go wrong: patches from 1 to 24 elements, every local index of the tent
vertex and both element orientations (shuffled vertex numbers), material jumps in eps and mu,
several right-hand sides, element counts around the 32 of a block.

Tolerances: those of the precision contract (FP64 1e-11, FP32 1e-5 against the oracle);
the two launch configurations run the same device code on the same inputs, so equality is asked."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import mtp_synth as S
import paper_1906_11029_gb300 as mtp
from _oracle_bridge import max_rel, rel_l2
from oracle.mesh import Mesh as OMesh
from oracle.mtp import Discretization
from oracle.pitch import pitch_tents

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
TOL = {mtp.MTP_FP64: 1e-11, mtp.MTP_FP32: 1e-5}


def _problem(name, seed=3):
    """(verts, elems, eps, mu): shuffled vertex numbers put the tent vertex at every local index."""
    rng = np.random.default_rng(seed)
    if name == "one_tet":
        v, e = np.array([[0., 0, 0], [1, .1, 0], [.2, .9, .1], [.1, .3, 1.1]]), np.array([[0, 1, 2, 3]], np.int32)
    else:
        n = {"cube1": 1, "cube2": 2, "graded3": 3}[name]
        v, e = S.cube_mesh(n, S.graded_coords(n, 8.0) if name == "graded3" else None)
        if name == "cube2":
            v = S.perturb_interior(v, 1.0 / n, 0.15, 7)
    perm = rng.permutation(len(v))
    w = np.empty_like(v)
    w[perm] = v
    e = perm[e].astype(np.int32)
    return w, e, rng.uniform(1.0, 3.0, len(e)), rng.uniform(1.0, 2.0, len(e))


def _oracle(v, e, eps, mu, p, T, vals):
    disc = Discretization(OMesh(v, e, eps, mu), p)
    Y, _ = disc.evolve(disc.moments_from_lattice(vals), pitch_tents(v, e, eps, mu, T, 0.5))
    return disc.eval_lattice(disc.y_coeffs(Y))


@pytest.mark.parametrize("p", [1, 2, 3, 4])
@pytest.mark.parametrize("name,T", [("one_tet", 0.1), ("cube1", 0.1), ("cube2", 0.05), ("graded3", 0.02)])
def test_apex_kernel_matches_oracle(name, T, p):
    v, e, eps, mu = _problem(name)
    vals = np.random.default_rng(p).standard_normal((len(e), (p + 1) * (p + 2) * (p + 3) // 6, 6))
    ref = _oracle(v, e, eps, mu, p, T, vals)
    for prec in (mtp.MTP_FP64, mtp.MTP_FP32):
        mesh = mtp.Mesh(3, v, e, eps, mu, p=p, precision=prec, n_rhs=2)
        tents = mesh.pitch(T, 0.5)
        outs = []
        for launch in (0, 2):
            tents.set_launch(launch)
            st = mesh.state_from_lattice(torch.tensor(np.stack([vals, -2.0 * vals]), device=DEV))
            tents.evolve(st)
            outs.append(st.clone())
            got = mesh.state_to_lattice(st).cpu().numpy()
            for g, s in ((got[0], 1.0), (got[1], -2.0)):
                assert rel_l2(g, s * ref) <= TOL[prec] and max_rel(g, s * ref) <= TOL[prec], (launch, rel_l2(g, s * ref))
        assert torch.equal(outs[0], outs[1])


def test_apex_batch_of_all_degrees_equals_single_evolves():
    v, e, eps, mu = _problem("cube2")
    for prec in (mtp.MTP_FP64, mtp.MTP_FP32):
        for degrees in ((1, 2), (3, 1, 2), (4, 2, 3, 1)):
            tents, states, ref = [], [], []
            for i, p in enumerate(degrees):
                mesh = mtp.Mesh(3, v, e, eps, mu, p=p, precision=prec, n_rhs=1 + i % 2)
                tents.append(mesh.pitch(0.04, 0.5))
                st = torch.randn(mesh.state_shape, generator=torch.Generator().manual_seed(i), dtype=torch.float64)
                states.append(st.to(DEV, mesh.torch_dtype()))
                ref.append(states[-1].clone())
                tents[-1].evolve(ref[-1])
            mtp.Batch(tents).evolve(states)
            # one set of device functions compiled into two kernels: equal up to contraction choices
            for a, b in zip(states, ref):
                assert rel_l2(a.cpu().numpy(), b.cpu().numpy()) <= (1e-13 if prec == mtp.MTP_FP64 else 1e-6)


@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("p", [1, 2, 3, 4, 5])
def test_lattice_exchange_and_energy(dim, p):
    """Element counts 1, 31 .. 33 of a longer mesh; values against the oracle's energy and the exact roundtrip."""
    full_v, full_e = S.square_mesh(5) if dim == 2 else S.cube_mesh(2)
    rng = np.random.default_rng(p)
    for ne in (1, 31, 32, 33):
        e = full_e[:ne]
        used = np.unique(e)
        back = np.full(len(full_v), -1)
        back[used] = np.arange(len(used))
        v, e = full_v[used], back[e].astype(np.int32)
        eps, mu = rng.uniform(1, 3, ne), rng.uniform(1, 2, ne)
        nf, nb = (3, (p + 1) * (p + 2) // 2) if dim == 2 else (6, (p + 1) * (p + 2) * (p + 3) // 6)
        vals = rng.standard_normal((2, ne, nb, nf))
        disc = Discretization(OMesh(v, e, eps, mu), p)
        want = [disc.energy(disc.fields_at_flat_front(disc.moments_from_lattice(x))) for x in vals]
        for prec, tol in ((mtp.MTP_FP64, 1e-11), (mtp.MTP_FP32, 1e-5)):
            mesh = mtp.Mesh(dim, v, e, eps, mu, p=p, precision=prec, n_rhs=2)
            st = mesh.state_from_lattice(torch.tensor(vals, device=DEV))
            out = mesh.state_to_lattice(st).cpu().numpy()
            assert rel_l2(out, vals) <= tol and max_rel(out, vals) <= tol
            assert np.allclose(mesh.energy(st), want, rtol=tol, atol=0)
