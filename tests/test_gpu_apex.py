"""Apex tent kernels (3D, p = 1..4; 2D, p = 1..5), their many-instance forms, and the lattice / energy
kernels at the sizes where they can go wrong: patches from one element to the most that is accepted
(32 in 3D, 16 in 2D), every local index of the tent vertex and both element orientations (shuffled
vertex numbers), material jumps in eps and mu, several right-hand sides, element counts around the
32 of a block.

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
    if name == "one_tri":
        v, e = np.array([[0., 0], [1, .1], [.3, .8]]), np.array([[0, 1, 2]], np.int32)
    elif name in ("square1", "square3"):
        v, e = S.square_mesh(int(name[-1]))
        v = S.perturb_interior(v, 1.0 / 3, 0.15, 7)
    elif name == "fan16":
        t = 2 * np.pi * np.arange(16) / 16
        v = np.concatenate([[[0.0, 0.0]], np.stack([np.cos(t), np.sin(t)], 1)])
        e = np.array([[0, 1 + i, 1 + (i + 1) % 16] for i in range(16)], np.int32)
    elif name == "ball32":   # octahedron with every face split in four, coned from its centre
        v = [np.zeros(3)] + [s * x for x in np.eye(3) for s in (1.0, -1.0)]
        mid, e = {}, []

        def middle(a, b):
            if (min(a, b), max(a, b)) not in mid:
                mid[(min(a, b), max(a, b))] = len(v)
                v.append((v[a] + v[b]) / np.linalg.norm(v[a] + v[b]))
            return mid[(min(a, b), max(a, b))]

        for a in (1, 2):
            for b in (3, 4):
                for c in (5, 6):
                    ab, bc, ca = middle(a, b), middle(b, c), middle(c, a)
                    e += [[0, a, ab, ca], [0, b, ab, bc], [0, c, bc, ca], [0, ab, bc, ca]]
        v, e = np.array(v), np.array(e, np.int32)
    elif name == "one_tet":
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


_CASES = [(n, T, p) for n, T in (("one_tet", 0.1), ("cube1", 0.1), ("cube2", 0.05), ("graded3", 0.02), ("ball32", 0.06))
          for p in (1, 2, 3, 4)]
_CASES += [(n, T, p) for n, T in (("one_tri", 0.2), ("square1", 0.2), ("square3", 0.1), ("fan16", 0.1)) for p in (1, 2, 3, 4, 5)]


@pytest.mark.parametrize("name,T,p", _CASES)
def test_apex_kernel_matches_oracle(name, T, p):
    v, e, eps, mu = _problem(name)
    dim = v.shape[1]
    nf, nb = (3, (p + 1) * (p + 2) // 2) if dim == 2 else (6, (p + 1) * (p + 2) * (p + 3) // 6)
    vals = np.random.default_rng(p).standard_normal((len(e), nb, nf))
    ref = _oracle(v, e, eps, mu, p, T, vals)
    for prec in (mtp.MTP_FP64, mtp.MTP_FP32):
        mesh = mtp.Mesh(dim, v, e, eps, mu, p=p, precision=prec, n_rhs=2)
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


@pytest.mark.parametrize("name,degrees", [("cube2", (1, 2)), ("cube2", (3, 1, 2)), ("cube2", (4, 2, 3, 1)), ("cube2", (5, 2)),
                                          ("square3", (5, 1, 3)), ("square3", (4, 2))])
def test_batch_of_all_degrees_equals_single_evolves(name, degrees):
    v, e, eps, mu = _problem(name)
    for prec in (mtp.MTP_FP64, mtp.MTP_FP32):
        if prec == mtp.MTP_FP64 and name == "cube2" and max(degrees) == 5:
            continue    # FP64 p = 5 in 3D needs more shared memory than a block may have
        tents, states, ref = [], [], []
        for i, p in enumerate(degrees):
            mesh = mtp.Mesh(v.shape[1], v, e, eps, mu, p=p, precision=prec, n_rhs=1 + i % 2)
            tents.append(mesh.pitch(0.04, 0.5))
            st = torch.randn(mesh.state_shape, generator=torch.Generator().manual_seed(i), dtype=torch.float64)
            states.append(st.to(DEV, mesh.torch_dtype()))
            ref.append(states[-1].clone())
            tents[-1].evolve(ref[-1])
        mtp.Batch(tents).evolve(states)
        # FP64: the same arithmetic compiled into another kernel; FP32 batches with p = 5 run the general one
        for a, b in zip(states, ref):
            assert rel_l2(a.cpu().numpy(), b.cpu().numpy()) <= (1e-13 if prec == mtp.MTP_FP64 else 1e-5)


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


@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("p", [1, 2, 3, 4, 5])
def test_lattice_exchange_many_elements(dim, p):
    """More elements (over all right-hand sides) than the small kernels take, not a multiple of 32, against one
    right-hand side at a time, which they do take: 1e-13 in FP64, an FP32 rounding for an FP32 state, the same
    bits for split precision (products in one order)."""
    v, e = S.square_mesh(27) if dim == 2 else S.cube_mesh(5)
    one, nrhs = np.ones(len(e)), 2 if dim == 2 else 4
    for prec, tol in ((mtp.MTP_FP64, 1e-13), (mtp.MTP_FP32, 2.0 ** -23), (mtp.MTP_FP32_SPLIT, 0.0)):
        many = mtp.Mesh(dim, v, e, one, one, p=p, precision=prec, n_rhs=nrhs)
        few = mtp.Mesh(dim, v, e, one, one, p=p, precision=prec)
        nf, nb = many.state_shape[-2:]
        vals = torch.tensor(np.random.default_rng(p).standard_normal((nrhs, len(e), nb, nf)), device=DEV)
        st, want = many.state_from_lattice(vals), torch.cat([few.state_from_lattice(x[None].contiguous()) for x in vals])
        assert (st - want).norm().item() <= tol * want.norm().item()
        back, want = many.state_to_lattice(st), torch.cat([few.state_to_lattice(x[None].contiguous()) for x in st])
        assert (back - want).norm().item() <= 1e-13 * want.norm().item()


@pytest.mark.parametrize("dim", [2, 3])
def test_vertex_without_elements(dim):
    """A vertex that no element uses has a tent of no elements; the rest of the mesh is not affected."""
    v, e = S.square_mesh(2) if dim == 2 else S.cube_mesh(1)
    one = np.ones(len(e))
    outs = []
    for extra in (0, 1):
        vv = np.concatenate([v, np.full((extra, dim), 5.0)])
        mesh = mtp.Mesh(dim, vv, e, one, one, p=2, precision=mtp.MTP_FP64)
        tents = mesh.pitch(0.1, 0.5)
        assert len(tents.get()["vertex"]) == len(mesh.pitch(0.1, 0.5, device=True).get()["vertex"])
        for launch in (0, 2):
            tents.set_launch(launch)
            st = torch.ones(mesh.state_shape, dtype=torch.float64, device=DEV)
            tents.evolve(st)
            outs.append(st)
    assert all(torch.equal(outs[0], o) for o in outs[1:])


@pytest.mark.parametrize("name,p", [("cube2", 1), ("cube2", 2), ("ball32", 2), ("one_tet", 2), ("cube2", 3)])
def test_apex_adjoint_matches_directional_differences(name, p):
    """Gradients w.r.t. the initial state, eps and mu along one direction each against central differences of
    FP64 evolves (h = 1e-6: about 1e-9 of rounding and h^2 of truncation; FP32 adds its own 1e-5)."""
    v, e, eps, mu = _problem(name)
    T = 0.05
    rng = np.random.default_rng(p)
    ws = np.ones(len(e))
    ref = mtp.Mesh(3, v, e, eps, mu, p=p)
    Y0 = torch.tensor(rng.standard_normal(ref.state_shape), device=DEV)
    dY, de, dm = torch.tensor(rng.standard_normal(ref.state_shape), device=DEV), rng.standard_normal(len(e)), rng.standard_normal(len(e))

    def J(h, which):
        m = mtp.Mesh(3, v, e, eps + (h * de if which == 1 else 0), mu + (h * dm if which == 2 else 0), p=p)
        Y = Y0 + h * dY if which == 0 else Y0.clone()
        m.pitch(T, 0.5, wavespeed=ws).evolve(Y)
        return 0.5 * Y.square().sum().item()

    want = [(J(1e-6, k) - J(-1e-6, k)) / 2e-6 for k in range(3)]
    scale = Y0.square().sum().item()
    for prec, tol in ((mtp.MTP_FP64, 1e-8), (mtp.MTP_FP32, 1e-5)):
        if prec == mtp.MTP_FP64 and p > 2:
            continue    # the differences above cover the forward; cube2's FP64 gradients run at p = 1, 2
        m = mtp.Mesh(3, v, e, eps, mu, p=p, precision=prec)
        t = m.pitch(T, 0.5, wavespeed=ws)
        for every in (0, 3):
            Y = Y0.to(m.torch_dtype()).requires_grad_(True)
            pe, pm = (torch.tensor(x, device=DEV, requires_grad=True) for x in (eps, mu))
            YT = mtp.mtp_evolve_autograd(Y, pe, pm, t, every)
            if name == "ball32" and prec == mtp.MTP_FP64:    # patch beyond the adjoint's shared memory: refused
                with pytest.raises(mtp.MtpError, match="shared memory"):
                    torch.autograd.grad(0.5 * YT.square().sum(), (Y, pe, pm))
                continue
            gY, ge, gm = torch.autograd.grad(0.5 * YT.square().sum(), (Y, pe, pm))
            got = [(gY.double() * dY).sum().item(), (ge.cpu().numpy() * de).sum(), (gm.cpu().numpy() * dm).sum()]
            for a, b in zip(got, want):
                assert abs(a - b) <= tol * scale, (prec, every, got, want)


@pytest.mark.parametrize("n,p,wide", [(2, 1, 0), (3, 2, 0), (2, 3, 0), (22, 1, 1), (22, 2, 1), (22, 3, 1), (2, 4, 0), (2, 5, 0)])
def test_split_shapes_match_fp64(n, p, wide):
    """Split precision on both sides of the layer-width rule against FP64 (FP32 operator: 1e-5), and the
    persistent walk against per-layer launches (the same bits)."""
    v, e = S.cube_mesh(n)
    x = 2.0 ** (3 * v) / 8       # graded, so that layers are wide
    eps = 1 + np.random.default_rng(n).random(len(e))
    outs = []
    for prec in (mtp.MTP_FP64, mtp.MTP_FP32_SPLIT):
        if prec == mtp.MTP_FP64 and p == 5:
            prec = mtp.MTP_FP32     # FP64 has no p = 5 in 3D
        m = mtp.Mesh(3, x if wide else v, e, eps, np.ones(len(e)), p=p, precision=prec)
        t = m.pitch(0.002 if wide else 0.1, 0.5)
        ptr = t.get()["layer_ptr"]
        assert (ptr[-1] > 152 * (len(ptr) - 1)) == bool(wide)
        Y0 = torch.tensor(np.random.default_rng(p).standard_normal(m.state_shape), device=DEV)
        Y = Y0.to(m.torch_dtype(), copy=True)
        t.evolve(Y)
        outs.append(Y.double())
    Z = Y0.clone()
    t.set_launch(2)
    t.evolve(Z)
    assert torch.equal(Z, outs[1])
    assert ((outs[0] - outs[1]).norm() / outs[0].norm()).item() < 1e-5
