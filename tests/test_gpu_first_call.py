"""What the first call on a mesh allocates: exchange and energy need geometry, patches and small tables; the apex
kernels' records come with the first call that runs such a kernel."""
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import mtp_synth as S
import paper_1906_11029_gb300 as mtp

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("dim,n,prec", [(3, 24, mtp.MTP_FP32), (3, 24, mtp.MTP_FP64), (2, 200, mtp.MTP_FP64)])
def test_exchange_does_not_allocate_evolve_records(dim, n, prec):
    """Of an element the exchange holds 32 FP64 of geometry, its vertices and its patch entries (12 bytes of local
    numbers and an index each): under 352 bytes; 4 MB for tables and 2 MB of granularity for each of
    at most sixteen buffers and pools.  The records of 896 or 1792 bytes a tetrahedron, 768 a triangle in FP64, would not fit in that."""
    v, e = S.square_mesh(n) if dim == 2 else S.cube_mesh(n)
    one = np.ones(len(e))
    warm = mtp.Mesh(dim, v, e, one, one, p=1, precision=prec)
    vals = torch.zeros(warm.lattice_shape, dtype=torch.float64, device=DEV)
    state = warm.state_from_lattice(vals)
    warm.energy(state)
    mesh = mtp.Mesh(dim, v, e, one, one, p=1, precision=prec)
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    mesh.state_from_lattice(vals, state)
    mesh.energy(state)
    torch.cuda.synchronize()
    used = before - torch.cuda.mem_get_info()[0]
    assert used <= 352 * len(e) + 4 * (1 << 20) + 16 * (2 << 20)


@pytest.mark.parametrize("dim,p", [(2, 3), (3, 2)])
def test_first_evolves_from_several_threads(dim, p):
    """Tents handles of one mesh whose first evolves start together in threads and streams of their own: the bits of
    a mesh that was used before."""
    v, e = S.square_mesh(6) if dim == 2 else S.cube_mesh(3)
    one = np.ones(len(e))
    mesh, ref = (mtp.Mesh(dim, v, e, one, one, p=p) for _ in range(2))
    Y0 = torch.tensor(np.random.default_rng(p).standard_normal(mesh.state_shape), device=DEV)
    mesh.energy(Y0)     # the mesh itself is on the device
    want = Y0.clone()
    ref.pitch(0.1, 0.5).evolve(want)
    tents, got = [mesh.pitch(0.1, 0.5) for _ in range(4)], [Y0.clone() for _ in range(4)]
    torch.cuda.synchronize()
    barrier, errors = threading.Barrier(4), []

    def work(i):
        try:
            s = torch.cuda.Stream()
            barrier.wait()
            tents[i].evolve(got[i], stream=s.cuda_stream)
        except Exception as ex:
            errors.append(ex)

    threads = [threading.Thread(target=work, args=(i,)) for i in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors
    assert all(torch.equal(g, want) for g in got)
