"""A first call whose device copies do not fit reports MTP_ENOMEM and leaves nothing half made: with room again, the
same handle works.  Meshes and tent lists that several threads use first, at once."""
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
MB = 1 << 20


def _without_room(left, call):
    """call() with `left` bytes of device memory free."""
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    rest = torch.empty(torch.cuda.mem_get_info()[0] - left, dtype=torch.uint8, device=DEV)
    try:
        with pytest.raises(mtp.MtpError) as ex:
            call()
        assert ex.value.code == mtp.MTP_ENOMEM
    finally:
        del rest
        torch.cuda.empty_cache()


def test_handles_survive_a_first_call_without_room():
    """The geometry of 82 944 tetrahedra is 21 MB, the list of 953 297 tents 27 MB in arrays of at most 8; 10 MB are left."""
    v, e = S.cube_mesh(24)
    one = np.ones(len(e))
    mesh, ref = (mtp.Mesh(3, v, e, one, one, p=1) for _ in range(2))
    tents, rtents = (m.pitch(0.3, 0.5, device=True) for m in (mesh, ref))
    assert 28 * tents.info["n_tents"] > 25 * MB
    vals = torch.randn(mesh.lattice_shape, generator=torch.Generator().manual_seed(0), dtype=torch.float64).to(DEV)
    state, want = mesh.new_state(vals.device), mesh.new_state(vals.device)
    ref.state_from_lattice(vals, want)
    _without_room(10 * MB, lambda: mesh.state_from_lattice(vals, state))
    mesh.state_from_lattice(vals, state)
    assert torch.equal(state, want)
    for m, s in ((mesh, state), (ref, want)):
        m.energy(s)
    _without_room(10 * MB, lambda: tents.evolve(state))
    assert torch.equal(state, want)
    tents.evolve_layers(state, 0, 3)
    rtents.evolve_layers(want, 0, 3)
    assert torch.equal(state, want)


def test_first_exchanges_from_several_threads():
    v, e = S.cube_mesh(8)
    one = np.ones(len(e))
    ref = mtp.Mesh(3, v, e, one, one, p=3)
    vals = torch.randn(ref.lattice_shape, generator=torch.Generator().manual_seed(0), dtype=torch.float64).to(DEV)
    want = ref.state_from_lattice(vals)
    for _ in range(5):
        mesh = mtp.Mesh(3, v, e, one, one, p=3)
        got = [torch.zeros_like(want) for _ in range(4)]
        torch.cuda.synchronize()
        barrier, errors = threading.Barrier(4), []

        def work(i):
            try:
                s = torch.cuda.Stream()
                barrier.wait()
                mesh.state_from_lattice(vals, got[i], stream=s.cuda_stream)
                s.synchronize()
            except Exception as ex:
                errors.append(ex)

        threads = [threading.Thread(target=work, args=(i,)) for i in range(4)]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
        assert not errors
        assert all(torch.equal(g, want) for g in got)
