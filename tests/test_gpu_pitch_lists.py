"""The device pitcher's lists: rounds whose tents fill a block's list before the launch's last round, and meshes with
more vertices than resident threads (several a thread); the tent list stays that of the host, bit for bit, and the
device memory within what the header states."""
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import mtp_synth as S
import paper_1906_11029_gb300 as mtp
from test_gpu_pitch import _same

pytestmark = pytest.mark.gpu


def _square(n):
    """S.square_mesh without its Python loops."""
    x = np.linspace(0.0, 1.0, n + 1)
    Y, X = np.meshgrid(x, x, indexing="ij")
    j, i = np.divmod(np.arange(n * n), n)
    a = i + (n + 1) * j
    e = np.stack([np.stack([a, a + 1, a + n + 2], 1), np.stack([a, a + n + 2, a + n + 1], 1)], 1).reshape(-1, 3)
    return np.stack([X.ravel(), Y.ravel()], 1), e.astype(np.int32)


# 15: 256 vertices in one block, a tenth of them a round: full after about 50 of 128 rounds; 40: several blocks;
# 600: 361 201 vertices, more than 152 x 8 blocks of 256
@pytest.mark.parametrize("n,T", [(15, 0.5), (40, 0.2), (600, 0.001)])
def test_full_lists_and_many_vertices(n, T):
    v, e = _square(n)
    v = S.perturb_interior(v, 1.0 / n, 0.15, 3)
    one = np.ones(len(e))
    mesh = mtp.Mesh(2, v, e, one, one, p=1)
    want, got = mesh.pitch(T, 0.5), mesh.pitch(T, 0.5, device=True)
    _same(got.get(), want.get())
    assert got.info == want.info


def test_device_memory_per_vertex():
    """The least free memory seen from another thread while a mesh of 361 201 vertices is pitched: the header's 280
    bytes a vertex and 12 a directed edge (2.2 million), with 20 MB for modules and allocation granularity."""
    v, e = _square(600)
    one = np.ones(len(e))
    mesh = mtp.Mesh(2, v, e, one, one, p=1)
    mesh.pitch(0.0005, 0.5, device=True)
    torch.cuda.synchronize()
    before = least = torch.cuda.mem_get_info()[0]
    done = threading.Event()

    def watch():
        nonlocal least
        while not done.is_set():
            least = min(least, torch.cuda.mem_get_info()[0])

    th = threading.Thread(target=watch)
    th.start()
    try:
        mesh.pitch(0.005, 0.5, device=True)
    finally:
        done.set()
        th.join()
    assert before - least <= 280 * len(v) + 12 * 2_200_000 + 20_000_000
