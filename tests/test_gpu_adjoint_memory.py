"""The default checkpoint plan of the gradient (one segment where there is room, about sqrt(layers) where there is
not, the same gradients either way), and its report of a forward evolve that fails in the last layer."""
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


def test_default_plan_falls_back_when_memory_is_short():
    """8^3 x 6, p = 2, FP64: all layers in one segment take about 200 MB, checkpoints every sqrt(layers) 60 MB; 140 MB
    are left free."""
    w = S.adjoint_cube(n=8, p=2, T=0.4)
    mesh = mtp.Mesh(3, w.verts, w.elems, w.eps, w.mu, p=2)
    Y, lam = (torch.tensor(np.random.default_rng(i).standard_normal(mesh.state_shape), device=DEV) for i in (1, 2))

    def outputs():
        return [torch.empty_like(Y)] + [torch.empty(len(w.elems), dtype=torch.float64, device=DEV) for _ in range(2)]

    tents, out = [mesh.pitch(w.T, 0.5, wavespeed=np.ones(len(w.elems))) for _ in range(2)], [outputs() for _ in range(2)]
    mtp.mtp_adjoint(tents[0].h, Y, lam, *out[0], 0)
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    rest = torch.empty(before - 140 * MB, dtype=torch.uint8, device=DEV)
    try:
        mtp.mtp_adjoint(tents[1].h, Y, lam, *out[1], 0)
        torch.cuda.synchronize()
    finally:
        del rest
        torch.cuda.empty_cache()
    for a, b in zip(*out):     # sums by atomics: their order may differ
        assert (a - b).norm().item() <= 1e-13 * a.norm().item()


@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("every", [0, 2])
def test_overflow_in_the_last_layer_is_reported(dim, every):
    """The gradient reports a forward evolve that first becomes non-finite in its last layer, as the evolve does.  Such
    an amplitude exists for some states: the largest one that all layers but the last bear is above that of the whole."""
    v, e = S.square_mesh(1) if dim == 2 else S.cube_mesh(1)
    one = np.ones(len(e))
    mesh = mtp.Mesh(dim, v, e, one, one, p=1, precision=mtp.MTP_FP32)
    tents = mesh.pitch(0.1, 0.5)
    nl = tents.info["n_layers"]

    def survives(Y, exponent, layers):
        Z = Y * 2.0 ** exponent
        try:
            tents.evolve_layers(Z, 0, layers)
        except mtp.MtpError as ex:
            assert ex.code == mtp.MTP_ENUMERIC
            return False
        return True

    def limit(Y, layers):
        lo, hi = 0.0, 127.0
        while hi - lo > 0.01:
            mid = 0.5 * (lo + hi)
            lo, hi = (mid, hi) if survives(Y, mid, layers) else (lo, mid)
        return lo, hi

    for seed in range(200):
        Y = torch.randn(mesh.state_shape, generator=torch.Generator().manual_seed(seed)).to(DEV)
        a, b = limit(Y, nl)[1], limit(Y, nl - 1)[0]
        if a < b:
            break
    else:
        pytest.fail("no state overflows in the last layer alone")
    Z = Y * 2.0 ** b
    l0, ge, gm = torch.empty_like(Z), *(torch.empty(len(e), dtype=torch.float64, device=DEV) for _ in range(2))
    with pytest.raises(mtp.MtpError) as ex:
        mtp.mtp_adjoint(tents.h, Z, torch.zeros_like(Z), l0, ge, gm, every)
    assert ex.value.code == mtp.MTP_ENUMERIC
