"""Launch choices of the DAG walk follow the layers that hold the tents, not their average width: a few small elements
make many narrow layers while most tents stay in wide ones (152 SMs, where two CTAs of the kernel fit)."""
import numpy as np
import pytest

import mtp_synth as S
import paper_1906_11029_gb300 as mtp


def _cube(n, pull=0.0):
    """Kuhn cube with its middle vertex moved by a part of the element size towards the next one on the diagonal."""
    v, e = S.cube_mesh(n)
    v = v.copy()
    v[np.argmin(np.linalg.norm(v - 0.5, axis=1))] += pull / n
    return v, e


def _tents(mesh, T, p=2, precision=mtp.MTP_FP32):
    v, e = mesh
    one = np.ones(len(e))
    return mtp.Mesh(v.shape[1], v, e, one, one, p=p, precision=precision).pitch(T, 0.5)


def _widths(t):
    n = np.diff(t.get()["layer_ptr"])
    return n.mean(), (n.astype(float) ** 2).sum() / n.sum()


def test_uneven_layers_take_the_ctas_of_the_wide_ones():
    t = _tents(_cube(20, 0.95), 0.02)
    mean, weighted = _widths(t)
    assert mean < 152 < 304 < weighted          # one CTA per SM on average, three where the tents are
    assert mtp.mtp_tents_walk(t.h, 152, 2)[0] == 2
    t = _tents(_cube(20, 0.95), 0.02, 3)
    assert mtp.mtp_tents_walk(t.h, 152, 2)[0] == 2
    t = _tents(_cube(16, 0.97), 0.02)           # few wide layers among many that hold a few tents
    assert _widths(t)[0] < 60
    assert mtp.mtp_tents_walk(t.h, 152, 2)[0] == 1


@pytest.mark.parametrize("n,T,want", [(3, 0.1, 1), (13, 0.1, 1), (20, 0.02, 2), (24, 0.02, 3)])
def test_even_layers(n, T, want):
    t = _tents((S.perturb_interior(S.cube_mesh(n)[0], 1.0 / n, 0.15, 11029), S.cube_mesh(n)[1]), T)
    assert mtp.mtp_tents_walk(t.h, 152, 3) == (want, 0)
    assert mtp.mtp_tents_walk(t.h, 152, 1) == (1, 0)
    assert mtp.mtp_tents_walk(t.h, 1, 3)[0] == 3        # every layer is wide for one SM


def test_split_item_shape():
    for p, mesh, T, want in ((2, _cube(24, 0.95), 0.02, 0), (2, _cube(16, 0.97), 0.02, 2), (3, _cube(6), 0.1, 2),
                             (4, _cube(6), 0.1, 0)):
        t = _tents(mesh, T, p, mtp.MTP_FP32_SPLIT)
        assert mtp.mtp_tents_walk(t.h, 152, 2)[1] == want
    t = _tents(S.square_mesh(4), 0.1, 2, mtp.MTP_FP32_SPLIT)
    assert mtp.mtp_tents_walk(t.h, 152, 2) == (1, 0)


def test_arguments():
    t = _tents(_cube(2), 0.1)
    for sms, fit in ((0, 1), (152, 0)):
        with pytest.raises(mtp.MtpError) as ex:
            mtp.mtp_tents_walk(t.h, sms, fit)
        assert ex.value.code == mtp.MTP_EINVAL
