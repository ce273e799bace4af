"""The line between the two forms of the lattice exchange, in device time and in values."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import mtp_synth as S
import paper_1906_11029_gb300 as mtp

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _mesh(n_elems, p, prec):
    """48 tetrahedra with as many right-hand sides as make n_elems elements."""
    v, e = S.cube_mesh(2)
    one = np.ones(len(e))
    return mtp.Mesh(3, v, e, one, one, p=p, precision=prec, n_rhs=n_elems // len(e))


@pytest.mark.parametrize("to_lattice", [True, False])
@pytest.mark.parametrize("prec", [mtp.MTP_FP32, mtp.MTP_FP64])
def test_fewer_elements_take_no_longer(prec, to_lattice):
    """1920 elements (13 per SM of 152) against 3072: the form for many elements takes the same time for both, so the
    other one must not run where it takes longer.  A fifth for the timer."""
    times = []
    for n in (1920, 3072):
        mesh = _mesh(n, 4, prec)
        vals = torch.randn(mesh.lattice_shape, dtype=torch.float64, device=DEV)
        state = mesh.state_from_lattice(vals)

        def calls(k):
            for _ in range(k):
                if to_lattice:
                    mesh.state_to_lattice(state, vals)
                else:
                    mesh.state_from_lattice(vals, state)

        calls(3)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()      # the calls' device time alone
        with torch.cuda.graph(graph):
            calls(20)
        best = float("inf")
        for _ in range(5):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            graph.replay()
            b.record()
            b.synchronize()
            best = min(best, a.elapsed_time(b))
        times.append(best)
    assert times[0] <= 1.2 * times[1], times


@pytest.mark.parametrize("prec", [mtp.MTP_FP32, mtp.MTP_FP64])
@pytest.mark.parametrize("p", [1, 4])
def test_values_on_both_sides_of_the_line(p, prec):
    """1200 and 1248 elements lie around 8 per SM of 152, 2400 and 2448 around 16: the same values to the rounding of a
    product of n_basis terms (4 .. 35) in FP64, and of the state."""
    for few, many in ((1200, 1248), (2400, 2448)):
        a, b = _mesh(few, p, prec), _mesh(many, p, prec)
        vals = torch.randn(b.lattice_shape, generator=torch.Generator().manual_seed(p), dtype=torch.float64).to(DEV)
        sa, sb = a.state_from_lattice(vals[:a.n_rhs].contiguous()), b.state_from_lattice(vals)
        eps = 1e-14 if prec == mtp.MTP_FP64 else 2.0 ** -22
        scale = sb.abs().max().item()
        assert (sa - sb[:a.n_rhs]).abs().max().item() <= 35 * eps * scale
        va, vb = a.state_to_lattice(sa), b.state_to_lattice(sb)
        assert (va - vb[:a.n_rhs]).abs().max().item() <= 35 * eps * vb.abs().max().item() * 35
