"""Lattices of more than 65535 rows of tiles (8 lattice rows each), the limit of a grid's
second dimension: the FP64 step against the oracle, the FP32 step against the strips
that are asked for, at the sizes next to the limit and beyond."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ny", [524280, 524284, 1048568])
def test_fp64(ny):
    from oracle import oracle as O
    from paper_2212_07848_gb300.lattice import Lattice
    g = Lattice(4, ny, -4.2, 0.9, 1e-5, precision="fp64")
    o = O.OracleLattice(4, ny, -4.2, 0.9, 1e-5)
    for lat in (g, o):
        lat.init(0.7, 5, 0.02)
        lat.step(1)
    fg, fo = g.populations(), o.populations()
    assert np.max(np.abs(fg - fo) / np.abs(fo)) < 1e-12   # the FP64 parity bound
    g.close()


@pytest.mark.parametrize("nx,ny,stencil,tau", [(4, 524284, 4, 0.8), (4, 1048600, 8, 0.8),
                                               (12, 600004, 6, 0.9), (4, 524280, 4, 0.8)])
def test_fp32(nx, ny, stencil, tau):
    from paper_2212_07848_gb300 import abi
    from paper_2212_07848_gb300.lattice import Lattice
    states = []
    for kernel in (abi.LB_KERNEL_AUTO, abi.LB_KERNEL_OVERLAP):
        g = Lattice(nx, ny, -4.2, tau, 1e-5, stencil=stencil)
        g.set_kernel(kernel)
        g.init(0.7, 5, 0.02)
        g.step(2)
        states.append(g.download_state())
        g.close()
    assert np.isfinite(states[0]).all()
    assert np.array_equal(*states)
