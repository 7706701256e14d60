"""FP32 lattices large enough for strips by default: the automatic strips and bands against
another cut of the same lattice.  The arithmetic of a site does not depend on the cut, so
the states are equal bit for bit, at every boundary of a strip or a band."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,stencil,tau", [(4096, 4096, 4, 1.0), (2048, 2048, 8, 1.0),
                                               (1540, 1100, 4, 1.0), (900, 1800, 6, 1.0),
                                               (4100, 2052, 8, 0.8)])
def test_automatic_cut(nx, ny, stencil, tau):
    from paper_2212_07848_gb300 import abi
    from paper_2212_07848_gb300.lattice import Lattice
    states = []
    for kernel, strip in ((abi.LB_KERNEL_AUTO, 0), (abi.LB_KERNEL_PLAIN, 37)):
        g = Lattice(nx, ny, -4.2, tau, 1e-5, stencil=stencil)
        g.set_kernel(kernel)
        if strip:
            g.set_strip_height(strip)
        g.init(0.7, 5, 0.02)
        g.step(3)
        states.append(g.download_state())
        g.close()
    assert np.isfinite(states[0]).all()
    assert np.array_equal(*states)
