"""The layouts of the FP32 step kernel (strips of 64 and of 128 threads, tiles) at the
sizes where their cutting can go wrong: one pair of columns, strips a part of a
warp wide, several bands of rows side by side (with rows left over, or fewer rows
than bands), strips that do not divide the width, the last tile a part of one.  The
arithmetic of a site is the same in every layout, so the states are equal bit for
bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _run(nx, ny, stencil, tau, kernel, strip, precision="fp32"):
    from paper_2212_07848_gb300.lattice import Lattice
    g = Lattice(nx, ny, -4.2, tau, 1e-5, stencil=stencil, precision=precision)
    g.set_kernel(kernel)
    if strip:
        g.set_strip_height(strip)
    g.init(0.7, 5, 0.02)
    pow2 = (nx & (nx - 1)) == 0 and (ny & (ny - 1)) == 0
    if pow2:
        g.sk_config(3, 3)
    g.step(7)
    out = g.download_state(), g.structure_factor()[0] if pow2 else None
    g.close()
    return out


@pytest.mark.parametrize("stencil,tau", [(4, 1.0), (4, 0.8), (6, 1.0), (8, 0.8)])
@pytest.mark.parametrize("nx,ny", [(4, 4), (4, 100), (12, 20), (32, 32), (60, 8), (64, 64),
                                   (124, 12), (132, 36), (252, 20), (256, 16), (260, 12),
                                   (516, 8), (1028, 8)])
def test_layouts_agree(nx, ny, stencil, tau):
    from paper_2212_07848_gb300 import abi
    ref, sk = _run(nx, ny, stencil, tau, abi.LB_KERNEL_AUTO, 0)
    assert np.isfinite(ref).all()
    for kernel, strips in ((abi.LB_KERNEL_PLAIN, (1, 3, ny)), (abi.LB_KERNEL_OVERLAP, (0, 2, ny))):
        for strip in strips:
            got, s = _run(nx, ny, stencil, tau, kernel, strip)
            assert np.array_equal(ref, got), (kernel, strip)
            assert sk is None or np.array_equal(sk, s), (kernel, strip)


@pytest.mark.parametrize("nx,ny", [(4, 4), (20, 12), (132, 36), (512, 260)])
def test_fp64_tiles_match_the_oracle(nx, ny):
    """Both FP64 tile shapes (below and above 2^17 sites), odd edges included; the
    library's FP64 parity bound after a few steps."""
    from oracle import oracle as O
    from paper_2212_07848_gb300.lattice import Lattice
    g = Lattice(nx, ny, -4.2, 0.9, 1e-5, stencil=6, precision="fp64")
    o = O.OracleLattice(nx, ny, -4.2, 0.9, 1e-5, stencil=6)
    for lat in (g, o):
        lat.init(0.7, 5, 0.02)
        lat.step(5)
    fg, fo = g.populations(), o.populations()
    assert np.max(np.abs(fg - fo) / np.abs(fo)) < 1e-12
    g.close()


@pytest.mark.parametrize("stencil", [4, 8])
@pytest.mark.parametrize("strip", [1, 5, 64])
def test_ensemble_bands_match_lattices(stencil, strip):
    """Replicas narrow enough for several bands per tile, with rows left over."""
    from paper_2212_07848_gb300 import abi
    from paper_2212_07848_gb300.ensemble import Ensemble
    from paper_2212_07848_gb300.lattice import Lattice
    reps = [(16, 36, -4.0, 1.0, 1e-5, 0.7), (64, 20, -4.2, 0.9, 1e-5, 0.69),
            (260, 12, -4.1, 1.0, 1e-5, 0.7), (4, 8, -4.0, 1.0, 1e-5, 0.7)]
    for launch in (abi.LB_ENS_PER_STEP, abi.LB_ENS_PERSISTENT):
        e = Ensemble(reps, stencil=stencil, seed=2)
        e.set_resident(abi.LB_ENS_RESIDENT_OFF)
        e.set_launch(launch)
        e.set_strip_height(strip)
        e.init(0.01)
        e.step(35)
        e.sync()
        for r, (nx, ny, G, tau, kT, rho0) in enumerate(reps):
            g = Lattice(nx, ny, G, tau, kT, stencil=stencil)
            g.set_replica(r)
            g.init(rho0, 2, 0.01)
            g.step(35)
            assert np.array_equal(g.populations(), e.populations(r)), (launch, r)
            g.close()
        e.close()


@pytest.mark.parametrize("stencil,tau", [(4, 1.0), (4, 0.9), (8, 1.0), (8, 0.9)])
@pytest.mark.parametrize("nx,ny", [(32, 8), (32, 24), (64, 8), (64, 40), (128, 32), (128, 256)])
def test_resident_shapes_match_tiles(nx, ny, stencil, tau):
    """Fewer pairs than threads, a last round of pairs that some threads sit out, one
    CTA and clusters of up to eight (128 x 256), windows ending in a sample."""
    from paper_2212_07848_gb300 import abi
    from paper_2212_07848_gb300.ensemble import Ensemble
    reps = [(nx, ny, -4.0 - 0.1 * r, tau, 1e-5, 0.7) for r in range(3)]
    out = []
    for mode in (abi.LB_ENS_RESIDENT_ON, abi.LB_ENS_RESIDENT_OFF):
        e = Ensemble(reps, stencil=stencil, seed=4)
        e.set_resident(mode)
        assert e.num_resident == (3 if mode == abi.LB_ENS_RESIDENT_ON else 0)
        e.set_launch(abi.LB_ENS_PERSISTENT)
        e.init(0.01)
        pow2 = (ny & (ny - 1)) == 0
        if pow2:
            e.sk_config(4, 4)
        e.step(1)
        e.step(12)
        e.sync()
        out.append([e.populations(r) for r in range(3)] +
                   ([e.structure_factor(r)[0] for r in range(3)] if pow2 else []))
        e.close()
    assert all(np.array_equal(a, b) for a, b in zip(*out))


@pytest.mark.parametrize("nx,ny,nz,precision,tau", [
    (32, 4, 3, "fp32", 1.0), (32, 32, 33, "fp32", 0.8), (96, 84, 50, "fp32", 1.0),
    (64, 64, 64, "fp32", 1.0), (32, 8, 200, "fp32", 1.0), (32, 12, 9, "fp64", 1.0),
    (64, 64, 20, "fp64", 0.8)])
def test_3d_default_strip_agrees(nx, ny, nz, precision, tau):
    """The default cut along z against one strip, single planes and a remainder."""
    from paper_2212_07848_gb300.lattice3 import Lattice3
    states = []
    for strip in (0, nz, 1, 2):
        g = Lattice3(nx, ny, nz, -3.6, tau, 1e-6, precision=precision)
        if strip:
            g.set_strip(strip)
        g.init(0.7, 5, 0.02)
        g.step(4)
        states.append(g.populations())
        g.close()
    assert np.isfinite(states[0]).all()
    for s in states[1:]:
        assert np.array_equal(states[0], s)
