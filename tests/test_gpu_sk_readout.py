"""The radial and moment read-outs of S(k) where their index arithmetic can go
wrong: the smallest box, long thin boxes, more bins than there are modes, one
bin.  The reference sums the library's own S(k) in FP64 over numpy index grids;
both sides add at most a few thousand FP64 terms of one sign, so they agree to
about 1e-13 and 1e-12 is asked for."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

LN2 = float(np.log(2.0))


def _folded(n):
    m = np.arange(n)
    return np.where(m <= n // 2, m, m - n)


@pytest.mark.parametrize("nx,ny", [(4, 4), (4, 256), (512, 4), (8, 64), (256, 256)])
@pytest.mark.parametrize("nbins", [1, 0, 4096])
def test_bins_and_moments(nx, ny, nbins):
    from paper_2212_07848_gb300.lattice import Lattice
    nbins = nbins or max(nx, ny) // 2
    g = Lattice(nx, ny, -3.6, 1.0, 1e-5)
    g.init(LN2, 7, 0.01)
    g.sk_config(1, 1)
    g.step(3)
    half, n = g.structure_factor()
    bins, nb = g.structure_factor(nbins)
    assert n == nb == 3
    S = np.empty((ny, nx))
    S[:, :nx // 2 + 1] = half
    for kx in range(nx // 2 + 1, nx):
        S[:, kx] = half[(-np.arange(ny)) % ny, nx - kx]
    L = max(nx, ny)
    q = np.hypot(*np.meshgrid(_folded(nx) * (L / nx), _folded(ny) * (L / ny)))
    b = np.rint(q).astype(int)
    b[0, 0] = -1
    keep = (b >= 0) & (b < nbins)
    cnt = np.bincount(b[keep], minlength=nbins)
    ref = np.bincount(b[keep], S[keep], minlength=nbins) / np.maximum(cnt, 1)
    assert np.array_equal(np.isnan(bins), cnt == 0)
    assert np.allclose(bins[cnt > 0], ref[cnt > 0], rtol=1e-12, atol=0.0)
    m = g.sk_moments()
    assert abs(m[0] / S.sum() - 1.0) < 1e-12
    assert abs(m[1] / (2 * np.pi / L * q * S).sum() - 1.0) < 1e-12
    g.close()


def test_ensemble_bins_equal_a_lattice():
    from paper_2212_07848_gb300.ensemble import Ensemble
    from paper_2212_07848_gb300.lattice import Lattice
    reps = [(64, 64, -4.0, 1.0, 1e-6, LN2), (128, 128, -4.4, 1.0, 1e-6, 0.7)]
    e = Ensemble(reps, seed=3)
    e.init(1e-3)
    e.sk_config(2, 2)
    e.step(6)
    for r, (nx, ny, G, tau, kT, rho0) in enumerate(reps):
        g = Lattice(nx, ny, G, tau, kT)
        g.set_replica(r)
        g.init(rho0, 3, 1e-3)
        g.sk_config(2, 2)
        g.step(6)
        a, na = e.structure_factor(r, nx // 2)
        b, nb = g.structure_factor(nx // 2)
        assert na == nb == 3 and np.array_equal(a, b, equal_nan=True)
        g.close()


def test_readout_reports_a_nonfinite_state():
    from paper_2212_07848_gb300 import abi
    from paper_2212_07848_gb300.lattice import Lattice
    g = Lattice(32, 32, -3.6, 1.0, 1e-5)
    g.init(LN2, 1, 0.0)
    g.sk_config(1, 1)
    f = g.populations()
    f[1, 3, 4] = np.nan
    g.set_populations(f)
    g.step(1)
    with pytest.raises(abi.LbError):
        g.structure_factor(16)
    g.init(LN2, 1, 0.0)
    g.step(1)
    assert np.isfinite(g.structure_factor(16)[0][1:]).all()
    g.close()


@pytest.mark.parametrize("nx,ny,nz", [(32, 4, 4), (32, 64, 8), (64, 4, 128)])
@pytest.mark.parametrize("nbins", [1, 0, 5000])
def test_shells_moments_and_axes_in_3d(nx, ny, nz, nbins):
    from paper_2212_07848_gb300.lattice3 import Lattice3
    g = Lattice3(nx, ny, nz, -3.6, 1.0, 1e-5, precision="fp64")
    g.init(LN2, 5, 0.01)
    g.sk_config(4, 4)
    g.sk_full()
    g.step(4)
    rho = g.density()
    S = np.abs(np.fft.fftn(rho - rho.mean())) ** 2 / rho.size
    S[0, 0, 0] = 0.0
    L = max(nx, ny, nz)
    qz, qy, qx = np.meshgrid(*(_folded(n) * (L / n) for n in (nz, ny, nx)), indexing="ij")
    q = np.sqrt(qx ** 2 + qy ** 2 + qz ** 2)
    b = np.rint(q).astype(int)
    b[0, 0, 0] = -1
    nbins = nbins or b.max() + 1
    keep = (b >= 0) & (b < nbins)
    cnt = np.bincount(b[keep], minlength=nbins)
    ref = np.bincount(b[keep], S[keep], minlength=nbins) / np.maximum(cnt, 1)
    got, n = g.structure_factor(nbins)
    # numpy's FFT and the device's differ by a few FP64 roundings of the largest mode
    assert n == 1 and np.abs(got - ref).max() < 1e-11 * S.max()
    assert np.array_equal(got == 0.0, cnt == 0)
    m = g.sk_moments()
    assert abs(m[0] / S.sum() - 1.0) < 1e-11
    assert abs(m[1] / (2 * np.pi / L * q * S).sum() - 1.0) < 1e-11
    axes, _ = g.structure_factor_axes()
    want = np.concatenate([S[0, 0, 1:nx // 2 + 1], S[0, 1:ny // 2 + 1, 0], S[1:nz // 2 + 1, 0, 0]])
    assert np.abs(axes - want).max() < 1e-11 * S.max()
    g.close()


@pytest.mark.parametrize("nx,ny,nz,precision", [(96, 4, 3, "fp32"), (160, 12, 5, "fp64"),
                                                (32, 20, 7, "fp32")])
def test_axis_profiles_of_other_sizes(nx, ny, nz, precision):
    """Sizes with a part of a 128-column chunk, fewer rows than warps and an odd
    number of planes."""
    from paper_2212_07848_gb300.lattice3 import Lattice3
    g = Lattice3(nx, ny, nz, -3.6, 0.9, 1e-5, precision=precision)
    g.init(LN2, 5, 0.01)
    g.sk_config(3, 3)
    g.step(3)
    rho = g.density()
    S = np.abs(np.fft.fftn(rho - rho.mean())) ** 2 / rho.size
    axes, n = g.structure_factor_axes()
    want = np.concatenate([S[0, 0, 1:nx // 2 + 1], S[0, 1:ny // 2 + 1, 0], S[1:nz // 2 + 1, 0, 0]])
    # FP32: the sampled density is rounded to FP32 (2^-24 of the deviations, on every site)
    tol = 1e-11 if precision == "fp64" else 2e-6
    assert n == 1 and np.abs(axes - want).max() < tol * want.max()
    g.close()
