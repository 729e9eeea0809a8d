"""GPU parity of the FP64 entry points whose SU(3) products run on the integer
units: D and its adjoint and Gaussian smearing, on fields whose magnitude varies
strongly from site to site, at the ends of the FP64 range and with non-finite
entries (where a site is evaluated in FP64 instead), one to three right-hand sides."""
import numpy as np
import pytest

from lattice_inputs import haar_su3_field, gaussian_spinors
from oracle import dirac as od
from oracle.smear import gaussian_smear
from tests._gpu import lattice, to_dev, to_np, torch

pytestmark = pytest.mark.gpu

DIMS = [(4, 4, 4, 4), (6, 4, 2, 8), (2, 2, 2, 2)]


def _field(dims, n, seed, spread, scale):
    psi = gaussian_spinors(dims, n, seed)
    rng = np.random.default_rng(seed + 1)
    mag = 10.0 ** rng.uniform(-spread, spread, psi.shape[:-2])
    psi *= mag[..., None, None] * scale
    psi[:, 0, 0, 0] = 0.0  # whole sites of zeros among the neighbours
    return psi


def _local_max(psi):
    """Largest component of each site's stencil (the site and its eight neighbours)."""
    m = np.maximum(np.abs(psi.real), np.abs(psi.imag)).max(axis=(-1, -2))
    out = m.copy()
    for ax in range(1, 5):
        out = np.maximum(out, np.maximum(np.roll(m, 1, ax), np.roll(m, -1, ax)))
    return out[..., None, None]


# a few units of 2^-56 of the stencil's largest component per direction on the
# device, and up to 50 FP64 roundings of 2^-53 of it in the oracle: below 1e-14
TOL = 1e-14


@pytest.mark.parametrize("dims", DIMS)
@pytest.mark.parametrize("n", [1, 2, 3])
@pytest.mark.parametrize("spread,scale", [(0, 1.0), (12, 1.0), (3, 1e-285), (3, 1e-305), (3, 1e270), (3, 1e299)])
def test_dirac_over_magnitudes(dims, n, spread, scale):
    U = haar_su3_field(dims, 5)
    psi = _field(dims, n, 11, spread, scale)
    V = int(np.prod(dims))
    with lattice(dims, U, 0.13) as (L, h):
        x = to_dev(psi.reshape(n, V, 4, 3))
        out = torch.empty_like(x)
        for dag in (False, True):
            L.lqcd_apply_dirac(h, x, out, dagger=dag)
            ref = np.stack([(od.apply_Ddag if dag else od.apply_D)(U, 0.13, psi[k]) for k in range(n)])
            assert np.all(np.abs(to_np(out, dims) - ref) <= TOL * _local_max(psi) + 1e-320)


@pytest.mark.parametrize("n", [1, 2])
def test_dirac_non_finite_entries_stay_local(n):
    dims = (4, 4, 4, 4)
    U = haar_su3_field(dims, 6)
    psi = _field(dims, n, 13, 0, 1.0)
    psi[0, 1, 2, 3, 0, 1, 2] = np.inf
    psi[n - 1, 2, 2, 1, 3, 0, 0] = np.nan
    hit = ~np.isfinite(_local_max(np.where(np.isfinite(psi), psi, np.inf)))
    with np.errstate(invalid="ignore"):
        ref = np.stack([od.apply_D(U, 0.13, psi[k]) for k in range(n)])
    with lattice(dims, U, 0.13) as (L, h):
        x = to_dev(psi.reshape(n, -1, 4, 3))
        out = torch.empty_like(x)
        L.lqcd_apply_dirac(h, x, out)
        got = to_np(out, dims)
    clean = np.broadcast_to(~hit, ref.shape)
    assert np.array_equal(np.isfinite(got), np.isfinite(ref))
    fine = clean & np.isfinite(ref)
    assert np.all(np.abs(got - ref)[fine] <= TOL * 10)


@pytest.mark.parametrize("dims", DIMS)
@pytest.mark.parametrize("n", [1, 2, 3])
@pytest.mark.parametrize("spread,scale", [(0, 1.0), (12, 1.0), (2, 1e-305), (2, 1e290)])
def test_gaussian_step_over_magnitudes(dims, n, spread, scale):
    U = haar_su3_field(dims, 7)
    q = _field(dims, n, 17, spread, scale)
    V = int(np.prod(dims))
    with lattice(dims, U, 0.13) as (L, h):
        x = to_dev(q.reshape(n, V, 4, 3))
        out = torch.empty_like(x)
        L.lqcd_smear_gaussian(h, x, out, alpha=0.7, n_iter=1)
        ref = gaussian_smear(U, q, 0.7, 1)
        assert np.all(np.abs(to_np(out, dims) - ref) <= TOL * _local_max(q) + 1e-320)


@pytest.mark.parametrize("dims", DIMS)
@pytest.mark.parametrize("alpha", [4.0, -0.3, 0.0, 1e-310])
def test_gaussian_steps_over_coefficients(dims, alpha):
    """Five normalised steps: zero and negative alpha, and a subnormal one, which has no
    integer form and takes FP64 arithmetic."""
    U = haar_su3_field(dims, 8)
    q = _field(dims, 2, 19, 0, 1.0)
    q[1] = 0.0
    q[1, 1, 1, 1, 1, 2, 0] = 1.0  # a point source: most neighbours are zero
    scale = 1.0 / (1.0 + 6.0 * alpha)
    with lattice(dims, U, 0.13) as (L, h):
        x = to_dev(q.reshape(2, -1, 4, 3))
        out = torch.empty_like(x)
        L.lqcd_smear_gaussian(h, x, out, alpha=alpha, n_iter=5, normalise=True)
        got = to_np(out, dims)
    ref = gaussian_smear(U, q, alpha, 5) * scale**5
    # a few FP64 roundings of the largest intermediate value per step, in the oracle and here
    assert np.all(np.abs(got - ref) <= 5 * TOL * max(1.0, (1.0 + 6.0 * abs(alpha)) * abs(scale)) ** 5 * np.abs(q).max())


@pytest.mark.parametrize("alpha", [4.0, 0.6])
def test_gaussian_steps_keep_more_than_fp64(alpha):
    """25 normalised steps against extended precision.  A step rounds by at most 2^-55 of
    the vector (58-bit limbs, sums of six products) and the result by 2^-53 once: 8.1e-16
    in the 2-norm even if all errors line up.  The rounding of 1 / (1 + 6 alpha) to FP64
    alone would give up to 25 * 2^-53 = 2.8e-15."""
    dims = (4, 4, 4, 4)
    U = haar_su3_field(dims, 9)
    q = gaussian_spinors(dims, 1, 23)
    with lattice(dims, U, 0.13) as (L, h):
        x = to_dev(q.reshape(1, -1, 4, 3))
        out = torch.empty_like(x)
        L.lqcd_smear_gaussian(h, x, out, alpha=alpha, n_iter=25, normalise=True)
        got = to_np(out, dims)
    Q = np.clongdouble
    u, ref, a = U.astype(Q), q[0].astype(Q), np.longdouble(alpha)
    for _ in range(25):
        hq = 0
        for mu in range(3):
            um = u[..., mu, :, :]
            fwd = (um[..., None, :, :] * np.roll(ref, -1, 3 - mu)[..., None, :]).sum(-1)
            bwd = (np.conj(np.swapaxes(um, -1, -2))[..., None, :, :] * ref[..., None, :]).sum(-1)
            hq = hq + fwd + np.roll(bwd, 1, 3 - mu)
        ref = (ref + a * hq) / (1 + 6 * a)
    d = got[0].astype(Q) - ref
    assert float(np.sqrt((np.abs(d) ** 2).sum() / (np.abs(ref) ** 2).sum())) < 8.1e-16
