"""Calls at the limits of what the entry points accept: several streams on one context,
inputs that are not finite, of extreme size or of very different size within a site, and
more right-hand sides than a workspace takes at a time."""
import ctypes
import threading

import numpy as np
import pytest

from lattice_inputs import eps_su3_field, haar_su3_field, gaussian_spinors
from oracle import dirac as od
from oracle import smear as osm
from tests._gpu import lattice, to_dev, to_np, torch

pytestmark = pytest.mark.gpu


def test_streams_share_a_context():
    """D and Gaussian smearing of one context on several streams without a synchronisation:
    created streams in turn, streams whose handle is that of a destroyed one with work still
    pending, and the per-thread stream, which is another one in each thread.  The workspace
    that they share is handed over in order: the results are those of single calls."""
    dims, n = (8, 8, 8, 8), 64
    with lattice(dims, haar_su3_field(dims, 41), 0.12) as (L, h):
        x = [to_dev(gaussian_spinors(dims, 1, 42 + k).reshape(1, -1, 4, 3)).repeat(n, 1, 1, 1) for k in range(2)]
        calls = [lambda q, o: L.lqcd_apply_dirac(h, q, o),
                 lambda q, o: L.lqcd_smear_gaussian(h, q, o, alpha=0.5, n_iter=3, normalise=True)]
        ref = [[torch.empty_like(q) for q in x] for _ in calls]
        for f, r in zip(calls, ref):
            for q, o in zip(x, r):
                f(q, o)
        torch.cuda.synchronize()

        def compare(out):
            torch.cuda.synchronize()
            for c, k, o in out:
                assert torch.equal(o, ref[c][k])

        streams = [torch.cuda.Stream(), torch.cuda.Stream()]
        out = []
        for k in range(8):
            with torch.cuda.stream(streams[k % 2]):
                out.append((k // 2 % 2, k % 2, torch.empty_like(x[0])))
                calls[out[-1][0]](x[k % 2], out[-1][2])
        compare(out)

        rt, out = torch.cuda.cudart(), [(0, k % 2, torch.empty_like(x[0])) for k in range(8)]
        torch.cuda.synchronize()
        for c, k, o in out:
            s = ctypes.c_void_p()
            assert int(rt.cudaStreamCreate(ctypes.addressof(s))) == 0
            with torch.cuda.stream(torch.cuda.ExternalStream(s.value)):
                calls[c](x[k], o)
            assert int(rt.cudaStreamDestroy(s.value)) == 0
        compare(out)

        lib, per_thread = L.load(), ctypes.c_void_p(2)  # cudaStreamPerThread
        out = [(0, k % 2, torch.empty_like(x[0])) for k in range(8)]
        torch.cuda.synchronize()
        for c, k, o in out:
            t = threading.Thread(target=lambda: lib.lqcd_apply_dirac(h, x[k].data_ptr(), o.data_ptr(), n, 0, per_thread))
            t.start()
            t.join()
        compare(out)


def test_captured_smearing_beside_ape():
    """Replays of a captured Gaussian smearing beside APE smearing on another stream: the two
    have no workspace in common."""
    dims, n = (8, 8, 8, 8), 32
    with lattice(dims, haar_su3_field(dims, 45), 0.12) as (L, h):
        src = to_dev(gaussian_spinors(dims, 1, 46).reshape(1, -1, 4, 3)).repeat(n, 1, 1, 1)
        ref, out = torch.empty_like(src), torch.empty_like(src)
        L.lqcd_smear_ape(h, 0.5, 2)
        L.lqcd_smear_gaussian(h, src, ref, alpha=0.5, n_iter=4, normalise=True)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            L.lqcd_smear_gaussian(h, src, out, alpha=0.5, n_iter=4, normalise=True)
        links = torch.empty(int(np.prod(dims)) * 36, dtype=torch.complex128, device="cuda")
        one, two = torch.cuda.Stream(), torch.cuda.Stream()
        for _ in range(4):
            out.zero_()
            torch.cuda.synchronize()
            with torch.cuda.stream(one):
                graph.replay()
            with torch.cuda.stream(two):
                L.lqcd_smear_ape(h, 0.5, 2, links)
            torch.cuda.synchronize()
            assert torch.equal(out, ref)


@pytest.mark.parametrize("dims,n", [((4, 4, 4, 4), 3), ((8, 8, 8, 16), 2)])
def test_largest_iteration_cap(dims, n):
    """max_iter = 2^31 - 1 ends like any other cap that is not reached: one cluster per pair
    (4^4) and the loop of launches, on the default and on a created stream."""
    cap = 2**31 - 1
    with lattice(dims, haar_su3_field(dims, 43), 0.12) as (L, h):
        b = to_dev(gaussian_spinors(dims, n, 44).reshape(n, -1, 4, 3))
        for prec in (L.LQCD_PREC_MIXED_FP16, L.LQCD_PREC_MIXED_BF16):
            res = []
            for stream in (None, torch.cuda.Stream()):
                for m in (20000, cap):
                    x = torch.empty_like(b)
                    with torch.cuda.stream(stream):
                        before = L.lqcd_launch_count()
                        rc, st = L.lqcd_solve_batch(h, b, x, L.solver_params(tol=1e-10, max_iter=m, precision=prec,
                                                                             timeout_ms=20000.0))
                    assert rc == 0
                    res.append((st, x, L.lqcd_launch_count() - before))
            for st, x, _ in res[1:]:
                assert st == res[0][0] and torch.equal(x, res[0][1])
            # no more kernels than with a cap that is out of reach as well
            assert res[3][2] <= res[2][2]


@pytest.mark.parametrize("mu", [0, 1, 2, 3])
def test_nan_link_stays_nan(mu):
    """A link with a NaN entry: D is NaN where the link enters and nowhere else, and no
    solve reports success."""
    dims = (4, 4, 4, 4)
    U = haar_su3_field(dims, 5)
    U[1, 2, 3, 0, mu, 1, 0] = np.nan
    psi = gaussian_spinors(dims, 2, 7)
    with np.errstate(invalid="ignore"):
        ref = np.stack([od.apply_D(U, 0.12, psi[k]) for k in range(2)])
    with lattice(dims, U, 0.12) as (L, h):
        x = to_dev(psi.reshape(2, -1, 4, 3))
        out = torch.empty_like(x)
        L.lqcd_apply_dirac(h, x, out)
        got = to_np(out, dims)
        assert np.array_equal(np.isnan(got), np.isnan(ref)) and np.isnan(ref).any()
        fine = ~np.isnan(ref)
        assert np.abs(got - ref)[fine].max() <= 1e-13
        for kw in (dict(precision=L.LQCD_PREC_FP64), dict(precision=L.LQCD_PREC_FP64, solver=L.LQCD_SOLVER_CG),
                   dict(precision=L.LQCD_PREC_MIXED_BF16), dict(precision=L.LQCD_PREC_MIXED_FP16)):
            rc, st = L.lqcd_solve_batch(h, x, out, L.solver_params(tol=1e-10, rhs_block=2, **kw))
            assert rc == L.LQCD_ERR_NONFINITE and all(s["status"] == rc for s in st), kw


def _singular_field(dims):
    """A field whose x link at one site is one, as are the links of its four spatial staples:
    U + alpha S = 0 there for alpha = -1/4, and its projection is NaN."""
    U = haar_su3_field(dims, 6)
    t, z, y, x = 1, 2, 1, 0
    one = np.eye(3)
    lx, ly, lz, _ = dims
    U[t, z, y, x, 0] = one
    for dz, dy in ((0, 1), (0, -1), (1, 0), (-1, 0)):
        zz, yy = (z + dz) % lz, (y + dy) % ly
        U[t, zz, yy, x, 0] = one
        mu = 1 if dy else 2
        for xx in (x, (x + 1) % lx):
            if dy + dz > 0:
                U[t, z, y, xx, mu] = one
            else:
                U[t, zz, yy, xx, mu] = one
    return U


@pytest.mark.parametrize("dims", [(4, 4, 4, 4), (6, 4, 4, 2)])
@pytest.mark.parametrize("steps", [1, 2, 3])
def test_nan_smeared_links_stay_nan(dims, steps):
    """APE links that are NaN: later APE steps and Gaussian smearing give NaN where, and only
    where, FP64 arithmetic gives it (a temporal link that is not SU(3) selects it; smearing
    does not read it)."""
    U = _singular_field(dims)
    q = gaussian_spinors(dims, 2, 8).reshape(2, -1, 4, 3)
    q[1] = 0.0
    q[1, 5, 2, 1] = 1.0  # most vectors zero
    res = []
    for general in (True, False):
        with lattice(dims, kappa=0.12) as (L, h):
            W = U.copy()
            if general:
                W[0, 0, 0, 0, 3] *= 2.0
            u = to_dev(W.reshape(-1))
            L.lqcd_set_gauge_general(h, u)
            links, src = torch.empty_like(u), to_dev(q)
            out = torch.empty_like(src)
            L.lqcd_smear_ape(h, -0.25, steps, links)
            L.lqcd_smear_gaussian(h, src, out, alpha=0.7, n_iter=2, ape_links=True, normalise=True)
            links = links.reshape(-1, 4, 9)[:, :3].contiguous()
            res.append((links.cpu().numpy(), out.cpu().numpy()))
    for a, b in zip(*res):
        assert np.isnan(a).any() and np.array_equal(np.isnan(a), np.isnan(b))
        fine = ~np.isnan(a)
        assert np.abs(a - b)[fine].max() <= 1e-9


@pytest.mark.parametrize("alpha", [1e6, 1e9, -1e9, 1e14, 1e40])
def test_ape_large_alpha(alpha):
    """The projection onto SU(3) of sums far above 1, whose determinants leave the range
    of FP32: the tolerance of the same field at alpha = 0.5."""
    dims = (4, 6, 4, 4)
    U = eps_su3_field(dims, 0.5, 3)
    V = int(np.prod(dims))
    with lattice(dims, U, 0.12) as (L, h):
        out = torch.empty(V * 36, dtype=torch.complex128, device="cuda")
        L.lqcd_smear_ape(h, alpha, 2, out)
        got = out.cpu().numpy().reshape(U.shape)
    assert np.max(np.abs(got - osm.ape_smear(U, alpha, 2))) < 1e-12


@pytest.mark.parametrize("prec", ["fp16", "bf16"])
@pytest.mark.parametrize("scale", [1e-100, 1e-30, 1e-18, 1e26, 1e100])
def test_mixed_solve_scaled_sources(prec, scale):
    """Sources of any overall size beside one of size 1: the FP64 residual meets the tolerance,
    and the reported one (FP32 components) is that residual."""
    dims, tol = (4, 4, 4, 8), 1e-10
    b = gaussian_spinors(dims, 3, 9).reshape(3, -1, 4, 3) * np.array([1.0, scale, -scale])[:, None, None, None]
    with lattice(dims, haar_su3_field(dims, 10), 0.13) as (L, h):
        p = L.LQCD_PREC_MIXED_FP16 if prec == "fp16" else L.LQCD_PREC_MIXED_BF16
        bd = to_dev(b)
        x, y = torch.empty_like(bd), torch.empty_like(bd)
        rc, st = L.lqcd_solve_batch(h, bd, x, L.solver_params(tol=tol, precision=p))
        L.lqcd_apply_dirac(h, x, y)
        s = torch.tensor([1.0, scale, scale], dtype=torch.float64, device="cuda").reshape(3, 1, 1, 1)
        rel = [float(torch.linalg.vector_norm(((y - bd) / s)[k]) / torch.linalg.vector_norm((bd / s)[k])) for k in range(3)]
        assert rc == 0
        for k in range(3):
            assert 0.0 < rel[k] <= 1.01 * tol
            assert abs(st[k]["true_rel_residual"] - rel[k]) <= 0.01 * rel[k]


ROWS = [(1.0, 1e-9, 1e-9, 1e-9), (1e-9, 1.0, 1e-9, 1e-9), (1e-12, 1e-12, 1.0, 1e-12), (1e-6, 1e-6, 1e-6, 1.0),
        (1.0, 0.0, 0.0, 0.0), (1.0, 0.03, 0.03, 0.03), (1.0, 0.2, 0.1, 0.06)]


def _row_max(psi):
    """Largest component that enters each row of D psi: the row's own, and those of the two
    rows that the neighbours' spin projection gives it."""
    m = np.maximum(np.abs(psi.real), np.abs(psi.imag)).max(axis=-1)  # [..., 4]
    def hop(ax, pair):
        v = np.maximum(m, m[..., pair])
        return np.maximum(np.roll(v, 1, ax), np.roll(v, -1, ax))
    out = m.copy()
    for mu in range(4):
        out = np.maximum(out, hop(m.ndim - 2 - mu, [3, 2, 1, 0] if mu < 2 else [2, 3, 0, 1]))
    return out


@pytest.mark.parametrize("rows", ROWS)
@pytest.mark.parametrize("share", [1.0, 0.03, 0.2])
@pytest.mark.parametrize("dims", [(4, 4, 4, 4), (6, 4, 2, 8)])
def test_dirac_rows_of_different_size(rows, share, dims):
    """Spin rows whose size differs by many orders within a site, on all sites or on some large
    ones, keep the precision of FP64 arithmetic row by row."""
    U = haar_su3_field(dims, 11)
    psi = gaussian_spinors(dims, 2, 12)
    some = np.random.default_rng(13).random(psi.shape[:-2]) < share
    psi *= np.where(some[..., None], 1e3 * np.array(rows), 1.0)[..., None]
    psi[1, 0] *= 1e-5
    with lattice(dims, U, 0.13) as (L, h):
        x = to_dev(psi.reshape(2, -1, 4, 3))
        out = torch.empty_like(x)
        for dag in (False, True):
            L.lqcd_apply_dirac(h, x, out, dagger=dag)
            ref = np.stack([(od.apply_Ddag if dag else od.apply_D)(U, 0.13, psi[k]) for k in range(2)])
            # up to 50 FP64 roundings of 2^-53 of that, here and in the oracle: below 1e-14
            err = np.abs(to_np(out, dims) - ref).max(-1)
            assert np.all(err <= 1e-14 * _row_max(psi))


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (8, 8, 8, 8)])
def test_first_dirac_allocates_nothing(dims):
    """The first D on a context enqueues work only: what it needs came with the gauge field."""
    with lattice(dims, haar_su3_field(dims, 13), 0.12) as (L, h):
        x = to_dev(gaussian_spinors(dims, 2, 14).reshape(2, -1, 4, 3))
        out = torch.empty_like(x)
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        L.lqcd_apply_dirac(h, x, out)
        torch.cuda.synchronize()
        assert torch.cuda.mem_get_info()[0] == free


def test_gradient_nan_coefficient():
    """A NaN coefficient of a time slice without sources is not lost: 0 NaN = NaN."""
    dims = (4, 4, 4, 4)
    src = np.zeros((2, 256, 4, 3), dtype=np.complex128)
    src[0, 3, 1, 2] = src[1, 9, 0, 0] = 1.0  # time slice 0
    with lattice(dims, haar_su3_field(dims, 15), 0.12) as (L, h):
        s = to_dev(src)
        sol = torch.empty_like(s)
        prm = L.solver_params(tol=1e-10, precision=L.LQCD_PREC_FP64, rhs_block=2)
        assert L.lqcd_solve_batch(h, s, sol, prm)[0] == 0
        coef = np.ones((4, 6), dtype=np.complex128)
        dU = torch.zeros(256 * 36, dtype=torch.complex128, device="cuda")
        assert L.lqcd_gradient(h, s, sol, coef, prm, dU=dU)[1] == 0
        coef[2, 3] = np.nan  # a slice without sources
        _, rc, st = L.lqcd_gradient(h, s, sol, coef, prm, dU=dU)
        assert rc == L.LQCD_ERR_NONFINITE and all(q["status"] == rc for q in st)


def test_several_chunks_of_right_hand_sides():
    """More right-hand sides than the limbs' workspaces take at a time (12 for D and the FP64
    solver, 3 for smearing on this lattice), with a ragged last chunk: the bits of calls with
    one right-hand side each."""
    dims = (12, 12, 12, 24)
    n, V = 14, int(np.prod(dims))
    U = eps_su3_field(dims, 0.35, 27)
    g = torch.Generator(device="cuda").manual_seed(28)
    x = torch.view_as_complex(torch.randn(n, V, 4, 3, 2, dtype=torch.float64, device="cuda", generator=g))
    x *= torch.logspace(-3, 3, n, dtype=torch.float64, device="cuda")[:, None, None, None]
    x[3] = 0.0
    x[3, 17, 2, 1] = 1.0  # converges at another iteration
    x[12] = 0.0
    with lattice(dims, U, 0.115) as (L, h):
        prm = L.solver_params(tol=1e-6, precision=L.LQCD_PREC_FP64, rhs_block=n)
        calls = [lambda q, o: L.lqcd_apply_dirac(h, q, o), lambda q, o: L.lqcd_apply_dirac(h, q, o, dagger=True),
                 lambda q, o: L.lqcd_smear_gaussian(h, q, o, alpha=0.7, n_iter=2),
                 lambda q, o: L.lqcd_solve_batch(h, q, o, prm)]
        for f in calls:
            whole, one = torch.empty_like(x), torch.empty_like(x)
            st = f(x, whole)
            sts = [f(x[k:k + 1], one[k:k + 1]) for k in range(n)]
            assert torch.equal(whole, one)
            if isinstance(st, tuple):
                assert st[0] == 0 and st[1] == [s[1][0] for s in sts]
                assert len({s["iterations"] for s in st[1]}) > 2
