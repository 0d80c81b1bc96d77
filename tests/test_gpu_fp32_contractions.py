"""The FP32 contractions (three BF16 parts per operand on the tensor cores) at the edges of their
tiles: transducer counts around one and two 128-wide tiles and 32-wide K chunks, odd node counts,
and the plain adjoint of a BF16 job; and the forward that
allocates nothing (its operands formed in the kernel, one CTA or a cluster per tile).

Reference: the sums in complex128 on the same FP32 tables. Tolerance: an operand carries about six
FP32 roundings (phase, sine, amplitude, products), two operands sqrt(12) 2^-24 = 2.1e-7 relative
for rounding errors of random sign; sums of up to ~100 terms in FP32 add the same again; 1e-6
leaves a factor of two and is below the 7.6e-6 that one lost low part (2^-17) would leave. The
preconditioned operands divide by dgamma, a difference of FP32 angles of size 2 pi / N with an
error of 2^-23: N 2^-24 on top.
"""
import ctypes
import math

import numpy as np
import pytest
import torch

from paper_2211_00316_gb300 import phantoms as P
from paper_2211_00316_gb300 import rbx

pytestmark = pytest.mark.gpu

F, C0 = 4e5, P.C_WATER


def tables(g, seed):
    rng = np.random.default_rng(seed)
    X, Y = (v[g.mask()] for v in g.coords())
    th = 2 * np.pi * np.arange(g.n_xducers) / g.n_xducers
    dx, dy = X - g.ring_radius * np.cos(th)[:, None], Y - g.ring_radius * np.sin(th)[:, None]
    s = np.hypot(dx, dy)
    T = (s / C0 * (1 + 0.01 * np.sin(40 * X + th[:, None]))).astype(np.float32)
    a = (s ** -0.5).astype(np.float32)
    a[rng.random(a.shape) < 0.02] = 0.0                       # uncovered entries
    gam = np.arctan2(dy, dx).astype(np.float32)
    K = rng.integers(0, 3, a.shape).astype(np.uint8)
    return T, a, gam, K


def rel(x, y):
    return float(np.linalg.norm(x - y) / np.linalg.norm(y))


@pytest.mark.parametrize("n", [3, 16, 17, 31, 32, 33, 127, 128, 129, 144, 257])
@pytest.mark.parametrize("nx,ny", [(24, 24), (41, 37)])
def test_against_complex128(n, nx, ny):
    g = P.Geometry(nx=nx, ny=ny, dx=1e-3, n_xducers=n, ring_radius=(min(nx, ny) - 1) * 0.5e-3 - 1.5e-3)
    T, a, gam, K = tables(g, n)
    rng = np.random.default_rng(7)
    cov = a > 0
    w = 2 * math.pi * F
    Cg = (8 * math.pi * w / C0) ** -0.5
    G = np.where(cov, Cg * a.astype(np.float64) * np.exp(2j * np.pi * (F * T.astype(np.float64) - K / 4 + 0.125)), 0)
    gd = gam.astype(np.float64)
    d = np.roll(gd, -1, 0) - np.roll(gd, 1, 0)
    d = 0.5 * np.abs(np.mod(d + np.pi, 2 * np.pi) - np.pi)
    d[~(np.roll(cov, -1, 0) & np.roll(cov, 1, 0))] = 0
    U = np.where(cov, d / np.where(cov, G, 1), 0)
    kap = np.exp(1j * gd)
    dm = (1e-9 * rng.standard_normal((ny, nx))).astype(np.float32)
    v = w * w * g.dx ** 2 * dm[g.mask()].astype(np.float64)
    R = (rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))).astype(np.complex64)
    Rs = 0.5 * (R + R.T).astype(np.complex128)
    want = {"forward": (G * v) @ G.T, "plain": w * w * g.dx ** 2 * (G.conj() * (Rs @ G.conj())).sum(0),
            "pre": 2 * ((U * (Rs @ U)).sum(0) - (kap * U * (Rs @ (kap.conj() * U))).sum(0))}
    dev = [torch.tensor(t, device="cuda") for t in (T, a, gam, K)]
    exits = torch.zeros((n, n - 1, 4), device="cuda")
    Rd, dmd = torch.tensor(R, device="cuda"), torch.tensor(dm, device="cuda")
    D = torch.empty((n, n), dtype=torch.complex64, device="cuda")
    vd, err = torch.tensor(v.astype(np.float32), device="cuda"), ctypes.create_string_buffer(256)
    assert rbx.load().rbx_forward_noalloc(dev[0].data_ptr(), dev[1].data_ptr(), dev[3].data_ptr(), vd.data_ptr(), n, a.shape[1],
                                          F, C0, D.data_ptr(), torch.cuda.current_stream().cuda_stream or None, err, 256) == 0
    assert rel(D.cpu().numpy(), want["forward"]) <= 1e-6
    for prec in (rbx.RBX_FP32, rbx.RBX_BF16):
        job = rbx.Job()
        job.set_geometry(g, precision=prec)
        job.set_tables(*dev, exits)
        assert rel(job.adjoint(F, Rd, False).cpu().numpy(), want["plain"]) <= 1e-6
        if prec == rbx.RBX_FP32:
            assert rel(job.forward(F, dmd).cpu().numpy(), want["forward"]) <= 1e-6
            assert rel(job.adjoint(F, Rd, True).cpu().numpy(), want["pre"]) <= 1e-6 + n * 2.0 ** -24
        job.close()


def test_more_than_65535_node_tiles():
    """Tables of equal entries, 8.5 million nodes: every node's plain adjoint is the first one's,
    whichever tile it falls in; so is the preconditioned one's (its two transducer neighbours differ by the
    same angle)."""
    n, m = 3, 3320
    g = P.Geometry(nx=m, ny=m, dx=1e-4, n_xducers=n, ring_radius=(m - 1) * 0.5e-4 - 3e-4, mask_frac=0.999,
                   ds_frac=4.0)
    x = int(g.mask().sum())
    assert x > 65535 * 128
    dev = [torch.full((n, x), val, dtype=dt, device="cuda")
           for val, dt in ((1e-4, torch.float32), (3.0, torch.float32), (0.0, torch.float32), (1, torch.uint8))]
    dev[2] += torch.tensor([0.3, 2.4, -1.9], device="cuda")[:, None]
    R = torch.tensor(np.random.default_rng(1).standard_normal((n, n)), device="cuda").to(torch.complex64)
    job = rbx.Job()
    job.set_geometry(g, precision=rbx.RBX_FP32)
    job.set_tables(*dev, torch.zeros((n, n - 1, 4), device="cuda"))
    for pre in (False, True):
        out = job.adjoint(F, R, pre)
        assert bool(torch.isfinite(torch.view_as_real(out)).all()) and float(out[0].abs()) > 0
        assert bool((out == out[0]).all())
    job.close()


# (12, 2), (10, 4), (25, 2), (3, 4), (2, 4), (1, 4): partial sums and CTAs of a cluster per tile pair, by
# noalloc_shape on 152 SMs; all with a ragged last tile, with node counts that are no multiple of 4 or
# of a chunk, and all but the fifth with CTAs that get fewer chunks or none
@pytest.mark.parametrize("n,x", [(257, 2337), (250, 4001), (150, 4827), (500, 1203), (600, 1251), (1000, 1299)])
def test_noalloc_clusters(n, x):
    rng = np.random.default_rng(n)
    T = rng.uniform(1e-6, 1e-4, (n, x)).astype(np.float32)
    a = rng.uniform(2.0, 30.0, (n, x)).astype(np.float32)
    a[rng.random(a.shape) < 0.02] = 0.0
    K = rng.integers(0, 3, a.shape).astype(np.uint8)
    v = rng.standard_normal(x).astype(np.float32)
    G = (8 * math.pi * 2 * math.pi * F / C0) ** -0.5 * a.astype(np.float64) * np.exp(
        2j * np.pi * (F * T.astype(np.float64) - K / 4 + 0.125))
    dev = [torch.tensor(t, device="cuda") for t in (T, a, K, v)]
    D = torch.empty((n, n), dtype=torch.complex64, device="cuda")
    err = ctypes.create_string_buffer(256)
    assert rbx.load().rbx_forward_noalloc(*[t.data_ptr() for t in dev], n, x, F, C0, D.data_ptr(),
                                          torch.cuda.current_stream().cuda_stream or None, err, 256) == 0
    D = D.cpu().numpy()
    assert rel(D, (G * v.astype(np.float64)) @ G.T) <= 1e-6
    assert np.array_equal(D, D.T)


@pytest.mark.parametrize("n", [3, 16, 17, 31, 32, 33, 64, 65, 95, 97, 127, 128, 129, 144, 257])
@pytest.mark.parametrize("nx,ny", [(24, 24), (41, 37)])
def test_split_against_complex128(n, nx, ny):
    """Split BF16 at the same edges, and with fewer chunks than stages. Two parts leave 2^-18 of an operand, and lo lo
    2^-18 of a product: 3 x 2^-18 = 1.2e-5 of every product; 2e-5 leaves the FP32 roundings room, the
    preconditioned operands' dgamma on top."""
    g = P.Geometry(nx=nx, ny=ny, dx=1e-3, n_xducers=n, ring_radius=(min(nx, ny) - 1) * 0.5e-3 - 1.5e-3)
    T, a, gam, K = tables(g, n)
    rng = np.random.default_rng(8)
    cov = a > 0
    w = 2 * math.pi * F
    G = np.where(cov, (8 * math.pi * w / C0) ** -0.5 * a.astype(np.float64) *
                 np.exp(2j * np.pi * (F * T.astype(np.float64) - K / 4 + 0.125)), 0)
    gd = gam.astype(np.float64)
    d = np.roll(gd, -1, 0) - np.roll(gd, 1, 0)
    d = 0.5 * np.abs(np.mod(d + np.pi, 2 * np.pi) - np.pi)
    d[~(np.roll(cov, -1, 0) & np.roll(cov, 1, 0))] = 0
    U = np.where(cov, d / np.where(cov, G, 1), 0)
    kap = np.exp(1j * gd)
    dm = (1e-9 * rng.standard_normal((ny, nx))).astype(np.float32)
    v = w * w * g.dx ** 2 * dm[g.mask()].astype(np.float64)
    R = (rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))).astype(np.complex64)
    Rs = 0.5 * (R + R.T).astype(np.complex128)
    job = rbx.Job()
    job.set_geometry(g, precision=rbx.RBX_BF16X3)
    job.set_tables(*[torch.tensor(t, device="cuda") for t in (T, a, gam, K)], torch.zeros((n, n - 1, 4), device="cuda"))
    Rd = torch.tensor(R, device="cuda")
    assert rel(job.forward(F, torch.tensor(dm, device="cuda")).cpu().numpy(), (G * v) @ G.T) <= 2e-5
    assert rel(job.adjoint(F, Rd, True).cpu().numpy(),
               2 * ((U * (Rs @ U)).sum(0) - (kap * U * (Rs @ (kap.conj() * U))).sum(0))) <= 2e-5 + n * 2.0 ** -24
    assert rel(job.adjoint(F, Rd, False).cpu().numpy(), w * w * g.dx ** 2 * (G.conj() * (Rs @ G.conj())).sum(0)) <= 1e-6
    job.close()
