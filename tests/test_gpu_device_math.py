"""The integrator's float64 device functions against what they stand for: the tabulated normals against Box-Muller by the
library functions (every 21-bit field, bit for bit), the FENE floor taken by the bits of s against the
comparison it replaces, the reciprocal of the pair forces against the division."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_2206_05851_gb300 import bdra
from paper_2206_05851_gb300 import build as B
from paper_2206_05851_gb300 import inputs as I

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def dev():
    import torch
    lib = B.build()
    torch.cuda.init()
    out = os.path.join(HERE, "_build", f"device_checks_{os.getpid()}.so")
    os.makedirs(os.path.dirname(out), exist_ok=True)
    r = subprocess.run([B._nvcc(), *B.ARCH, *B.COMMON, "-fmad=false", "-I", B.CSRC, "-shared", "-o", out,
                        os.path.join(HERE, "device_checks.cu"), lib, "-Xlinker", f"-rpath={os.path.dirname(lib)}"],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    yield ctypes.CDLL(out)
    os.unlink(out)


def _p(a):
    return a.ctypes.data_as(ctypes.c_void_p)


def test_tabulated_normals_are_the_library_functions_bits(dev):
    bad = ctypes.c_ulonglong(1)
    assert dev.check_noise(ctypes.byref(bad)) == 0
    assert bad.value == 0


def test_noise_diagnostic_shares_the_tables_and_gives_them_back():
    """bd_philox_normals draws as the integrator does, from the tables: the same values with and without a float64 context
    that holds them, which reads them after a call, and no memory kept when the last user is gone."""
    import torch
    ctr = np.random.default_rng(1).integers(0, 2 ** 24, size=(5000, 4)).astype(np.uint32)
    out = [np.zeros((5000, 3)) for _ in range(3)]
    torch.cuda.synchronize()
    bdra.bd_philox_normals(5, ctr, bdra.BD_PREC_FP64, out[0])
    free = torch.cuda.mem_get_info()[0]
    bdra.bd_philox_normals(5, ctr, bdra.BD_PREC_FP64, out[1])
    assert torch.cuda.mem_get_info()[0] == free
    chains = [I.Chain(n_beads=12, n_replicas=3, spring=I.SPRING_FENE, flow=I.FLOW_SHEAR, b=30.0, rate=0.1)]
    wl = I.custom(chains, 1e-3, 5, 10)
    runs = []
    for ask in (False, True):
        ctx = bdra.Context(chains, wl.dt, 5, 1, I.initial_positions(wl, seed=3), precision=bdra.BD_PREC_FP64, max_windows=2,
                           stream=torch.cuda.current_stream().cuda_stream)
        ctx.step(5)
        if ask:
            bdra.bd_philox_normals(5, ctr, bdra.BD_PREC_FP64, out[2])
        ctx.step(5)
        runs.append(ctx.positions(True))
        ctx.close()
    np.testing.assert_array_equal(runs[0], runs[1])
    np.testing.assert_array_equal(out[0], out[1])
    np.testing.assert_array_equal(out[0], out[2])


@pytest.mark.parametrize("Hinvb", [1.0, 0.25, 0.0])
def test_fene_floor_by_bits_is_the_comparison(dev, Hinvb):
    """s < smin is floored and counted; a NaN s (of either sign) takes smin, as fmax does, and is not counted. The bond
    lengths are dyadic, so that s is exact and the host's expressions give the same bits."""
    H, smin, nan, inf = 1.5, 2.0 ** -9, np.nan, np.inf
    u = np.array([[62, 12, 10], [63, 12, 10], [62, 12, 9], [64, 0, 0], [128, 0, 0], [0, 0, 0], [1, 0, 0], [124, 24, 20],
                  [126, 24, 20]]) / 64.0           # first: s = smin exactly with Hinvb = 1; [124, 24, 20] with 1/4
    odd = np.array([[nan, 0, 0], [-nan, 0, 0], [0, nan, 1], [inf, 0, 0], [-inf, 1, 0], [inf, nan, 0], [1e200, 0, 0]])
    r = np.random.default_rng(4)
    q = np.ascontiguousarray(np.concatenate([u, odd, r.integers(-160, 160, size=(1000, 3)) / 128.0]))
    c, fl = np.zeros(len(q)), np.zeros(len(q), dtype=np.int32)
    assert dev.check_spring(ctypes.c_int64(len(q)), _p(q), ctypes.c_double(H), ctypes.c_double(Hinvb), ctypes.c_double(smin),
                            _p(c), _p(fl)) == 0
    with np.errstate(all="ignore"):
        s = 1.0 - Hinvb * (q * q).sum(axis=1)
        want = H / np.fmax(s, smin)
    np.testing.assert_array_equal(fl, (s < smin).astype(np.int32))
    np.testing.assert_array_equal(c, want)
    assert np.isnan(s).any() and (fl[:len(u)].any() or Hinvb == 0.0)


@pytest.mark.parametrize("prec", [bdra.BD_PREC_FP64, bdra.BD_PREC_FP32])
def test_bonds_that_are_not_numbers_count_no_overextension(prec):
    """A NaN bead in a FENE chain; a Hooke chain whose squared bond overflows (s = 1 - 0 inf); a sound chain beside them."""
    import torch
    chains = [I.Chain(n_beads=12, n_replicas=3, spring=k, flow=I.FLOW_SHEAR, b=30.0, rate=0.1)
              for k in (I.SPRING_FENE, I.SPRING_HOOKE, I.SPRING_FENE)]
    pos = I.initial_positions(I.custom(chains, 1e-4, 5, 10), seed=3)
    pos[4], pos[16, 1] = np.nan, 1e200
    ctx = bdra.Context(chains, 1e-4, 5, 1, pos, precision=prec, max_windows=2, stream=torch.cuda.current_stream().cuda_stream)
    ctx.step(10)
    n, end = ctx.info().overextensions, ctx.positions()
    ctx.close()
    assert np.isnan(end[:12]).any() and np.isfinite(end[24:]).all()
    assert n == 0


def test_reciprocal_of_pair_forces(dev):
    """Within one unit in the last place of 1 / x: two Newton-Raphson steps square a relative error of 2^-20 twice, so the last
    multiply-add rounds a value within 2^-53 (2^-26) of the reciprocal, and 1 / x is its correctly rounded neighbour. Zero and
    infinite squared distances (coincident and overflowing beads) as the division."""
    r = np.random.default_rng(8)
    rnd = np.ldexp(r.uniform(1.0, 2.0, 400_000), r.integers(-1020, 1020, 400_000))
    two = np.ldexp(1.0, np.arange(-1020, 1020))
    far = (1e12 * np.arange(1, 514)) ** 2
    x = np.concatenate([rnd, two, np.nextafter(two, 0.0), np.nextafter(two, np.inf), far, [1e30, 1e36]])
    x = np.ascontiguousarray(np.concatenate([x, -x[:1000], [0.0, -0.0, np.inf, -np.inf]]))
    y = np.zeros(len(x))
    assert dev.check_recip(ctypes.c_int64(len(x)), _p(x), _p(y)) == 0
    with np.errstate(divide="ignore"):
        want = 1.0 / x
    np.testing.assert_array_equal(y[-4:], want[-4:])
    ulps = np.abs(y[:-4].view(np.int64) - want[:-4].view(np.int64))
    assert ulps.max() <= 1
