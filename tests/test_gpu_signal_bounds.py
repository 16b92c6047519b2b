"""The signal speeds of FP64 states, of which only the largest counts: each
cell's is bounded in FP32 and evaluated in FP64 where it may be the largest.
Patches of two kinds of cell, a hot gas at rest and a dense stream whose
speeds differ by a part in 1e5 to a fifth, in units and at ratios of specific
heats where FP32 is short of range or of digits: the speeds are the oracle's,
bit for bit."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1705_10774_gb300 import build as B
from paper_1705_10774_gb300 import ics
from paper_1705_10774_gb300.dispatch import Dispatch
from oracle import Oracle

DELTAS = [s * d for d in (1e-5, 3e-5, 1e-4, 3e-4, 1e-3, 3e-3, 1e-2, 3e-2, 0.1, 0.2) for s in (1, -1)]


def _sum(gamma, rho, p, b, v):
    a2, b2 = gamma * p / rho, [x * x / rho for x in b]
    s = a2 + sum(b2)
    return sum(map(abs, v)) + sum(np.sqrt(0.5 * (s + np.sqrt((a2 + sum(b2) - 2 * x) ** 2 + 4 * x * (sum(b2) - x)))) for x in b2)


def _two_kinds(gamma, scale, b):
    """A patch per entry of DELTAS: rows of alternating cells, the stream's
    speed 1 + delta times the hot gas's.  Pressure and field are uniform."""
    lay = ics.cartesian((len(DELTAS), 1, 1), (32, 4, 4))
    X, Y, Z = lay.base_cells
    stream = np.broadcast_to(np.arange(X) % 2 == 1, (Z, Y, X))
    hot, cold = _sum(gamma, 1.0, 1.0, b, (0,)), _sum(gamma, 100.0, 1.0, b, (0,))
    v = np.zeros((3, Z, Y, X))
    v[1] = np.where(stream, (1 + np.repeat(DELTAS, 32)) * hot - cold, 0.0) * scale
    one = np.ones((Z, Y, X))
    f = ics.Fields(rho=np.where(stream, 100.0, 1.0), v=v, p=one * scale ** 2, bx=one * b[0] * scale,
                   by=one * b[1] * scale, bz=one * b[2] * scale, gamma=gamma)
    return lay, ics.to_patches(lay, f)


def _same_speeds(lay, state, gamma, **kw):
    kw.update(gamma=gamma, cfl=0.2, base_cells=lay.base_cells, box_len=lay.box_len, time_mode=0)
    o = Oracle(lay.n, lay.lo, **kw)
    o.set_state(*state)
    loaded = o.get_times()[2].copy()
    o.advance(max_sweeps=2)
    for precision in (0, 2):
        g = Dispatch(lay.n, lay.lo, precision=precision, **kw)
        g.set_state(*state)
        assert np.array_equal(g.pack(np.arange(lay.npatch), device=False)[1][:, 2], loaded)
        g.advance(max_sweeps=2)
        speed, ref = g.pack(np.arange(lay.npatch), device=False)[1][:, 2], o.get_times()[2]
        if precision == 0:
            assert np.array_equal(speed, ref)
            assert all(np.array_equal(a, b) for a, b in zip(g.get_state(), o.get_state()))
        else:  # the tolerance of the parity tests; cancellation in p at most p / E of the digits
            assert np.max(np.abs(speed / ref - 1)) <= 1e-11 / (gamma - 1)
        g.close()


@pytest.mark.parametrize("gamma", [1.0001, 1.00001, 1.000001])
def test_nearly_isothermal_gas(gamma):
    """gamma - 1 taken from gamma in FP32 is off by up to a twentieth."""
    lay, state = _two_kinds(gamma, 1.0, (0.0, 0.0, 0.0))
    _same_speeds(lay, state, gamma)


@pytest.mark.parametrize("b", [0.0, 0.8])
@pytest.mark.parametrize("scale", [1e-9, 1e9, 4e9, 1e10, 1e12, 1e15])
def test_units_of_large_and_small_velocities(scale, b):
    """The fourth power of a speed leaves FP32's range at 4e9: a magnetised
    gas's speed came out up to 28 % low, and finite."""
    lay, state = _two_kinds(5.0 / 3.0, scale, (b, b, b))
    _same_speeds(lay, state, 5.0 / 3.0)


# ------------------------------------------------------- the bounds themselves

SRC = r"""
#include "dsp_fast.cuh"
__global__ void kernel(const double *in, int n, double gamma, float *above, float *below) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  double U[5];
  for (int k = 0; k < 5; k++) U[k] = in[(long long)k * n + i];
  const double *f = in + 5ll * n + i;
  dsp::fast::signal_bounds(U, f[0], f[n], f[2ll * n], f[3ll * n], f[4ll * n], f[5ll * n], (float)gamma, (float)(gamma - 1.0),
                           above[i], below[i]);
}
extern "C" int run(const double *in, int n, double gamma, float *above, float *below) {
  kernel<<<(n + 255) / 256, 256>>>(in, n, gamma, above, below);
  return (int)cudaDeviceSynchronize();
}
"""
GAMMA = 5.0 / 3.0
N = 1 << 18


@pytest.fixture(scope="module")
def bounds(tmp_path_factory):
    """(above, below) of FP64 cells: signal_bounds, compiled by itself."""
    d = tmp_path_factory.mktemp("bounds")
    (d / "b.cu").write_text(SRC)
    subprocess.check_call([B._nvcc(), "-O3", "-std=c++17", *B.ARCH, "-fmad=false", "-shared", "-Xcompiler", "-fPIC", "-I", B.CSRC,
                           "-I", os.path.join(B.ROOT, "include"), str(d / "b.cu"), "-o", str(d / "b.so")])
    lib = ctypes.CDLL(str(d / "b.so"))

    def call(U, faces, gamma):
        a = torch.from_numpy(np.stack([*U, *faces])).cuda()
        out = torch.empty((2, a.shape[1]), dtype=torch.float32, device="cuda")
        torch.cuda.synchronize()
        P = ctypes.c_void_p
        assert lib.run(P(a.data_ptr()), a.shape[1], ctypes.c_double(gamma), P(out[0].data_ptr()), P(out[1].data_ptr())) == 0
        return out.cpu().numpy().astype(np.float64)

    return call


def _cells(rho, v, p, faces, gamma=GAMMA):
    b2 = sum((0.5 * (faces[2 * k] + faces[2 * k + 1])) ** 2 for k in range(3))
    return [rho, *(rho * x for x in v), p / (gamma - 1) + 0.5 * rho * sum(x * x for x in v) + 0.5 * b2], faces


def _true(U, faces, gamma=GAMMA):
    """The speeds of the same cells, p from the conserved values as the kernels take it."""
    v, b = [m / U[0] for m in U[1:4]], [0.5 * (faces[2 * k] + faces[2 * k + 1]) for k in range(3)]
    p = (gamma - 1) * (U[4] - 0.5 * U[0] * sum(x * x for x in v) - 0.5 * sum(x * x for x in b))
    return _sum(gamma, U[0], np.maximum(p, 1e-20 * U[0]), b, v)


def _hold(bounds, U, faces, gamma=GAMMA, some=0.5):
    above, below = bounds(U, faces, gamma)
    t = _true(U, faces, gamma)
    assert np.all(above >= t) and np.all(~(below > t))
    # and they are of use: within 1e-4 wherever the pressure is not lost in E
    tight = (above <= 1.0001 * t) & (below >= 0.999 * t)
    assert tight.mean() >= some


def _draw(seed):
    r = np.random.default_rng(seed)
    return r, np.exp(r.normal(size=N)), r.normal(size=(3, N)), np.exp(2 * r.normal(size=N)), r.normal(size=(3, N))


@pytest.mark.parametrize("kind", ["sound speed near the Alfven speed", "nearly along an axis"])
def test_bounds_hold_where_the_discriminant_cancels(bounds, kind):
    """s^2 - 4 a^2 b^2 loses half its digits for a field along an axis with
    equal sound and Alfven speeds: the fast speed was off by 3e-4."""
    r, rho, v, p, _ = _draw(1)
    near = np.abs(1 + np.exp(r.uniform(np.log(1e-9), 0, N)) * r.choice([-1, 1], N))
    along = near * np.sqrt(GAMMA * p)
    across = 0 * p if kind.startswith("sound") else np.sqrt(p) * np.exp(r.uniform(np.log(1e-9), np.log(1e-2), N))
    for axis in range(3):
        f = [0 * p] * 6
        f[2 * axis] = f[2 * axis + 1] = along
        f[(2 * axis + 2) % 6] = f[(2 * axis + 3) % 6] = across
        _hold(bounds, *_cells(rho, 0 * v, p, f))


@pytest.mark.parametrize("gamma", [5.0 / 3.0, 1.4, 1.0001, 1.000001])
@pytest.mark.parametrize("scale", [1e-7, 1e-3, 1.0, 1e5, 1e10, 1e13])
def test_bounds_hold_across_units(bounds, scale, gamma):
    _, rho, v, p, b = _draw(2)
    _hold(bounds, *_cells(rho, scale * v, scale ** 2 * p, [scale * x for x in b for _ in range(2)], gamma), gamma)
    for r in (1e-24, 1e-12, 1e12, 1e24):  # densities
        _hold(bounds, *_cells(r * rho, 1e2 * v, 1e4 * r * p, [1e2 * np.sqrt(r) * x for x in b for _ in range(2)], gamma), gamma)


def test_bounds_hold_between_opposite_faces(bounds):
    """A cell's field is the mean of its faces; the difference of two FP32
    faces of opposite sign has the faces' error, not its own."""
    r, rho, v, p, b = _draw(3)
    f = []
    for x in b:
        big = np.exp(r.uniform(0, np.log(1e9), N))
        f += [x - big, x + big]
    _hold(bounds, *_cells(rho, v, p, f))


def test_ambipolar_limit_beyond_fp32():
    """The step limit of the ambipolar term as a speed, B^2 / rho times a
    coefficient: B^2 times it overflows FP32 in the dense rows, whose limit is a
    tenth of the thin ones'."""
    lay = ics.cartesian((2, 1, 1), (16, 8, 4))
    X, Y, Z = lay.base_cells
    odd = np.broadcast_to(np.arange(Y)[:, None] % 2 == 1, (Z, Y, X))
    one = np.ones((Z, Y, X))
    f = ics.Fields(rho=np.where(odd, 1e24, 1e22), v=np.zeros((3, Z, Y, X)), p=1e20 * one, bx=np.where(odd, 3e9, 1e9),
                   by=0 * one, bz=0 * one, gamma=GAMMA)
    state = ics.to_patches(lay, f)
    kw = dict(gamma=GAMMA, cfl=0.4, base_cells=lay.base_cells, box_len=lay.box_len, time_mode=0, rho_i=1.0,
              gamma_ad=0.4 / (0.1 * 1e20 * lay.dx))
    o = Oracle(lay.n, lay.lo, **kw)
    o.set_state(*state)
    o.advance(max_sweeps=1)
    ref = o.get_times()[2]
    assert np.all(ref > 1e15)
    for precision in (0, 2):
        g = Dispatch(lay.n, lay.lo, precision=precision, **kw)
        g.set_state(*state)
        g.advance(max_sweeps=1)
        speed = g.pack(np.arange(lay.npatch), device=False)[1][:, 2]
        g.close()
        assert np.max(np.abs(speed / ref - 1)) <= (0 if precision == 0 else 1e-11)
