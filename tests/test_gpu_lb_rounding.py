"""Rounding of the LB collision, to the last bit: one step of the library against
the same operations in the same order in numpy."""
import numpy as np
import pytest

from paper_2503_06610_gb300 import inputs as I

pytestmark = pytest.mark.gpu

E = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0),
     (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1),
     (0, -1, 1)]
R = np.float32


def fma(a, b, c):
    """Rounded once: 113 bits hold a product of two FP32 values and its sum with a third of comparable size."""
    q = np.longdouble
    return (q(a) * q(b) + q(c)).astype(R) if np.ndim(a) or np.ndim(b) or np.ndim(c) else R(q(a) * q(b) + q(c))


def dot(e, v):
    """e . v by sums and differences in the order x, y, z."""
    r = None
    for c, a in zip(e, v):
        if c:
            r = (a if c > 0 else -a) if r is None else (r + a if c > 0 else r - a)
    return r


def collide_by_pairs(f, F, g, omega, shifted):
    """FP32 collision of the streamed populations f [19][N], a pair (e_i, -e_i) after the other; returns f*, u, rho."""
    total, m = f[0].copy(), [np.zeros_like(f[0]) for _ in range(3)]
    for i in range(1, 19, 2):
        total = total + (f[i] + f[i + 1])
        d = f[i] - f[i + 1]
        for a in range(3):
            if E[i][a]:
                m[a] = m[a] + (d if E[i][a] > 0 else -d)
    rho = R(1) + total if shifted else total
    base = total if shifted else rho
    F = [fma(rho, R(g[a]), F[a]) for a in range(3)]
    inv = R(1) / rho
    u = [fma(R(0.5), F[a], m[a]) * inv for a in range(3)]
    omc, cS = R(1) - omega, fma(R(-0.5), omega, R(1))
    uu = R(1.5) * fma(u[2], u[2], fma(u[1], u[1], u[0] * u[0]))
    uF = R(3) * fma(u[2], F[2], fma(u[1], F[1], u[0] * F[0]))
    out = [None] * 19
    w = R(1) / R(3)
    out[0] = fma(omc, f[0], fma(omega * w, fma(-rho, uu, base), -((cS * w) * uF)))
    for i in range(1, 19, 2):
        w = R(1) / R(18) if i < 7 else R(1) / R(36)
        ow = omega * w
        A, B, C = ow * rho, ow * base, cS * w
        eu, eF = dot(E[i], u), dot(E[i], F)
        even = fma(C, fma(R(9) * eu, eF, -uF), fma(A, fma(R(4.5) * eu, eu, -uu), B))
        odd = R(3) * fma(A, eu, C * eF)
        out[i] = fma(omc, f[i], even) + odd
        out[i + 1] = fma(omc, f[i + 1], even) - odd
    return np.stack(out), np.stack(u), rho


def channel(storage, shifted, dims, tau=0.8):
    nx, ny, nz = dims
    from paper_2503_06610_gb300 import nh
    ch = nh.Channel(dict(nx=nx, ny=ny, nz=nz, walls_z=False, anchoring="none", shifted=shifted, tau=tau, g=(1e-5, 3e-6, -2e-6),
                         K=0.005, q0=0.2, W0=0.0, dt_fd=1000, precision="fp32", storage=storage, **I.LESLIE_ALIGN_09))
    N = nx * ny * nz
    rng = np.random.Generator(np.random.PCG64(7))
    ch.set_fields(I.tilted_director(nx, ny, nz, amplitude=0.5, seed=1), rng.uniform(-0.02, 0.02, size=(3, N)),
                  1.0 + rng.uniform(-0.01, 0.01, size=N))
    ch.step(3)
    return ch


def stream(f, dims):
    nx, ny, nz = dims
    return np.stack([np.roll(f[i].reshape(nz, ny, nx), (e[2], e[1], e[0]), (0, 1, 2)).ravel() for i, e in enumerate(E)])


def step_by_pairs(ch, dims, shifted, tau):
    """The next step of the channel: what collide_by_pairs makes of its state, and what the library does."""
    f, F = ch.get_populations().reshape(19, -1).astype(R), ch.get_force().reshape(3, -1).astype(R)
    want = collide_by_pairs(stream(f, dims), F, (1e-5, 3e-6, -2e-6), R(1.0 / tau), shifted)
    ch.step(1)
    _, u, rho = ch.get_fields()
    return want, (ch.get_populations().reshape(19, -1), np.asarray(u).reshape(3, -1), np.asarray(rho).ravel())


# 16-bit stores: an odd row (one site a thread), rows of four (four sites), 256-site rows staged in shared memory
@pytest.mark.parametrize("storage,bits", [("f16s", 11), ("bf16s", 8)])
@pytest.mark.parametrize("dims", [(33, 18, 9), (64, 64, 28), (256, 64, 64)])
def test_16_bit_stores_round_as_by_pairs(storage, bits, dims):
    ch = channel(storage, True, dims)
    (want, wu, wrho), (got, u, rho) = step_by_pairs(ch, dims, True, 0.8)
    assert np.array_equal(u.astype(R), wu) and np.array_equal(rho.astype(R), wrho)
    mant, exp = np.frexp(want.astype(np.float64))  # to nearest even at the store's significand
    want = np.ldexp(np.round(mant * 2.0 ** bits) * 2.0 ** -bits, exp)
    normal = np.abs(want) > 2.0 ** -10 * np.abs(want).max()  # F16S: above the store's subnormal range
    assert normal.mean() > 0.9
    assert np.array_equal(got[normal], want[normal])


# sites per thread by size: odd rows, small blocks, two sites; pairs of steps collide with the same code
@pytest.mark.parametrize("dims", [(33, 18, 9), (64, 64, 28)])
@pytest.mark.parametrize("tau", [0.7, 1.1])
def test_unshifted_fp32_rounds_as_by_pairs(dims, tau):
    ch = channel("f32", False, dims, tau)
    (want, wu, wrho), (got, u, rho) = step_by_pairs(ch, dims, False, tau)
    assert np.array_equal(u.astype(R), wu) and np.array_equal(rho.astype(R), wrho)
    assert np.array_equal(got.astype(R), want)


# 7.5e5 sites and more: pairs of steps
@pytest.mark.parametrize("dims", [(48, 40, 24), (160, 120, 40)])
@pytest.mark.parametrize("tau", [0.55, 0.7, 0.8, 1.0, 1.1, 1.478])
@pytest.mark.parametrize("walls", [True, False])
def test_shifted_fp32_errors_do_not_grow_with_the_steps(dims, tau, walls):
    """Velocity of 250 steps against FP64.  A step rounds u a few times, to 2^-24 of it each; errors that are not the
    same at every site and step add as their root mean square, sqrt(250) * 2^-24 = 0.94e-6 for one a step, less what
    viscosity takes away.  A bias of the weights by 2^-25 would give 250 / tau * 2^-25 = 7.5e-6 / tau."""
    from paper_2503_06610_gb300 import nh
    nx, ny, nz = dims
    N = nx * ny * nz
    n = np.zeros((3, N))
    n[2] = 1.0  # uniform: no force from the director
    x, y, z = np.meshgrid(np.arange(nx), np.arange(ny), np.arange(nz), indexing="ij")
    kx, ky = 2 * np.pi / nx, 2 * np.pi / ny
    prof = np.sin(np.pi * (z + 0.5) / nz) if walls else 1.0 + 0.3 * np.sin(2 * np.pi * z / nz)
    u = 2e-3 * np.stack([(prof * f).transpose(2, 1, 0).ravel() for f in (1 + 0.3 * np.cos(ky * y), 0.6 + np.cos(kx * x + 1),
                                                                         0.3 * np.cos(kx * x - ky * y))])
    out = []
    for precision, storage in (("fp64", "f64"), ("fp32", "f32")):
        ch = nh.Channel(dict(nx=nx, ny=ny, nz=nz, walls_z=walls, anchoring="none", shifted=True, tau=tau, g=(2.0 ** -20, 0.0, 0.0),
                             K=0.005, q0=0.0, W0=0.0, dt_fd=1000, precision=precision, storage=storage, **I.LESLIE_ALIGN_09))
        ch.set_fields(n, u.astype(R).astype(np.float64))
        ch.step(250)
        out.append(np.asarray(ch.get_fields()[1]).ravel())
    assert np.linalg.norm(out[1] - out[0]) < 250 ** 0.5 * 2.0 ** -24 * np.linalg.norm(out[0])
