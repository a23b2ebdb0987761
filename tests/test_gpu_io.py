"""Initial state, field output and conserved totals (the integer forms and the FP64 forms
they fall back to) against the oracle's equilibria and recovery, over speeds up to
0.99999, scales on both sides of the integer forms' exponent ranges, and node counts that
leave a ragged last block."""
import pytest
import torch

import oracle.rlb_oracle as O
from paper_1211_3286_gb300 import inputs as I

pytestmark = pytest.mark.gpu
EPS = 2.0 ** -53


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1211_3286_gb300 import build
    build.build()


def _node_fields(shape, lattice, scale):
    """Seeded e, u, n with speeds from 0 to 0.99999 in all directions."""
    N = shape[0] * shape[1] * shape[2]
    r = torch.from_numpy(I.uniform(77, 1, 6 * N)).reshape(6, N)
    d = 2.0 * r[:3] - 1.0
    if lattice == "d2q9":
        d[2] = 0.0
    d = d / d.norm(dim=0)
    speed = torch.tensor([0.0, 1e-9, 0.3, 0.7, 0.9, 0.99, 0.99999], dtype=torch.float64)[torch.arange(N) % 7]
    u = (d * speed).reshape((3,) + shape)
    e = (scale * (0.5 + r[3])).reshape(shape)
    n = (scale * (0.5 + r[4])).reshape(shape)
    return e, u, n


@pytest.mark.parametrize("lattice, precision, scale", [
    ("d3q19", "fp64", 1.0), ("d3q19", "fp64", 2.0 ** -890), ("d3q19", "fp64", 2.0 ** -950),
    ("d3q19", "fp64", 2.0 ** 860), ("d3q19", "fp64", 2.0 ** 900), ("d2q9", "fp64", 1.0), ("d2q9", "fp64", 2.0 ** -950),
    ("d3q19", "fp32", 1.0), ("d3q19", "fp32", 2.0 ** -60), ("d3q19", "fp32", 2.0 ** -70), ("d3q19", "fp32", 2.0 ** 60),
])
@pytest.mark.parametrize("shape", [(1, 1, 1), (3, 5, 37)])
def test_initial_state_and_fields_vs_oracle(lattice, precision, scale, shape):
    """State: |a - b| <= (24 + 8 gamma^2) 2^-53 D per population, with D the node's sigma
    (g) or N0 (f): the oracle rounds about 24 terms of size D, and gamma^2 = 1/(1 - u^2)
    amplifies the rounding of u^2 by 2 gamma^2; FP32 storage adds one rounding, 2^-24 |b|.
    Fields (of the stored state, the oracle's moments of it): sums of 19 terms in FP64,
    64 x 2^-53 sum|g| for P and over sigma for u; n = N0 sqrt(1 - u^2) takes 2 gamma^2
    times u's error."""
    from paper_1211_3286_gb300.lattice import Lattice
    if lattice == "d2q9":
        shape = (1,) + shape[1:]
    e, u, n = _node_fields(shape, lattice, scale)
    lat = Lattice(shape, collision="mrt", tau_v=0.9, tau_e=0.55, tau_eps=0.8, precision=precision, lattice=lattice)
    lat.set_fields(e.cuda(), u[0].cuda(), u[1].cuda(), u[2].cuda(), n.cuda())
    st = lat.state("cpu").to(torch.float64)
    Q = lat.Q
    f, g = O.init_populations(e, u, n, lattice)
    g2 = 1.0 / (1.0 - (u * u).sum(0))
    sigma, N0 = 4.0 / 3.0 * e * g2, n * g2.sqrt()
    tol = (24.0 + 8.0 * g2) * EPS
    store = 2.0 ** -24 if precision == "fp32" else 0.0
    assert bool(((st[:Q] - f).abs() <= tol * N0 + store * f.abs()).all())
    assert bool(((st[Q:] - g).abs() <= tol * sigma + store * g.abs()).all())
    if not 2.0 ** -500 < scale < 2.0 ** 500:   # the recovery's T00^2 leaves the FP64 range
        lat.close()
        return
    fl = lat.fields("cpu")
    ref = O.recover(*O.moments(st[:Q], st[Q:]), check=False)
    sg, sf = st[Q:].abs().sum(0), st[:Q].abs().sum(0)
    g2 = ref.gamma ** 2
    du = 64 * EPS * sg / ref.sigma
    # the disc of the recovery amplifies its rounding by sigma / P = 4 gamma^2 near |u| = 1
    assert bool(((fl["P"] - ref.P).abs() <= 64 * EPS * sg).all())
    assert torch.equal(fl["e"], 3.0 * fl["P"])
    for k in range(3):
        assert bool(((fl[("ux", "uy", "uz")[k]] - ref.u[k]).abs() <= du).all())
    assert bool(((fl["n"] - ref.n).abs() <= 64 * EPS * sf + 2 * g2 * du * ref.n.abs()).all())
    tot = lat.totals()
    lat.close()
    N0, T00, M = O.moments(st[:Q], st[Q:])
    want = [N0.sum(), T00.sum(), M[0].sum(), M[1].sum(), M[2].sum()]
    for c in range(5):
        s = (sf if c == 0 else sg).sum()
        assert abs(float(tot[c]) - float(want[c])) <= 64 * EPS * float(s), c


def test_initial_fields_refused_as_before():
    """Inputs the initial state refuses: the integer form hands each to the FP64 checks."""
    from paper_1211_3286_gb300 import _lib as L
    from paper_1211_3286_gb300.lattice import Lattice
    inf, nan = float("inf"), float("nan")
    lat = Lattice((1, 1, 5))
    ok = [1e-2, 0.1, 0.0, 0.0, 1.0]
    for c, v in [(0, 0.0), (0, -1.0), (0, inf), (0, nan), (4, 0.0), (4, -1.0), (4, inf), (4, nan), (1, 1.0),
                 (1, -1.0), (2, 1.5), (3, nan), (3, inf)]:
        f = [torch.full((1, 1, 5), q, dtype=torch.float64) for q in ok]
        f[c][0, 0, 3] = v
        with pytest.raises(L.RlbError) as ex:
            lat.set_fields(*f)
        assert ex.value.code == L.RLB_EINVAL and "node 3" in str(ex.value)
    # the ends of what is accepted
    for c, v in [(0, 5e-324), (4, 1e300), (1, 1.0 - 2.0 ** -53), (0, 1e-300)]:
        f = [torch.full((1, 1, 5), q, dtype=torch.float64) for q in ok]
        f[c][0, 0, 3] = v
        lat.set_fields(*f)
    lat.close()


@pytest.mark.parametrize("lattice, precision", [("d3q19", "fp64"), ("d3q19", "fp32"), ("d2q9", "fp64")])
def test_velocity_output_keeps_its_relative_precision_at_any_speed(lattice, precision):
    """u of the stored state at speeds from 1e-2 down to 1e-13, against the momentum summed
    exactly and the recovery in 60 digits.  Sums of slow populations in FP64 are good to 2^-53 of
    the pair differences, at most 3 |u| sigma each, five of them, and the recovery adds three
    roundings: 16 x 2^-53 |u| for each component."""
    from decimal import Decimal, getcontext
    from fractions import Fraction
    from paper_1211_3286_gb300.lattice import Lattice
    getcontext().prec = 60
    N = 96
    shape = (1, 8, 12) if lattice == "d2q9" else (2, 4, 12)
    r = torch.from_numpy(I.uniform(78, 1, 5 * N)).reshape(5, N)
    d = 2.0 * r[:3] - 1.0
    if lattice == "d2q9":
        d[2] = 0.0
    speed = torch.tensor([10.0 ** -(2 + k) for k in range(12)], dtype=torch.float64)[torch.arange(N) % 12]
    u = (d / d.norm(dim=0) * speed).reshape((3,) + shape)
    e, n = (0.5 + r[3]).reshape(shape), (0.5 + r[4]).reshape(shape)
    lat = Lattice(shape, collision="mrt", tau_v=0.9, tau_e=0.55, tau_eps=0.8, precision=precision, lattice=lattice)
    lat.set_fields(e.cuda(), u[0].cuda(), u[1].cuda(), u[2].cuda(), n.cuda())
    g = lat.state("cpu").to(torch.float64)[lat.Q:].reshape(lat.Q, N)
    fl = lat.fields("cpu")
    lat.close()
    out = torch.stack([fl[k].reshape(N) for k in ("ux", "uy", "uz")])
    E, _ = O.lattice(lattice)
    for x in range(N):
        v = [Fraction(float(g[a, x])) for a in range(lat.Q)]
        M = [sum(int(E[a][k]) * v[a] for a in range(lat.Q)) for k in range(3)]
        dec = lambda q: Decimal(q.numerator) / Decimal(q.denominator)
        H = 2 * dec(sum(v)) + (dec(4 * sum(v) ** 2 - 3 * sum(m * m for m in M))).sqrt()
        want = [3 * dec(m) / H for m in M]
        size = float(sum(w * w for w in want).sqrt())
        for k in range(3):
            assert abs(float(Decimal(float(out[k, x])) - want[k])) <= 16 * EPS * size, (x, k, size)


def test_fp32_initial_state_is_the_fp64_equilibrium_rounded_once():
    """The integer form's FP32 state at scale 1 against the FP64 form's (the same fields times
    2^-70 lie outside the integer form's range), scaled back: equal bit for bit on 2^20 nodes,
    about one in 2^13 of which has a population next to a rounding tie."""
    from paper_1211_3286_gb300.lattice import Lattice
    shape = (64, 128, 128)
    e, u, n = _node_fields(shape, "d3q19", 1.0)
    u = 0.8 * u
    st = []
    for scale in (1.0, 2.0 ** -70):
        lat = Lattice(shape, collision="mrt", tau_v=0.9, tau_e=0.55, tau_eps=0.8, precision="fp32")
        lat.set_fields((e * scale).cuda(), u[0].cuda(), u[1].cuda(), u[2].cuda(), (n * scale).cuda())
        st.append(lat.state())
        lat.close()
    assert torch.equal(st[0], st[1] * 2.0 ** 70)
