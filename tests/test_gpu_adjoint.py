"""GPU adjoint (rlb_adjoint, hand-written reverse-mode kernels) against the oracle's
exact discrete gradient (reverse-mode differentiation of the CPU oracle) and against
central finite differences of the GPU forward run."""
import math

import numpy as np
import pytest
import torch

import oracle.rlb_oracle as O
from paper_1211_3286_gb300 import inputs as I

pytestmark = pytest.mark.gpu

ZG = ("zero_gradient", "periodic", "periodic")


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1211_3286_gb300 import build
    build.build()


def _obc(bc):
    return tuple(O.ZERO_GRADIENT if b == "zero_gradient" else O.PERIODIC for b in bc)


def _case(shape, kind, seed, taus, collision, bc, T):
    """Initial fields, targets from a perturbed run of the oracle."""
    if kind == "tube":
        e, ux, uy, uz, n = (torch.from_numpy(a) for a in I.shock_tube(shape[2]))
    else:
        e, ux, uy, uz, n = I.periodic_box(None, seed=seed, shape=shape)
        ux, uy, uz = 0.5 * ux, 0.5 * uy, 0.5 * uz
    u = torch.stack([ux, uy, uz])
    pert = torch.from_numpy(I.perturbation(e.numel(), seed=seed)).reshape(e.shape)
    tv, te, tp = taus
    prm_t = O.Params(collision=collision, tau_f=tv, tau_v=tv * 1.01, tau_e=te * 1.01, tau_eps=tp * 1.01, bc=_obc(bc))
    f, g = O.run(*O.init_populations(e * (1 + 1e-3 * pert), u, n), prm_t, T)
    tgt = O.fields(f, g)
    return e, u, n, tgt


def _gpu_grad(e, u, n, tgt, taus, collision, bc, T, K=0, w_P=1.0, w_u=1.0):
    from paper_1211_3286_gb300.adjoint import misfit_gradient
    from paper_1211_3286_gb300.lattice import Lattice
    tv, te, tp = taus
    lat = Lattice(tuple(e.shape), collision=collision, tau_f=tv, tau_v=tv, tau_e=te, tau_eps=tp, bc=bc)
    lat.set_fields(e.cuda(), u[0].cuda(), u[1].cuda(), u[2].cuda(), n.cuda())
    out = misfit_gradient(lat, T, tgt.P.cuda(), tgt.u[0].cuda(), tgt.u[1].cuda(), tgt.u[2].cuda(), w_P, w_u, K)
    lat.close()
    return out


@pytest.mark.parametrize("shape, kind, collision, bc, T", [
    ((1, 1, 24), "tube", "mrt", ZG, 30),
    ((1, 1, 24), "tube", "bgk", ZG, 30),
    ((4, 5, 6), "box", "mrt", ("periodic",) * 3, 8),
    ((3, 4, 7), "box", "mrt", ("periodic", "zero_gradient", "zero_gradient"), 6),
])
def test_adjoint_matches_oracle_discrete_gradient(shape, kind, collision, bc, T):
    taus = (0.9, 0.55, 0.8) if collision == "mrt" else (0.9, 0.9, 0.9)
    e, u, n, tgt = _case(shape, kind, 51, taus, collision, bc, T)
    loss, dtau, de0 = _gpu_grad(e, u, n, tgt, taus, collision, bc, T)
    prm = O.Params(collision=collision, tau_f=taus[0], tau_v=taus[0], tau_e=taus[1], tau_eps=taus[2], bc=_obc(bc))
    lref, dref, eref = O.misfit_and_gradient(e, u, n, prm, T, tgt.P, tgt.u)
    # J and its gradient are built from P - P* with |P - P*| ~ 1e-3 |P|: the 1e-14 field
    # agreement becomes ~1e-11 in J, hence the 1e-9 / 1e-8 bars
    assert abs(loss - lref) <= 1e-9 * abs(lref)
    if collision == "mrt":
        assert torch.allclose(dtau, dref, rtol=1e-8, atol=0), (dtau, dref)
    else:
        assert abs(dtau[0] - dref[0]) <= 1e-8 * abs(dref[0])   # tau_v only; oracle's tau_e/tau_eps unused by BGK
        assert dtau[1] == 0 and dtau[2] == 0
    err = float((de0.cpu() - eref).abs().max() / eref.abs().max())
    assert err < 1e-8, err


def test_checkpoint_interval_does_not_change_the_gradient():
    taus = (0.9, 0.55, 0.8)
    e, u, n, tgt = _case((1, 1, 40), "tube", 52, taus, "mrt", ZG, 45)
    base = _gpu_grad(e, u, n, tgt, taus, "mrt", ZG, 45, K=0)
    for K in (1, 4, 7, 45, 100):
        other = _gpu_grad(e, u, n, tgt, taus, "mrt", ZG, 45, K=K)
        assert other[0] == base[0]
        assert torch.equal(other[1], base[1])
        assert torch.equal(other[2], base[2])


def test_autograd_function_returns_the_adjoint_gradients():
    from paper_1211_3286_gb300.adjoint import shock_tube_misfit
    taus = (0.9, 0.55, 0.8)
    e, u, n, tgt = _case((1, 1, 32), "tube", 53, taus, "mrt", ZG, 20)
    tv, te, tp = (torch.tensor(t, dtype=torch.float64, requires_grad=True) for t in taus)
    e0 = e.clone().cuda().requires_grad_(True)
    loss = shock_tube_misfit(tv, te, tp, e0, [c.cuda() for c in u], n.cuda(),
                             (tgt.P.cuda(), tgt.u[0].cuda(), tgt.u[1].cuda(), tgt.u[2].cuda()), 20)
    loss.backward()
    l2, d2, e2 = _gpu_grad(e, u, n, tgt, taus, "mrt", ZG, 20)
    assert float(loss) == l2
    assert torch.equal(torch.stack([tv.grad, te.grad, tp.grad]), d2)
    assert torch.equal(e0.grad, e2)


def test_config5_1600_nodes_4000_steps_vs_central_differences():
    """Quasi-1D tube of 1600 nodes, FP64 MRT (0.9, 0.55, 0.8), 4000 steps, sqrt(T)
    checkpoints; target from a run with e0 perturbed by 1e-3 seed noise and the taus
    by 1 %.  Gradients against fourth-order central differences of the GPU forward
    misfit, normwise over each gradient vector: |FD - adjoint|_inf <= 1e-6 |adjoint|_inf.

    Step choice: after 4000 steps the misfit carries ~4e-11 relative round-off, so a
    difference quotient with h = 1e-6 tau is noise-dominated (its error grows as h
    shrinks); h = 3e-4 tau with the fourth-order stencil keeps both the truncation
    (O(h^4)) and the noise (~J_noise / h) below 1e-6."""
    from paper_1211_3286_gb300.lattice import Lattice
    L, T = 1600, 4000
    taus = (0.9, 0.55, 0.8)
    e, ux, uy, uz, n = (torch.from_numpy(a).cuda() for a in I.shock_tube(L))
    pert = torch.from_numpy(I.perturbation(L)).reshape(1, 1, L).cuda()

    def forward_fields(tv, te, tp, e0):
        lat = Lattice((1, 1, L), collision="mrt", tau_f=taus[0], tau_v=tv, tau_e=te, tau_eps=tp, bc=ZG)
        lat.set_fields(e0, ux, uy, uz, n)
        lat.step(T)
        fl = lat.fields("cuda")
        lat.close()
        return fl

    tf = forward_fields(taus[0] * 1.01, taus[1] * 1.01, taus[2] * 1.01, e * (1 + 1e-3 * pert))

    def J(tv, te, tp, e0):
        fl = forward_fields(tv, te, tp, e0)
        return float(((fl["P"] - tf["P"]) ** 2).sum() + ((fl["ux"] - tf["ux"]) ** 2).sum()
                     + ((fl["uy"] - tf["uy"]) ** 2).sum() + ((fl["uz"] - tf["uz"]) ** 2).sum())

    def d4(fun, h):
        return (-fun(2 * h) + 8 * fun(h) - 8 * fun(-h) + fun(-2 * h)) / (12 * h)

    from paper_1211_3286_gb300.adjoint import misfit_gradient
    lat = Lattice((1, 1, L), collision="mrt", tau_f=taus[0], tau_v=taus[0], tau_e=taus[1], tau_eps=taus[2], bc=ZG)
    lat.set_fields(e, ux, uy, uz, n)
    loss, dtau, de0 = misfit_gradient(lat, T, tf["P"], tf["ux"], tf["uy"], tf["uz"])
    lat.close()
    assert abs(loss - J(*taus, e)) <= 1e-12 * loss   # same GPU forward, only the sum order differs
    fd_tau = []
    for i in range(3):
        def shifted(dh, i=i):
            t = list(taus)
            t[i] += dh
            return J(*t, e)
        fd_tau.append(d4(shifted, 3e-4 * taus[i]))
    fd_tau = torch.tensor(fd_tau, dtype=torch.float64)
    assert float((fd_tau - dtau).abs().max() / dtau.abs().max()) <= 1e-6, (fd_tau, dtau)
    nodes = (0, 400, 799, 800, 1200, 1599)
    fd_e, ad_e = [], []
    for j in nodes:
        def shifted_e(dh, j=j):
            ee = e.clone()
            ee[0, 0, j] += dh
            return J(*taus, ee)
        fd_e.append(d4(shifted_e, 3e-4 * float(e[0, 0, j])))
        ad_e.append(float(de0[0, 0, j]))
    fd_e, ad_e = torch.tensor(fd_e), torch.tensor(ad_e)
    assert float((fd_e - ad_e).abs().max() / ad_e.abs().max()) <= 1e-6, (fd_e, ad_e)


@pytest.mark.parametrize("shape, kind, T, K", [
    ((1, 1, 400), "tube", 400, 100),     # four lanes per node, two warp roles (k_adj_step_ws), 4 segments
    ((1, 1, 1600), "tube", 200, 50),     # four lanes per node, 4 segments
    ((4, 100, 100), "box", 12, 4),       # one thread per node (k_adj_step: > 38,912 nodes), 3 segments
])
def test_adjoint_matches_oracle_at_mid_size(shape, kind, T, K):
    """MRT (0.9, 0.55, 0.8) gradients against the oracle's exact discrete gradient on
    lattices where the checkpoint segments span many steps: J to 1e-9, d tau and
    d e0 to 1e-8 (normwise).  The misfit is built from P - P* ~ 1e-3 P, so the 1e-13
    agreement of the forward fields becomes ~1e-10 in J and its gradient."""
    taus = (0.9, 0.55, 0.8)
    bc = ZG if kind == "tube" else ("periodic",) * 3
    e, u, n, tgt = _case(shape, kind, 54, taus, "mrt", bc, T)
    loss, dtau, de0 = _gpu_grad(e, u, n, tgt, taus, "mrt", bc, T, K=K)
    prm = O.Params(collision="mrt", tau_f=taus[0], tau_v=taus[0], tau_e=taus[1], tau_eps=taus[2], bc=_obc(bc))
    lref, dref, eref = O.misfit_and_gradient(e, u, n, prm, T, tgt.P, tgt.u)
    assert abs(loss - lref) <= 1e-9 * abs(lref), (loss, lref)
    assert float((dtau - dref).abs().max() / dref.abs().max()) <= 1e-8, (dtau, dref)
    err = float((de0.cpu() - eref).abs().max() / eref.abs().max())
    assert err <= 1e-8, err


@pytest.mark.parametrize("collision", ["mrt", "bgk"])
@pytest.mark.parametrize("bcx", ["zero_gradient", "periodic"])
@pytest.mark.parametrize("L", [1, 2, 31, 32, 33, 61])
def test_adjoint_of_tubes_around_the_tile_size(L, bcx, collision):
    """Quasi-1D gradients at the sizes where the tiles of the multi-step kernels change: one
    node, a tile that holds the whole lattice (wrapping or open), one node more, a ragged
    last tile; 25 steps (several launches, a ragged last segment) against the oracle's discrete
    gradient, with the bounds of test_adjoint_matches_oracle_discrete_gradient plus, for
    dJ/dtau, its rounding of about 2^-53 x 25 steps x 19 links x |lambda| |g| with |lambda| |g| <=
    2e3 J (the targets are 1e-3 off), below 1e-9 J: on one node, and nearly so on two, dJ/dtau
    is a sum that cancels (a single node stays at equilibrium)."""
    taus = (0.9, 0.55, 0.8) if collision == "mrt" else (0.9, 0.9, 0.9)
    bc = (bcx, "periodic", "periodic")
    e, u, n, tgt = _case((1, 1, L), "box", 55, taus, collision, bc, 25)
    loss, dtau, de0 = _gpu_grad(e, u, n, tgt, taus, collision, bc, 25)
    prm = O.Params(collision=collision, tau_f=taus[0], tau_v=taus[0], tau_e=taus[1], tau_eps=taus[2], bc=_obc(bc))
    lref, dref, eref = O.misfit_and_gradient(e, u, n, prm, 25, tgt.P, tgt.u)
    assert abs(loss - lref) <= 1e-9 * abs(lref)
    want = dref if collision == "mrt" else dref * torch.tensor([1.0, 0, 0])
    assert float((dtau - want).abs().max()) <= 1e-8 * float(dref.abs().max()) + 1e-9 * abs(lref)
    assert float((de0.cpu() - eref).abs().max()) <= 1e-8 * float(eref.abs().max())


def test_adjoint_passes_nan_targets_on():
    """A NaN in a target reaches the loss, the tau gradients and the initial field's gradient in
    its domain of dependence, and nowhere else."""
    taus, T = (0.9, 0.55, 0.8), 10
    e, u, n, tgt = _case((1, 1, 100), "tube", 56, taus, "mrt", ZG, T)
    tgt.P[0, 0, 50] = float("nan")
    loss, dtau, de0 = _gpu_grad(e, u, n, tgt, taus, "mrt", ZG, T)
    assert math.isnan(loss) and bool(torch.isnan(dtau).all())
    bad = torch.isnan(de0.cpu()).reshape(-1)
    assert bool(bad[45:56].all()) and not bool(bad[:50 - T - 1].any()) and not bool(bad[50 + T + 2:].any())


def test_adjoint_with_one_segment_of_66000_steps():
    """A checkpoint interval beyond the 65535 blocks of a grid's y (the rate cotangents take a
    segment's steps along it): the gradient equals the one with the default interval bit for bit."""
    taus, T = (0.9, 0.55, 0.8), 66000
    e, u, n, tgt = _case((1, 1, 8), "tube", 57, taus, "mrt", ZG, 3)
    a = _gpu_grad(e, u, n, tgt, taus, "mrt", ZG, T, K=T)
    b = _gpu_grad(e, u, n, tgt, taus, "mrt", ZG, T)
    assert a[0] == b[0] and torch.equal(a[1], b[1]) and torch.equal(a[2], b[2])


@pytest.mark.parametrize("collision", ["mrt", "bgk"])
def test_gradient_is_odd_in_the_misfit_weights(collision):
    """-w_P, -w_u give the negated gradient but for the walk's roundings, which carry no sign: at most
    about 0.64 x 2^-53 of a node's |lambda| (rms) per reverse step, 200 steps of them in quadrature
    14 times that, three standard deviations and |lambda| up to twice |dJ/de0|: 64 x 2^-53.
    Products cut off downwards would add up to some 700 x 2^-53."""
    taus = (0.9, 0.55, 0.8) if collision == "mrt" else (0.9, 0.9, 0.9)
    e, u, n, tgt = _case((1, 1, 48), "tube", 59, taus, collision, ZG, 200)
    a = _gpu_grad(e, u, n, tgt, taus, collision, ZG, 200)
    b = _gpu_grad(e, u, n, tgt, taus, collision, ZG, 200, w_P=-1.0, w_u=-1.0)
    assert b[0] == -a[0]
    assert float((a[2] + b[2]).abs().max()) <= 64 * 2.0 ** -53 * float(a[2].abs().max())


@pytest.mark.parametrize("collision", ["mrt", "bgk"])
def test_gradient_scales_with_the_misfit_weights_over_the_number_range(collision):
    """The gradient is linear in (w_P, w_u): powers of two that bring its largest component to
    2^1012, 2^-905 and 2^-1000 scale loss and gradients exactly, but for one rounding of what
    ends below the normal numbers."""
    taus = (0.9, 0.55, 0.8) if collision == "mrt" else (0.9, 0.9, 0.9)
    e, u, n, tgt = _case((1, 1, 40), "tube", 58, taus, collision, ZG, 25)
    base = _gpu_grad(e, u, n, tgt, taus, collision, ZG, 25)
    top = math.frexp(float(base[2].abs().max()))[1]
    for target in (1012, -905, -1000):
        w = 2.0 ** ((target - top) // 2)   # in two factors, each of them normal
        v = 2.0 ** ((target - top) - (target - top) // 2)
        got = _gpu_grad(e, u, n, tgt, taus, collision, ZG, 25, w_P=w * v, w_u=w * v)
        assert got[0] == base[0] * w * v
        assert torch.equal(got[1], base[1] * w * v) and torch.equal(got[2], base[2] * w * v), target


def test_gradient_of_a_tube_takes_no_more_memory_than_whole_states():
    """Device memory of a 2000-node tube's first gradient, 4000 steps in two segments: at most the
    two checkpoints, two buffers of K + 1 states and one more state, as with one launch per
    step, the two cotangents and the per-node results (38 + 9 values) and 32 MiB for
    allocation granularity."""
    from paper_1211_3286_gb300.adjoint import misfit_gradient
    from paper_1211_3286_gb300.lattice import Lattice
    L, T, K = 2000, 4000, 2000
    e, ux, uy, uz, n = (torch.from_numpy(a).cuda() for a in I.shock_tube(L))
    lat = Lattice((1, 1, L), collision="mrt", tau_f=0.9, tau_v=0.9, tau_e=0.55, tau_eps=0.8, bc=ZG)
    lat.set_fields(e, ux, uy, uz, n)
    lat.step(30)
    misfit_gradient(lat, 3, e / 3.0, ux, uy, uz)   # the kernels are loaded
    lat.close()
    lat = Lattice((1, 1, L), collision="mrt", tau_f=0.9, tau_v=0.9, tau_e=0.55, tau_eps=0.8, bc=ZG)
    lat.set_fields(e, ux, uy, uz, n)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    misfit_gradient(lat, T, e / 3.0, ux, uy, uz, checkpoint_every=K)
    used = free - torch.cuda.mem_get_info()[0]
    lat.close()
    assert used <= 8 * L * (38 * (2 + 2 * (K + 1) + 1) + 38 + 9) + (32 << 20), used


@pytest.mark.parametrize("shape, bc, Ts", [
    ((3, 4, 7), ("periodic", "zero_gradient", "zero_gradient"), (7, 8)),   # four lanes per node (k_adj_step_ws)
    ((4, 100, 100), ("periodic",) * 3, (5, 6)),                            # one thread per node (k_adj_step)
])
@pytest.mark.parametrize("collision", ["mrt", "bgk"])
def test_repeated_gradients_on_one_lattice_equal_fresh_ones(shape, bc, Ts, collision):
    """A lattice's first gradient is enqueued directly, the second captures a graph, later ones
    replay it, other weights capture it again, and another number of steps makes a new plan.
    Loss, gradients, the state left behind and the step count equal a fresh lattice's bit for
    bit, whichever of the handle's two buffers the state starts in."""
    from paper_1211_3286_gb300.adjoint import misfit_gradient
    from paper_1211_3286_gb300.lattice import Lattice
    taus = (0.9, 0.55, 0.8) if collision == "mrt" else (0.9, 0.9, 0.9)

    def lattice():
        return Lattice(shape, collision=collision, tau_f=taus[0], tau_v=taus[0], tau_e=taus[1], tau_eps=taus[2], bc=bc)

    def gradient(lat, seed, T, w, extra):
        e, ux, uy, uz, n = (t.cuda() for t in I.periodic_box(None, seed=seed, shape=shape))
        tgt = [(1.01 * e / 3.0), 0.9 * ux, 1.1 * uy, uz]
        lat.set_fields(e, 0.5 * ux, 0.5 * uy, 0.5 * uz, n)
        lat.step(extra)   # 0 or 1: the other buffer
        loss, dtau, de0 = misfit_gradient(lat, T, *tgt, *w)
        return torch.tensor([loss]), dtau, de0, lat.state(), torch.tensor([lat.steps_done()])

    kept = lattice()
    for T in Ts:
        for i, w in enumerate([(1.0, 1.0)] * 4 + [(2.5, 0.5)] * 2):
            a = gradient(kept, 90 + i, T, w, i % 2)
            fresh = lattice()
            b = gradient(fresh, 90 + i, T, w, i % 2)
            fresh.close()
            for p, q in zip(a, b):
                assert torch.equal(p, q), (T, i)
            assert int(a[4]) == T + i % 2
    kept.close()


def test_gradient_past_the_format_is_infinite_with_its_sign():
    """Weights that take dJ/de0 up to the largest double and past it, a power of two at a time: every
    component is the exactly scaled one, an infinity of its sign, or NaN (where infinities met
    on the way), never a finite value that has passed the format's end."""
    taus = (0.9, 0.55, 0.8)
    e, u, n, tgt = _case((1, 1, 40), "tube", 58, taus, "mrt", ZG, 3)
    tgt.P += 100.0
    base = _gpu_grad(e, u, n, tgt, taus, "mrt", ZG, 3)[2].cpu()
    top = math.frexp(float(base.abs().max()))[1]
    assert top > 4
    kinds = set()
    for k in range(1012 - top, 1024 - min(top, 3)):
        got = _gpu_grad(e, u, n, tgt, taus, "mrt", ZG, 3, w_P=2.0 ** k, w_u=2.0 ** k)[2].cpu()
        fine, inf = torch.isfinite(got), torch.isinf(got)
        assert torch.equal(got[fine], (base * 2.0 ** (k // 2) * 2.0 ** (k - k // 2))[fine]), k
        assert torch.equal(got[inf].sign(), base[inf].sign()), k
        kinds |= {"fine" if bool(fine.all()) else "past"}
    assert kinds == {"fine", "past"}


def test_gradient_refused_under_capture_leaves_the_lattice_as_it_was():
    """A gradient synchronises, so it is refused on a stream that is being captured.  Nothing has
    run then: the state, its place and the step count are what they were, and the next gradient
    equals a fresh lattice's (odd and even numbers of launches)."""
    import ctypes
    from paper_1211_3286_gb300 import _lib as L
    from paper_1211_3286_gb300.adjoint import misfit_gradient
    from paper_1211_3286_gb300.lattice import Lattice
    rt = ctypes.CDLL("libcudart.so.13")
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        e, ux, uy, uz, n = (torch.from_numpy(a).cuda() for a in I.shock_tube(60))
        tgt = [1.01 * e / 3.0, ux + 0.01, uy, uz]
        for T, sets in ((5, 1), (5, 2), (30, 1), (30, 2)):   # setting the fields changes the buffer
            lat = Lattice((1, 1, 60), collision="mrt", tau_f=0.9, tau_v=0.9, tau_e=0.55, tau_eps=0.8, bc=ZG)
            lat.set_fields(e, ux, uy, uz, n)
            first = misfit_gradient(lat, T, *tgt)   # the plan exists
            for _ in range(sets):
                lat.set_fields(e, ux, uy, uz, n)
            lat.step(3)
            before, steps = lat.state(), lat.steps_done()
            stream, graph = ctypes.c_void_p(s.cuda_stream), ctypes.c_void_p()
            torch.cuda.synchronize()
            assert rt.cudaStreamBeginCapture(stream, 2) == 0   # relaxed
            try:
                with pytest.raises(L.RlbError) as ex:
                    misfit_gradient(lat, T, *tgt)
            finally:
                rt.cudaStreamEndCapture(stream, ctypes.byref(graph))
                if graph:
                    rt.cudaGraphDestroy(graph)
                rt.cudaGetLastError()
            assert ex.value.code == L.RLB_ECUDA
            assert lat.steps_done() == steps and torch.equal(lat.state(), before)
            lat.set_fields(e, ux, uy, uz, n)
            again = misfit_gradient(lat, T, *tgt)
            lat.close()
            assert again[0] == first[0] and torch.equal(again[1], first[1]) and torch.equal(again[2], first[2])
