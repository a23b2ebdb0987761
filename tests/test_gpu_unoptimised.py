"""The integer kernels against the same source assembled without optimisation.

Their results are integers of the inputs, each rounded once, so both builds have to agree bit
for bit.  ptxas 13.0 has lost a carry between the 32-bit halves of a 64-bit sum (at -O1 and up,
not at -O0) where a correction that two opposite links take with opposite signs was folded
into the sum of the relaxation; the sources keep those sums apart (fx::relax says where), and
a sum that is not kept apart shows here as 2^-24 of a node's largest population.  Paths with FP32 or FP64
arithmetic of their own are left out: there the two builds contract products differently."""
import os
import shutil
import subprocess
import sys

import pytest
import torch

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = """
import hashlib, itertools, os, sys
sys.path.insert(0, os.getcwd())
import numpy as np, torch
from paper_1211_3286_gb300 import inputs as I
from paper_1211_3286_gb300.batch import TubeBatch
from paper_1211_3286_gb300.lattice import Lattice

def digest(t):
    return hashlib.md5(t.contiguous().cpu().numpy().tobytes()).hexdigest()

def run(shape, eta=0.0, lattice="d3q19", **kw):
    if shape[1] == 4:
        f = [torch.from_numpy(a).cuda().expand(shape).contiguous()
             for a in I.shock_tube(shape[2], **(I.PAPER_LATTICE_UNITS if eta else {}))]
    else:
        f = list(I.periodic_box(None, seed=3, shape=shape, device="cuda", umax=0.15 if eta else 0.3,
                                **(dict(e0=6e-7, n0=2e-7 / 0.0314) if eta else {})))
    if lattice == "d2q9":
        f[3] = torch.zeros_like(f[3])
    l = Lattice(shape, eta_over_s=eta, lattice=lattice, bc=("zero_gradient", "periodic", "periodic"), **kw)
    l.set_fields(*f)
    out = [digest(l.state())]
    for n in (12, 1):
        l.step(n)
        out.append(digest(l.state()))
    fl = l.fields()
    print(lattice, shape, eta, kw, out, digest(torch.stack([fl[k] for k in sorted(fl)])), l.totals())
    l.close()

T = dict(tau_f=0.7, tau_e=0.55, tau_eps=0.8)
for (co, tq), shape in itertools.product((("mrt", 0.0), ("mrt", 0.7), ("bgk", 0.0)),
                                         ((1, 1, 320), (1, 4, 320), (5, 4, 2000), (9, 37, 130), (10, 31, 128))):
    for tv in (0.9, 1.3):
        run(shape, collision=co, tau_q=tq, tau_v=tv, **T)
        if shape[0] == 1:
            run(shape, lattice="d2q9", collision=co, tau_q=tq, tau_v=tv, **T)
    run(shape, eta=0.1, collision=co, tau_f=0.0 if co == "bgk" else 0.6, tau_v=0.9, tau_e=0.05, tau_eps=0.1, tau_q=tq)
for nt in (5, 40):
    L, taus = I.tube_sweep(nt, seed=4, Lmin=1, Lmax=900)
    ps = [I.shock_tube(int(x)) for x in L]
    f = [torch.from_numpy(np.concatenate([p[k].reshape(-1) for p in ps])).cuda() for k in range(5)]
    for co in ("mrt", "bgk"):
        b = TubeBatch(L, taus, precision="fp64", collision=co)
        b.set_fields(*f)
        b.run(21)
        print(nt, co, digest(b.state()))
        b.close()
"""


def test_integer_kernels_do_not_depend_on_the_assembler_s_optimisation(tmp_path):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1211_3286_gb300 import build
    build.build()
    for d in ("paper_1211_3286_gb300", "include"):
        shutil.copytree(os.path.join(ROOT, d), tmp_path / d, ignore=shutil.ignore_patterns("_build", "__pycache__"))
    plain = "from paper_1211_3286_gb300 import build; build.build(extra_flags=['-Xptxas', '-O0'])"
    subprocess.run([sys.executable, "-c", plain], cwd=tmp_path, check=True)
    said = [subprocess.run([sys.executable, "-c", CHILD], cwd=where, check=True, capture_output=True, text=True).stdout
            for where in (ROOT, tmp_path)]
    a, b = (s.splitlines() for s in said)
    assert len(a) == len(b) > 50
    assert [(x, y) for x, y in zip(a, b) if x != y] == []
