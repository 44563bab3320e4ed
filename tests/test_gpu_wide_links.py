"""FP32 lattices of more than 2^29 sites index their links in 64 bits, by
kernels compiled apart.  A build that draws that line at no sites at all
(-DSU2_OFF32_MAX_VH=0) sends every lattice there: all launch shapes with slab
walks, persistent tiles and staged rows, both samplers, single phases with
trial output, the fused and the stand-alone plaquette, the Polyakov loop and
the correlator give the ordinary library's results bit by bit."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SCRIPT = r"""
import hashlib
import numpy as np, torch
from paper_1104_5432_gb300 import su2
from paper_1104_5432_gb300.csrc_info import _F32

def show(name, *arrays):
    h = hashlib.sha256()
    for a in arrays:
        h.update(np.ascontiguousarray(a).tobytes())
    print(name, h.hexdigest(), flush=True)

betas, seeds = [2.3, 0.7, 2.6, 1.2], [5, 6, 7, 8]
for cfg in range(14):
    B = su2.Lattice([6, 4, 2, 10], [2, 6, 4, 4], su2.F32)
    B.set_launch_config(cfg)
    B.set_slabs(2 if _F32[cfg][2] else 1)
    for creutz in (0.0, 1.7):
        B.set_sampler(creutz)
        B.batch_init(su2.HOT, seeds)
        p = B.batch_heatbath(betas, 2, seeds)
        m = B.batch_heatbath_measure(betas, 2, seeds, 1)
        show("batch %d %g" % (cfg, creutz), p, *m, *[B.get_links(l) for l in range(4)], B.plaquette(),
             *B.polyakov_loop(), B.polyakov_correlator(1),
             [list(B.stats(l).values()) for l in range(4)])
    B.close()
# one lattice: several tiles a persistent block (24^4: 5184 tiles of 32 links on
# 4864 blocks), rows of 32 links a warp (64^3 x 2)
for Ns, Nt, shapes in ((24, 24, (0, 10, 11, 12)), (64, 2, (5, 8, 9, 13))):
    for cfg in shapes:
        L = su2.Lattice(Ns, Nt, su2.F32)
        L.set_launch_config(cfg)
        L.set_slabs(4)
        L.init(su2.HOT, 9)
        p = L.heatbath(2.4, 2, 3)
        trials = torch.full((L.volume(),), -2, dtype=torch.int32, device="cuda")
        L.heatbath_phase(2.2, 3, 1, 3, trials)
        show("one %d %d" % (Ns, cfg), p, L.get_links(), trials.cpu().numpy(), list(L.stats().values()),
             L.plaquette())
        L.close()
"""


def test_64_bit_link_indices_give_the_same_bits():
    from paper_1104_5432_gb300 import build as b
    wide = b.build(force=True, defines=("SU2_OFF32_MAX_VH=0",),
                   lib_path=os.path.join(b.PKG, "libsu2gb300_wide.so"),
                   build_dir=os.path.join(b.BUILD, "wide"))
    out = []
    for lib in (b.build(), wide):
        env = dict(os.environ, SU2_LIBRARY=lib)
        env.pop("SU2_AUTOTUNE_CACHE", None)
        r = subprocess.run([sys.executable, "-c", SCRIPT], cwd=ROOT, env=env, capture_output=True,
                           text=True, timeout=1200)
        assert r.returncode == 0, (r.stdout + r.stderr)[-4000:]
        out.append(r.stdout.splitlines())
    assert len(out[0]) == 28 + 8
    assert out[0] == out[1]
