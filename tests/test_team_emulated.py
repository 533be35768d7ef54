"""Teams (clusters of CTAs on one chain) of the evolve kernels on the CPU.

``tests/simt/team_runtime.cpp`` runs the CTAs of a team side by side and
decides who goes first between two team barriers.  A failed split must end the
launch with its error, whatever the CTAs' order: a warp that reads the chain's
status late must not leave its CTA at another barrier than the rest.  And a team
must give the bits that one CTA gives, in every order.  Each run is a process
of its own, because barriers that do not match abort it."""
import os
import re
import shutil
import subprocess
import sys

import pytest

import test_kernels_emulated  # noqa: F401  (puts tests/simt on the path)
import build_emulated

pytestmark = pytest.mark.slow

HERE = os.path.dirname(os.path.abspath(__file__))
SIMT = os.path.join(HERE, "simt")


@pytest.fixture(scope="module")
def libs(tmp_path_factory):
    """The emulated library with its one-CTA-per-SM evolve launches as teams of 2 (and of 1)."""
    out = {}
    for team in (1, 2):
        tmp = str(tmp_path_factory.mktemp("team%d" % team))
        rewrite, host = build_emulated.rewrite, os.path.join(tmp, "simt")
        shutil.copytree(SIMT, host)
        shutil.copy(os.path.join(SIMT, "team_runtime.cpp"), os.path.join(host, "simt_runtime.cpp"))

        def teams(text):
            text = re.sub(r"simt::launch\(b\.n, (.*?), \[&\] \{ (evolve_fp64_wide_kernel|evolve_mixed_kernel)\((.*?), 1\); \}\)",
                          r"simt::launch_team(%d, b.n * %d, \1, [&] { \2(\3, %d); })" % (team, team, team), rewrite(text))
            return '#include "%s"\n' % os.path.join(SIMT, "team_prelude.h") + text
        old_here = build_emulated.HERE
        build_emulated.rewrite, build_emulated.HERE = teams, host
        try:
            out[team] = build_emulated.build(tmp)
        except FileNotFoundError as e:
            pytest.skip(str(e))
        finally:
            build_emulated.rewrite, build_emulated.HERE = rewrite, old_here
        text = "".join(open(os.path.join(tmp, f)).read() for f in ("hm_fp64.cpp", "hm_mixed.cpp"))
        assert text.count("simt::launch_team(%d" % team) == 2
    return out


PRELUDE = """
import ctypes, sys
import numpy as np
sys.path[:0] = [%r, %r]
from test_kernels_emulated import Emu
from paper_1910_09142_gb300 import binding
lib = ctypes.CDLL(sys.argv[1])
P, vp, i32, i64 = ctypes.POINTER, ctypes.c_void_p, ctypes.c_int32, ctypes.c_int64
for name, args in {"hm_create": [P(vp), ctypes.c_int, vp, ctypes.c_size_t, vp], "hm_destroy": [vp],
                   "hm_init_chain": [vp, P(binding.Params), vp, P(i64)], "hm_evolve": [vp, P(i64), i32],
                   "hm_evolve_partial": [vp, P(i64), i32, i32, vp],
                   "hm_measure_cluster": [vp, P(i64), i32, vp, i32], "hm_collapse": [vp, P(i64), i32, vp, vp],
                   "hm_set_mps": [vp, i64, P(i32), i32, vp, ctypes.c_size_t, i32, i32],
                   "hm_chain_stats": [vp, i64, vp],
                   "hm_get_mps": [vp, i64, P(i32), i32, vp, ctypes.c_size_t, P(i32), P(ctypes.c_size_t)],
                   "hm_last_error": [vp]}.items():
    getattr(lib, name).argtypes = args
lib.hm_last_error.restype = ctypes.c_char_p
prec = getattr(binding, sys.argv[2])
""" % (HERE, os.path.dirname(HERE))

FAILED_SPLIT = PRELUDE + """
cfg = dict(Lx=2, two_W=0, J_leg=1.0, J_rung=0.7, beta=0.2, tau=0.1, chi_max=4, cutoff=1e-12)
p = binding.params(**cfg, seed=3, precision=prec)
for value in (0.0, np.nan):
    e = Emu(lib)
    cid = e.init(p)
    dims = np.ones(5, dtype=np.int32)
    buf = np.full(12, value)
    e._ok(lib.hm_set_mps(e.h, cid, dims.ctypes.data_as(P(i32)), 4, buf.ctypes.data_as(vp), 12, 0, 0))
    e._ok(lib.hm_evolve(e.h, e._ids(cid), 1))
    st = np.zeros(12)
    rc = lib.hm_chain_stats(e.h, cid, st.ctypes.data_as(vp))
    assert rc == -4, rc                                   # HM_ERR_NUMERIC
    assert st[7] <= 1, st                                 # the chain stopped at its first truncating split
    e.close()
"""

SAMPLE = PRELUDE + """
cfg = dict(Lx=2, two_W=2, J_leg=1.0, J_rung=0.7, beta=0.2, tau=0.1, chi_max=16, cutoff=1e-12)
p = binding.params(**cfg, seed=3, chain_id=1, precision=prec)
e = Emu(lib)
cid = e.init(p)
done = np.zeros(1, dtype=np.int32)
while not done[0]:
    e._ok(lib.hm_evolve_partial(e.h, e._ids(cid), 1, 9, done.ctypes.data_as(vp)))
got = [t.tobytes() for t in e.mps(cid)] + [e.measure(cid, p).tobytes()]
env, lp = e.collapse(cid, p)
print(hash((tuple(got), tuple(env), lp)))
"""


def _run(lib, script, prec, first):
    env = dict(os.environ, SIMT_TEAM_FIRST=str(first), PYTHONHASHSEED="0")
    return subprocess.run([sys.executable, "-c", script, lib, prec], capture_output=True, text=True, env=env)


@pytest.mark.parametrize("prec", ["HM_FP64", "HM_MIXED"])
@pytest.mark.parametrize("first", [0, 1, 40, 511])
def test_a_failed_split_ends_the_team(libs, prec, first):
    r = _run(libs[2], FAILED_SPLIT, prec, first)
    assert r.returncode == 0, r.stderr[-2000:]


@pytest.mark.parametrize("prec", ["HM_FP64", "HM_MIXED"])
def test_a_team_gives_the_bits_of_one_cta(libs, prec):
    runs = [_run(libs[1], SAMPLE, prec, 0)] + [_run(libs[2], SAMPLE, prec, k) for k in (0, 3, 700)]
    assert all(r.returncode == 0 for r in runs), [r.stderr[-800:] for r in runs]
    assert len({r.stdout for r in runs}) == 1 and runs[0].stdout.strip()
