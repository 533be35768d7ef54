"""The pieces of a split's decomposition on the CPU emulation, at the sizes
where they can go wrong: column counts and row counts around the register
tiles (4 rows a lane, 8 lanes a column, 4 columns a super-column, 32 rows a
chunk, 128 rows a product task), odd super-column counts, noise and degenerate
columns; the records of a split that does not fit shared memory; both forms
of theta.  References: numpy in binary64, and the oracle.

Bars.  Conversions: equal.  Orthonormality and orthogonality after the
binary64-accurate steps: the first-order step leaves E^2 and E x (largest
angle) of the binary32 result's E <~ 3e-6, angles below 1e-4 outside the near
pairs: 1e-9 (relative overlaps of columns above binary32 resolution).
W - A V: binary32 rotations, 3e-5 of the largest entry (the bar of the existing
Jacobi tests).  The orthonormalised V: 4 sqrt(p) eps."""
import ctypes

import numpy as np
import pytest

import test_kernels_emulated  # noqa: F401  (puts tests/simt on the path)
import build_emulated
from oracle import chain as ochain
from oracle import mps as omps
from paper_1910_09142_gb300 import binding
from test_kernels_emulated import Emu

pytestmark = pytest.mark.slow


def _build(tmp, head, probes):
    """The emulated library with `head` before every kernel source."""
    rewrite, old = build_emulated.rewrite, build_emulated.PROBES
    build_emulated.rewrite = lambda text: head + rewrite(text)
    build_emulated.PROBES = old + probes
    try:
        return ctypes.CDLL(build_emulated.build(str(tmp)))
    except FileNotFoundError as e:
        pytest.skip(str(e))
    finally:
        build_emulated.rewrite, build_emulated.PROBES = rewrite, old


@pytest.fixture(scope="module")
def emu(tmp_path_factory):
    return _build(tmp_path_factory.mktemp("split"), "", ("split_harness.cu",))


def _ptr(a):
    return ctypes.c_void_p(a.ctypes.data)


def _ld4(n):
    return (((n + 3) >> 2) | 1) * 4


def test_conversions_equal_the_casts(emu):
    rng = np.random.default_rng(1)
    d = rng.standard_normal(4000) * 10.0 ** rng.integers(-46, 40, 4000)
    f32 = rng.standard_normal(4000).astype(np.float32) * np.float32(10.0) ** rng.integers(-44, 37, 4000).astype(np.float32)
    special = [0.0, -0.0, np.inf, -np.inf, 1e-45, -1e-45, 1.17549435e-38, 3.4028235e38]
    ties = 1.0 + np.arange(-5, 6) * 2.0 ** -24 + np.array([0, 2.0 ** -40])[:, None]   # halves between binary32 values
    d = np.concatenate([d, special, ties.reshape(-1), [3.4028235677973366e38, 1e300, 2.0 - 2.0 ** -26]])
    g = np.concatenate([f32, np.array(special, dtype=np.float32)])
    g = np.resize(g, len(d)).astype(np.float32)
    out, wide = np.zeros(len(d), dtype=np.float32), np.zeros(len(d))
    emu.hm_probe_convert(_ptr(d), _ptr(out), _ptr(g), _ptr(wide), len(d))
    with np.errstate(over="ignore"):
        want = d.astype(np.float32)
    assert np.array_equal(out.view(np.uint32), want.view(np.uint32))
    assert np.array_equal(wide.view(np.uint64), g.astype(np.float64).view(np.uint64))


def test_warp_truncation_matches_the_oracle(emu):
    emu.hm_probe_warp_trunc.argtypes = [ctypes.c_void_p, ctypes.c_int, ctypes.c_int, ctypes.c_double, ctypes.c_void_p]
    rng = np.random.default_rng(3)
    cases = [(np.sort(np.exp(rng.uniform(-12, 0, n)))[::-1], int(rng.integers(1, 130)), float(10 ** rng.uniform(-14, -2)))
             for n in list(range(1, 40)) + [63, 64, 65, 127, 128, 129, 400]]
    mult = np.sort(np.repeat([1.0, 0.3, 0.3 * (1 - 5e-9), 0.1, 1e-3], [1, 3, 2, 5, 3]))[::-1]
    cases += [(mult, chi, 1e-12) for chi in range(1, len(mult) + 1)]
    cases += [(np.array([0.7]), 4, 0.0), (np.array([1.0, 0.5, 0.0, 0.0]), 4, 0.0)]
    for s, chi, cut in cases:
        s = np.ascontiguousarray(s)
        out = np.zeros(3)
        emu.hm_probe_warp_trunc(_ptr(s), len(s), chi, cut, _ptr(out))
        k = omps.truncation_rank(s, chi, cut)
        assert int(out[0]) == k, (len(s), chi, cut)
        assert np.allclose(out[1:], [np.sum(s[:k] ** 2), np.sum(s[k:] ** 2)], rtol=1e-13, atol=0)


def _blocks():
    rng = np.random.default_rng(7)

    def graded(q, p, lo):
        u, v = np.linalg.qr(rng.standard_normal((q, p)))[0], np.linalg.qr(rng.standard_normal((p, p)))[0]
        return u @ np.diag(np.logspace(0, lo, p)) @ v.T
    out = {"%dx%d" % (q, p): graded(q, p, -5) for q, p in
           [(1, 1), (5, 3), (12, 12), (16, 16), (33, 17), (31, 31), (64, 20), (65, 33), (97, 18), (128, 19), (129, 21)]}
    out["degenerate"] = np.linalg.qr(rng.standard_normal((36, 36)))[0] @ np.diag(np.repeat([1.0, 0.5, 0.25], 12)) @ \
        np.linalg.qr(rng.standard_normal((36, 36)))[0].T
    noise = graded(40, 24, -3)
    noise[:, 12:] = noise[:, :12] @ rng.standard_normal((12, 12))      # rank 12: noise columns after the sweeps
    out["rank_deficient"] = noise
    out["null_columns"] = np.hstack([graded(30, 10, -2), np.zeros((30, 8))])
    return out


@pytest.mark.parametrize("case", list(_blocks()))
def test_binary32_block_to_binary64_accuracy(emu, case):
    A = _blocks()[case].astype(np.float32)
    q, p = A.shape
    W, V = np.zeros((p, _ld4(q)), dtype=np.float32), np.zeros((p, _ld4(p)), dtype=np.float32)
    W[:, :q], V[:, :p] = A.T, np.eye(p)
    W64, V64, out = np.zeros((p, q)), np.zeros((p, p)), np.zeros(2, dtype=np.int32)
    emu.hm_probe_svd(_ptr(W), q, p, _ptr(V), _ptr(W64), _ptr(V64), _ptr(out))
    assert 1 <= out[0] <= 30
    W64, V64, A = W64.T, V64.T, A.astype(np.float64)
    assert np.abs(W64 - A @ V64).max() <= 3e-5 * np.abs(A).max()
    assert np.abs(np.linalg.norm(V64, axis=0) - 1).max() <= 1e-9
    assert np.abs(V64.T @ V64 - np.eye(p)).max() <= 3e-5
    sv, ref = np.sort(np.linalg.norm(W64, axis=0))[::-1], np.linalg.svd(A, compute_uv=False)
    assert np.abs(sv - ref).max() <= 3e-6 * ref[0]
    d = np.linalg.norm(W64, axis=0)
    big = d > 3e-6 * d.max()
    G = np.abs(W64.T @ W64 - np.diag(d * d))[np.ix_(big, big)] / np.outer(d[big], d[big])
    if out[1] <= 2 * p:                     # the explicit pairs were done (else the kernel sweeps in binary64)
        assert G.max() <= (1e-9 if out[1] == 0 else 2e-6)


@pytest.mark.parametrize("p", [6, 7, 8, 9, 11, 12, 15, 16, 31, 32, 33, 60, 65, 130])
def test_orthonormalisation_reaches_binary64(emu, p):
    rng = np.random.default_rng(p)
    Q = np.linalg.qr(rng.standard_normal((p, p)))[0]
    V = np.zeros((p, _ld4(p)), dtype=np.float32)
    V[:, :p] = Q.T * (1 + 1e-5 * rng.random((p, 1))) + 1e-6 * rng.standard_normal((p, p)) / np.sqrt(p)
    V64 = np.zeros((p, p))
    start = V[:, :p].astype(np.float64)
    emu.hm_probe_ortho(_ptr(V), p, _ptr(V64))
    assert np.abs(V64 @ V64.T - np.eye(p)).max() <= 4 * np.sqrt(p) * 2.3e-16
    assert np.abs(V64 - start).max() <= 2e-5


def _check_one_sample(lib, prec):
    P, vp, i32, i64 = ctypes.POINTER, ctypes.c_void_p, ctypes.c_int32, ctypes.c_int64
    lib.hm_create.argtypes = [P(vp), ctypes.c_int, vp, ctypes.c_size_t, vp]
    lib.hm_destroy.argtypes = [vp]
    lib.hm_init_chain.argtypes = [vp, P(binding.Params), vp, P(i64)]
    lib.hm_evolve.argtypes = [vp, P(i64), i32]
    lib.hm_measure_cluster.argtypes = [vp, P(i64), i32, vp, i32]
    lib.hm_collapse.argtypes = [vp, P(i64), i32, vp, vp]
    lib.hm_last_error.argtypes = [vp]
    lib.hm_last_error.restype = ctypes.c_char_p
    cfg = dict(Lx=2, two_W=2, J_leg=1.0, J_rung=0.7, beta=0.2, tau=0.1, chi_max=16, cutoff=1e-12)
    e = Emu(lib)
    p = binding.params(**cfg, seed=3, chain_id=1, precision=getattr(binding, prec))
    cid = e.init(p)
    obs, env, lp = e.sample(cid, p)
    r = ochain.HybridChain(seed=3, chain_id=1, **cfg).sample()
    tol = 1e-10 if prec == "HM_FP64" else 1e-5
    assert np.abs(obs - r["obs"]).max() <= tol * max(1.0, np.abs(r["obs"]).max())
    assert env == r["env_out"] and abs(lp - r["logp"]) < 10 * tol
    e.close()


@pytest.mark.parametrize("prec", ["HM_FP64", "HM_MIXED", "HM_MIXED32"])
def test_records_in_the_workspace_and_tiled_theta(tmp_path, prec):
    """Every split with more records than shared memory holds (limit 2
    instead of 14), and theta always in tiles: one sample against the oracle."""
    lib = _build(tmp_path, "#define HM_SH_BLK 2\n#define HM_THETA_DIRECT 0.0\n", ())
    _check_one_sample(lib, prec)


@pytest.mark.parametrize("prec,smem", [("HM_MIXED", "kMaxSharedOptIn"), ("HM_MIXED", "0"), ("HM_MIXED32", "0")])
def test_blocks_beyond_shared_memory(tmp_path, prec, smem):
    """Every block of two columns or more takes the staged path, with two columns
    or more a staged block (as for bond caps up to about 2000) or one
    (above): one sample against the oracle."""
    lib = _build(tmp_path, "#define HM_WAVE_SMEM 48\n#define HM_STAGED_SMEM %s\n" % smem, ())
    _check_one_sample(lib, prec)


@pytest.mark.parametrize("prec", ["HM_FP64", "HM_MIXED"])
def test_nothing_is_read_that_was_not_written(emu, prec):
    """A split writes only the entries its charges allow.  With an arena full
    of NaN the state, susceptibility, observables, outcomes and log p of two
    samples are the bits they are with an arena of zeros."""
    P, vp, i32, i64 = ctypes.POINTER, ctypes.c_void_p, ctypes.c_int32, ctypes.c_int64
    for name, args in {"hm_create": [P(vp), ctypes.c_int, vp, ctypes.c_size_t, vp], "hm_destroy": [vp],
                       "hm_init_chain": [vp, P(binding.Params), vp, P(i64)], "hm_evolve": [vp, P(i64), i32],
                       "hm_measure_cluster": [vp, P(i64), i32, vp, i32], "hm_collapse": [vp, P(i64), i32, vp, vp],
                       "hm_measure_susceptibility": [vp, P(i64), i32, vp],
                       "hm_get_mps": [vp, i64, P(i32), i32, vp, ctypes.c_size_t, P(i32), P(ctypes.c_size_t)],
                       "hm_last_error": [vp]}.items():
        getattr(emu, name).argtypes = args
    emu.hm_last_error.restype = ctypes.c_char_p
    cfg = dict(Lx=3, two_W=2, J_leg=1.0, J_rung=0.7, beta=0.2, tau=0.1, chi_max=20, cutoff=1e-10)
    p = binding.params(**cfg, seed=4, chain_id=2, precision=getattr(binding, prec))
    runs = []
    for byte in (0, 255):
        e = Emu(emu)
        base = -e.mem.ctypes.data % 256
        e.mem[base + 256:] = byte                 # the context's error word lies in front
        cid = e.init(p)
        got = []
        for _ in range(2):
            e.evolve(cid)
            got += [t.copy() for t in e.mps(cid)]
            chi = np.zeros(2)
            e._ok(emu.hm_measure_susceptibility(e.h, e._ids(cid), 1, _ptr(chi)))
            env, lp = None, None
            got += [chi, e.measure(cid, p)]
            env, lp = e.collapse(cid, p)
            got += [np.array(env), np.array(lp)]
        runs.append(got)
        e.close()
    assert all(np.isfinite(x).all() and np.array_equal(x, y) for x, y in zip(*runs))
