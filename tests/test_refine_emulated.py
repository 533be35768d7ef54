"""The mixed kernel's finish of a block (refine_block) on the CPU emulation,
through each of its branches: no near pair, explicit rotations, binary64 sweeps.

Bars.  Overlaps of W's columns above binary32 resolution, relative: the first-order
step leaves E^2 and E x (largest angle) of the binary32 result's E <~ 3e-6, angles
below 1e-4 outside the near pairs, and an explicit rotation makes its pair orthogonal to
binary64: 1e-9.  Where three or more values lie close together the rotations of one
pass bring their overlaps back into each other, and so does one binary64 sweep: up
to E, 3e-6, among those columns.  V: unit columns to 1e-9.  W = A V: binary32 rotations,
3e-5 of the largest entry."""
import ctypes

import numpy as np
import pytest

import test_kernels_emulated  # noqa: F401  (puts tests/simt on the path)
from test_split_emulated import _build, _ld4, _ptr

pytestmark = pytest.mark.slow


@pytest.fixture(scope="module")
def emu(tmp_path_factory):
    return _build(tmp_path_factory.mktemp("refine"), "", ("refine_harness.cu",))


def _blocks():
    rng = np.random.default_rng(11)

    def block(q, s):
        p = len(s)
        u, v = np.linalg.qr(rng.standard_normal((q, p)))[0], np.linalg.qr(rng.standard_normal((p, p)))[0]
        return u @ np.diag(s) @ v.T

    def spread(p, lo=-3):
        return np.logspace(0, lo, p)
    out = {"none_24": (block(24, spread(24)), 0), "none_130x21": (block(130, spread(21)), 0)}
    s = spread(24)
    s[5] = s[4]
    out["pair_40x24"] = (block(40, s), 1)
    s = spread(24)
    s[8:11] = s[8]
    out["triple_40x24"] = (block(40, s), 1)
    s = spread(40, -5)
    s[3:9], s[20:26] = s[3], s[20]
    out["two_sixfold_60x40"] = (block(60, s), 1)
    s = spread(30, -4)
    s[6:10] = s[6] * (1 + 1e-7 * np.arange(4))
    out["four_1e-7_apart_33x30"] = (block(33, s), 1)
    s = spread(20, -4)
    s[6:10] = s[6] * (1 + 3e-3 * np.arange(4))
    out["four_3e-3_apart_140x20"] = (block(140, s), 1)
    out["degenerate_36"] = (block(36, np.repeat([1.0, 0.5, 0.25], 12)), 2)
    return out


@pytest.mark.parametrize("case", list(_blocks()))
def test_overlaps_end_below_the_bar(emu, case):
    A, branch = _blocks()[case]
    A = A.astype(np.float32)
    q, p = A.shape
    lw, lv = _ld4(q), _ld4(p)
    buf = np.zeros(p * (lw + lv) + 3 * p + 8, dtype=np.float32)
    buf = buf[(-buf.ctypes.data // 4) % 4:]
    buf[:p * lw].reshape(p, lw)[:, :q] = A.T
    buf[p * lw:p * (lw + lv)].reshape(p, lv)[:, :p] = np.eye(p)
    W, V, sig, out = np.zeros((p, q)), np.zeros((p, p)), np.zeros(p), np.zeros(4, dtype=np.int32)
    emu.hm_probe_refine(_ptr(buf), q, p, 1, _ptr(W), _ptr(V), _ptr(sig), _ptr(out))
    assert out[0] > 0 and out[1] > 0
    taken = 2 if out[1] > 1 or out[3] == 0 else out[2]
    assert taken == branch, out
    W, V, A = W.T, V.T, A.astype(np.float64)
    d = np.linalg.norm(W, axis=0)
    big = d > 3e-6 * d.max()
    G = np.abs(W.T @ W - np.diag(d * d))[np.ix_(big, big)] / np.outer(d[big], d[big])
    near = np.abs(d[big][:, None] ** 2 - d[big] ** 2) < 0.021 * np.maximum.outer(d[big] ** 2, d[big] ** 2)
    cluster = near.sum(axis=1) > 2              # a column and two others at least
    among = near & cluster[:, None] & cluster
    assert G[~among].max() <= 1e-9
    assert G.max() <= 3e-6
    assert np.abs(np.linalg.norm(V, axis=0) - 1).max() <= 1e-9
    assert np.abs(W - A @ V).max() <= 3e-5 * np.abs(A).max()
    ref = np.linalg.svd(A, compute_uv=False)
    assert np.abs(np.sort(d)[::-1] - ref).max() <= 3e-6 * ref[0]


# Blocks around the edge of the buffers (218 KB with one chain per SM, 109 KB with two): 1 = the
# wave layout fits, 2 = the unpadded one does, which keeps the sweeps in shared memory too.
@pytest.mark.parametrize("q,p,kb,want", [(163, 163, 218, 3), (169, 160, 218, 3), (165, 162, 218, 3), (166, 166, 218, 2),
                                         (168, 168, 218, 0), (118, 116, 109, 2), (126, 113, 109, 2), (117, 114, 109, 3),
                                         (120, 117, 109, 0)])
def test_layouts_at_the_edge_of_the_buffers(emu, q, p, kb, want):
    assert emu.hm_probe_layouts(q, p, ctypes.c_int64(kb * 1024)) == want


@pytest.mark.parametrize("chil,chir,polish", [(39, 38, 1), (38, 39, 1), (39, 38, 0), (40, 39, 1)])
def test_a_block_at_the_edge_of_the_buffer(emu, chil, chir, polish):
    """117 x 114 fits 109 KB without padding: no use of the scratch in global memory.  120 x 117 does not."""
    rng = np.random.default_rng(chil)
    theta = (rng.standard_normal((3 * chil, 3 * chir)) * np.logspace(0, -3, 3 * chir)).astype(np.float32)
    q, p = max(theta.shape), min(theta.shape)
    fits = q < 120
    X = None if fits else np.zeros(2 * q * p, dtype=np.float32)
    W, V, sig = np.zeros((p, q)), np.zeros((p, p)), np.zeros(p)
    emu.hm_probe_staged.argtypes = [ctypes.c_void_p, ctypes.c_int, ctypes.c_int, ctypes.c_void_p, ctypes.c_int] + \
        [ctypes.c_void_p] * 3
    code = emu.hm_probe_staged(_ptr(theta), chil, chir, None if fits else _ptr(X), polish, _ptr(W), _ptr(V), _ptr(sig))
    assert code > 0 and (code >= 1000) == bool(polish)
    # rows (l a) of theta against the block's order (a l), columns alike; W holds the transpose of a wide block
    A = theta.astype(np.float64).reshape(chil, 3, 3 * chir).transpose(1, 0, 2).reshape(3 * chil, 3 * chir)
    A = A.T if chir > chil else A
    W, V = W.T, V.T
    assert np.abs(W - A @ V).max() <= 3e-5 * np.abs(A).max()
    assert np.abs(np.linalg.norm(V, axis=0) - 1).max() <= (1e-9 if polish else 3e-7)
    d = np.linalg.norm(W, axis=0)
    G = np.abs(W.T @ W - np.diag(d * d)) / np.outer(d, d)
    assert G.max() <= 3e-6
    assert np.abs(np.sort(d)[::-1] - np.linalg.svd(A, compute_uv=False)).max() <= 3e-6 * d.max()


@pytest.mark.parametrize("n,chi,want", [(1, 3, 1), (1, 27, 1), (70, 27, 1), (1, 28, 8), (18, 64, 8), (19, 64, 4), (37, 256, 4),
                                        (38, 256, 2), (75, 256, 2), (76, 256, 1)])
def test_cluster_size_of_a_batch(emu, n, chi, want):
    assert emu.hm_probe_team(n, chi) == want
