"""States handed in by hm_set_mps that are not normalised or not finite, on the
CPU emulation of the kernels."""
import ctypes

import numpy as np
import pytest

import test_kernels_emulated  # noqa: F401  (puts tests/simt on the path)
import build_emulated
from paper_1910_09142_gb300 import binding
from test_kernels_emulated import Emu

pytestmark = pytest.mark.slow


@pytest.fixture(scope="module")
def emu(tmp_path_factory):
    try:
        lib = ctypes.CDLL(build_emulated.build(str(tmp_path_factory.mktemp("range"))))
    except FileNotFoundError as e:
        pytest.skip(str(e))
    P, vp, i32, i64 = ctypes.POINTER, ctypes.c_void_p, ctypes.c_int32, ctypes.c_int64
    for name, args in {"hm_create": [P(vp), ctypes.c_int, vp, ctypes.c_size_t, vp], "hm_destroy": [vp],
                       "hm_init_chain": [vp, P(binding.Params), vp, P(i64)],
                       "hm_set_mps": [vp, i64, P(i32), i32, vp, ctypes.c_size_t, i32, i32],
                       "hm_apply_ops": [vp, i64, P(i32), i32], "hm_last_error": [vp],
                       "hm_get_mps": [vp, i64, P(i32), i32, vp, ctypes.c_size_t, P(i32), P(ctypes.c_size_t)]}.items():
        getattr(lib, name).argtypes = args
    lib.hm_last_error.restype = ctypes.c_char_p
    return lib


def _apply(emu, prec, tensors, ops):
    """Return code of hm_apply_ops on a chain that holds `tensors`, and the state after it."""
    P32 = ctypes.POINTER(ctypes.c_int32)
    e = Emu(emu)
    cid = e.init(binding.params(Lx=len(tensors) // 2, two_W=0, beta=0.2, tau=0.1, chi_max=9, cutoff=0.0, seed=1,
                                precision=getattr(binding, prec)))
    dims = np.array([t.shape[0] for t in tensors] + [1], dtype=np.int32)
    buf = np.concatenate([t.reshape(-1) for t in tensors])
    e._ok(emu.hm_set_mps(e.h, cid, dims.ctypes.data_as(P32), len(tensors), buf.ctypes.data_as(ctypes.c_void_p),
                         len(buf), 0, 0))
    ops = np.array(ops, dtype=np.int32)
    rc = emu.hm_apply_ops(e.h, cid, ops.ctypes.data_as(P32), len(ops))
    state = e.mps(cid) if rc == 0 else None
    e.close()
    return rc, state


@pytest.mark.parametrize("prec", ["HM_FP64", "HM_MIXED", "HM_MIXED32"])
@pytest.mark.parametrize("exact", [1, 0])
@pytest.mark.parametrize("where", ["all", "one"])
def test_a_nan_is_an_error_of_any_split(emu, prec, exact, where):
    rng = np.random.default_rng(2)
    ten = [rng.standard_normal(s) for s in ((1, 3, 3), (3, 3, 9), (9, 3, 3), (3, 3, 1))]
    if where == "all":
        ten[1][:] = np.nan
    else:
        ten[1][0, 1, 2] = np.nan
    assert _apply(emu, prec, ten, [[1, 0, 1, exact]])[0] == binding.HM_ERR_NUMERIC


def _centre_pair(M):
    """A four-site state whose middle pair has theta = M (9 x 9)."""
    return [np.eye(3).reshape(1, 3, 3), np.ascontiguousarray(M).reshape(3, 3, 9), np.eye(9).reshape(9, 3, 3),
            np.eye(3).reshape(3, 3, 1)]


@pytest.mark.parametrize("prec", ["HM_FP64", "HM_MIXED", "HM_MIXED32"])
@pytest.mark.parametrize("top", [1e-6, 1.0, 1e5, 1e7, 1e12])
def test_a_graded_state_of_any_norm_splits(emu, prec, top):
    """Columns 1e-14 long that overlap with one of length `top`: squared norms up
    to 1e52 apart.  An exact move gives theta back, in orthonormal left vectors.
    Bar: 2e-6 of the largest entry, the mixed forms' binary32 theta (FP64: 1e-13)."""
    M = np.diag(np.full(9, 1e-14)) * (1 + np.arange(9.0)[:, None])
    M[0] = 1e-14
    M[0, 0] = top
    rc, state = _apply(emu, prec, _centre_pair(M), [[1, 0, 1, 1]])
    assert rc == 0
    U, R = state[1].reshape(9, -1), state[2].reshape(-1, 9)
    tol = 1e-13 if prec == "HM_FP64" else 2e-6
    assert np.abs(U @ R - M).max() <= tol * np.abs(M).max()
    big = np.linalg.norm(R, axis=1) > 1e-6 * top
    assert np.abs(np.linalg.norm(U[:, big], axis=0) - 1).max() <= tol


@pytest.mark.parametrize("prec", ["HM_FP64", "HM_MIXED"])
@pytest.mark.parametrize("scale", [1e-30, 1e-20, 1e-12, 1.0, 1e12, 3e18, 1e20, 1e37])
@pytest.mark.parametrize("kind", ["random", "graded"])
def test_left_vectors_are_orthonormal_at_any_scale(emu, prec, scale, kind):
    """The sweeps in binary32 leave columns shorter than 1e-15 alone and cannot sum
    squares above 1e38: binary64 sweeps take such blocks.  Bars: U R = theta to
    2e-6 of its largest entry (the mixed form's binary32 theta; FP64 1e-13), the
    vectors kept by an exact move orthonormal to 1e-9 (no two values are near)."""
    rng = np.random.default_rng(5)
    M = rng.standard_normal((9, 9))
    if kind == "graded":
        q = np.linalg.qr(rng.standard_normal((2, 9, 9)))[0]
        M = q[0] @ np.diag(np.logspace(0, -12, 9)) @ q[1].T
    M = M * scale
    rc, state = _apply(emu, prec, _centre_pair(M), [[1, 0, 1, 1]])
    assert rc == 0
    U, R = state[1].reshape(9, -1), state[2].reshape(-1, 9)
    assert np.abs(U @ R - M).max() <= (1e-13 if prec == "HM_FP64" else 2e-6) * np.abs(M).max()
    assert np.abs(U.T @ U - np.eye(U.shape[1])).max() <= 1e-9


def test_explicit_ops_on_a_labelled_chain_are_checked_too(emu):
    """Exact ops with bond gates do not keep the norm: weak gates entangle the
    pairs, then a rung's exp(10 S.S) takes up to e^10 an op, four times."""
    e = Emu(emu)
    p = binding.params(Lx=2, two_W=0, J_leg=0.5, J_rung=-40.0, beta=1.0, tau=0.5, chi_max=9, cutoff=0.0, seed=2,
                       precision=binding.HM_MIXED)
    cid = e.init(p, env=[0, 1, 1, 2])
    ops = np.array([[1, 3, 1, 0], [2, 3, 0, 0], [1, 3, 0, 0], [0, 3, 1, 0], [1, 3, 1, 0], [2, 3, 0, 0], [1, 3, 0, 0]] +
                   [[0, 2, 1, 1]] * 5 + [[1, 0, 1, 1]], dtype=np.int32)
    e._ok(emu.hm_apply_ops(e.h, cid, ops.ctypes.data_as(ctypes.POINTER(ctypes.c_int32)), len(ops)))
    A = e.mps(cid)
    assert np.linalg.norm(A[2]) > 1e19
    U = A[1].reshape(-1, A[1].shape[2])
    assert U.shape[1] >= 5 and np.abs(U.T @ U - np.eye(U.shape[1])).max() <= 1e-9
    e.close()
