"""The charge-block transfers of the measurement, the susceptibility and the
collapse (hm_transfer.cuh) on the CPU emulation, against the oracle: states
with charge labels in both frames, states without labels (one run a bond),
and a state whose legs are out of place (a SWAP applied by an explicit op
list), where an environment's charge shift is not the usual one.

Binary64 throughout; the oracle contracts the same tensors in another order,
so the bar is the kernels' 1e-10 relative."""
import ctypes

import numpy as np
import pytest

from oracle import chain as ochain
from oracle import collapse as ocollapse
from oracle import measure as omeasure
from oracle import mps as omps
from paper_1910_09142_gb300 import binding
from test_kernels_emulated import Emu, emu  # noqa: F401

pytestmark = pytest.mark.slow

BASE = dict(J_leg=1.0, J_rung=0.7, tau=0.1, cutoff=1e-12)
TOL = 1e-10


def _chi(e, lib, cid):
    out = np.zeros(2)
    e._ok(lib.hm_measure_susceptibility(e.h, e._ids(cid), 1, out.ctypes.data_as(ctypes.c_void_p)))
    return out


def _close(a, b):
    b = np.asarray(b, dtype=float)
    return np.abs(np.asarray(a) - b).max() <= TOL * max(1.0, np.abs(b).max())


def _region(ref):
    return sorted({k for i, j, _ in ref.meas_bonds for k in (i, j)})


@pytest.mark.parametrize("zx", [True, False])
@pytest.mark.parametrize("cfg", [dict(Lx=3, two_W=2, beta=0.2, chi_max=24), dict(Lx=3, two_W=0, beta=0.4, chi_max=9),
                                 dict(Lx=2, two_W=4, beta=0.2, chi_max=12)])
def test_labelled_states(emu, cfg, zx):  # noqa: F811
    """Two samples (the second starts in the S^x frame under the alternating
    schedule): observables, susceptibility, outcomes and log p."""
    full = dict(BASE, **cfg)
    e = Emu(emu)
    p = binding.params(**full, seed=2, chain_id=3, basis_zx=zx)
    cid = e.init(p)
    ref = ochain.HybridChain(seed=2, chain_id=3, basis_zx=zx, **full)
    for _ in range(2):
        e.evolve(cid)
        st = ref.evolve()
        assert _close(e.measure(cid, p), omeasure.measure(st, ref.meas_bonds))
        chi, raw = omeasure.susceptibility(st, ref.ladder, _region(ref), full["beta"])
        assert _close(_chi(e, emu, cid), [chi, raw])
        env, lp = e.collapse(cid, p)
        r = ref.sample()
        assert env == r["env_out"] and abs(lp - r["logp"]) < 1e-9
    e.close()


def _right_canonical(dims, seed):
    rng = np.random.default_rng(seed)
    n = len(dims) - 1
    st = omps.MPS([rng.standard_normal((dims[k], 3, dims[k + 1])) for k in range(n)], centre=n - 1)
    for k in range(n - 1, 0, -1):
        omps.move_left(st, k)
    st.tensors[0] /= np.linalg.norm(st.tensors[0])
    return st


def test_states_without_labels(emu):  # noqa: F811
    """hm_set_mps drops the charge labels: every bond is one run."""
    cfg = dict(BASE, Lx=3, two_W=2, beta=0.2, chi_max=16)
    e = Emu(emu)
    p = binding.params(**cfg, seed=2, chain_id=3)
    cid = e.init(p)
    ref = ochain.HybridChain(seed=2, chain_id=3, **cfg)
    n = ref.ladder.n_sites
    dims = [1, 3, 5, 7, 11, 6, 7, 3, 1][: n + 1]
    assert len(dims) == n + 1
    st = _right_canonical(dims, 4)
    d = np.array([t.shape[0] for t in st.tensors] + [1], dtype=np.int32)
    buf = np.concatenate([t.reshape(-1) for t in st.tensors])
    emu.hm_set_mps.argtypes = [ctypes.c_void_p, ctypes.c_int64, ctypes.POINTER(ctypes.c_int32), ctypes.c_int32,
                               ctypes.c_void_p, ctypes.c_size_t, ctypes.c_int32, ctypes.c_int32]
    e._ok(emu.hm_set_mps(e.h, cid, d.ctypes.data_as(ctypes.POINTER(ctypes.c_int32)), n,
                         buf.ctypes.data_as(ctypes.c_void_p), len(buf), 0, 1))
    assert _close(e.measure(cid, p), omeasure.measure(st, ref.meas_bonds))
    chi, raw = omeasure.susceptibility(st, ref.ladder, _region(ref), cfg["beta"])
    assert _close(_chi(e, emu, cid), [chi, raw])
    env, lp = e.collapse(cid, p)
    out, logp, _ = ocollapse.collapse(st, ref.ladder, ocollapse.BASIS_Z, 2, 3, 0)
    assert env == list(out) and abs(lp - logp) < 1e-9
    e.close()


def test_legs_out_of_place(emu):  # noqa: F811
    """A SWAP of a cluster site and its ancilla leaves a physical position
    with an ancilla's leg: the kernels still contract the stored tensors."""
    cfg = dict(BASE, Lx=3, two_W=2, beta=0.2, chi_max=24)
    e = Emu(emu)
    p = binding.params(**cfg, seed=2, chain_id=3)
    cid = e.init(p)
    ref = ochain.HybridChain(seed=2, chain_id=3, **cfg)
    e.evolve(cid)
    site = ref.ladder.cluster_sites[0]
    ops = np.array([[k, 0, 1, 1] for k in range(site)] + [[site, 1, 0, 0]] +
                   [[k, 0, 0, 1] for k in range(site - 1, -1, -1)], dtype=np.int32)
    emu.hm_apply_ops.argtypes = [ctypes.c_void_p, ctypes.c_int64, ctypes.c_void_p, ctypes.c_int32]
    e._ok(emu.hm_apply_ops(e.h, cid, ops.ctypes.data_as(ctypes.c_void_p), len(ops)))
    st = omps.MPS(e.mps(cid), 0)
    assert _close(e.measure(cid, p), omeasure.measure(st, ref.meas_bonds))
    chi, raw = omeasure.susceptibility(st, ref.ladder, _region(ref), cfg["beta"])
    assert _close(_chi(e, emu, cid), [chi, raw])
    e.close()


@pytest.mark.parametrize("prec", ["HM_FP64", "HM_MIXED"])
def test_a_gate_that_breaks_the_labels(emu, prec):  # noqa: F811
    """A bond gate on a cluster site and its ancilla breaks the charge rule: the
    chain drops its labels first, and its tensors' forbidden entries, which
    no split wrote, have to be zeros by then.  The arena starts full of NaN."""
    from oracle import model
    cfg = dict(BASE, Lx=3, two_W=2, beta=0.2, chi_max=24)
    e = Emu(emu)
    e.mem[-e.mem.ctypes.data % 256 + 256:] = 255        # behind the context's error word
    p = binding.params(**cfg, seed=2, chain_id=3, precision=getattr(binding, prec))
    cid = e.init(p)
    ref = ochain.HybridChain(seed=2, chain_id=3, **cfg)
    e.evolve(cid)
    before = [t.copy() for t in e.mps(cid)]
    site = ref.ladder.cluster_sites[0]
    ops = np.array([[k, 0, 1, 1] for k in range(site)] + [[site, 2, 0, 0]] +
                   [[k, 0, 0, 1] for k in range(site - 1, -1, -1)], dtype=np.int32)
    emu.hm_apply_ops.argtypes = [ctypes.c_void_p, ctypes.c_int64, ctypes.c_void_p, ctypes.c_int32]
    e._ok(emu.hm_apply_ops(e.h, cid, ops.ctypes.data_as(ctypes.c_void_p), len(ops)))
    st = omps.MPS(before, 0)
    for k in range(site):
        omps.move_right(st, k)
    omps.split(st, site, model.bond_gate(0.5 * 0.1 * 0.7), model.ABSORB_L, 24, 1e-12)   # tau / 2 on a rung
    for k in range(site, 0, -1):
        omps.move_left(st, k)
    a, b = omps.MPS(e.mps(cid)).to_dense(), st.to_dense()
    assert np.abs(a - np.sign(a @ b) * b).max() < (1e-10 if prec == "HM_FP64" else 1e-5)
    e.close()
