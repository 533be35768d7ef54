"""Blocks that one build of the evolve kernels holds in shared memory and the other
does not (GPU tests): 204 and 218 KB with one chain per SM, 104 and 109 KB with two.
An unlabelled state of 33 bonds has one block of 99 x 99 a split, one of 40 bonds
120 x 120.  Alone (a cluster, or one CTA for a block beyond its buffer) and in
a batch wider than the GPU the steps differ, so the bits may; both agree with the
oracle: FP64 to 1e-10, the mixed forms to 1e-5."""
import numpy as np
import pytest

from oracle import measure as omeasure
from oracle import model as omodel
from oracle import mps as omps

pytestmark = pytest.mark.gpu


def _state(chi, n, seed):
    """A random right-canonical state with its centre on site 0."""
    rng = np.random.default_rng(seed)
    d = [min(3 ** i, 3 ** (n - i), chi) for i in range(n + 1)]
    ten = [rng.standard_normal((d[i], 3, d[i + 1])) for i in range(n)]
    for k in range(n - 1, 0, -1):
        q, r = np.linalg.qr(ten[k].reshape(d[k], -1).T)
        ten[k] = q.T.reshape(d[k], 3, d[k + 1]).copy()
        ten[k - 1] = np.einsum("asb,cb->asc", ten[k - 1], r)
    ten[0] /= np.linalg.norm(ten[0])
    return ten


@pytest.mark.parametrize("prec,chi,tol", [("HM_FP64", 33, 1e-10), ("HM_FP64", 40, 1e-10), ("HM_MIXED", 40, 1e-5),
                                          ("HM_MIXED32", 40, 1e-5)])
def test_alone_and_in_a_wide_batch(prec, chi, tol):
    import torch
    from paper_1910_09142_gb300 import binding as b
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    cfg = dict(beta=0.1, tau=0.05, chi_max=chi, cutoff=1e-12)
    p = b.params(Lx=4, two_W=0, **cfg, precision=getattr(b, prec), seed=1)
    other = b.params(Lx=2, two_W=0, beta=0.1, tau=0.1, chi_max=4, cutoff=1e-8, precision=getattr(b, prec), seed=1)
    state = _state(chi, 8, 5)
    ladder = omodel.Ladder(4, 0, 1.0, 1.0)
    steps, tau = omodel.trotter_steps(cfg["beta"], cfg["tau"])
    ops, gates = omodel.schedule(ladder, steps, tau, omodel.SCHEDULE_PLAIN)
    ref = omps.evolve(omps.MPS([t.copy() for t in state], 0), ops, gates, chi, cfg["cutoff"])
    want = omeasure.measure(ref, ladder.measured_bonds())
    ctx = b.Context(b.query_memory(p) + (sms + 8) * b.query_memory(other) + (8 << 20))
    try:
        got = []
        for n in (1, sms + 8):
            cid = ctx.init_chain(p)
            rest = [ctx.init_chain(other) for _ in range(n - 1)]
            ctx.set_mps(cid, state)
            ctx.evolve([cid] + rest)
            got.append(ctx.measure([cid], b.num_obs(p))[0])
            assert ctx.stats(cid)[5] == chi                     # the bond cap was reached
            for c in [cid] + rest:
                ctx.free_chain(c)
    finally:
        ctx.close()
    scale = np.abs(want).max()
    assert np.abs(got[0] - want).max() <= tol * scale
    assert np.abs(got[1] - want).max() <= tol * scale
