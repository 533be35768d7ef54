"""A chain's result does not depend on the CTAs that work on it (GPU tests).

The evolve kernels give a chain a cluster of 8, 4 or 2 CTAs in small batches,
one CTA in batches near the SM count, and half an SM above it.  The same chain
alone, in a batch of a third of the SMs, one short of the SMs, and wider than the
GPU: state, observables, outcomes and log p bit for bit, whole and in slices."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

CFGS = [dict(Lx=5, two_W=4, beta=0.4, tau=0.1, chi_max=96, cutoff=1e-10),      # several blocks of 16 columns and more
        dict(Lx=3, two_W=0, beta=0.4, tau=0.1, chi_max=20, cutoff=1e-10),      # fewer blocks than CTAs
        dict(Lx=1, two_W=2, beta=0.3, tau=0.1, chi_max=16, cutoff=0.0)]        # one bond at a time, no environment


@pytest.mark.parametrize("prec", ["HM_FP64", "HM_MIXED", "HM_MIXED32"])
@pytest.mark.parametrize("cfg", CFGS)
def test_results_do_not_depend_on_the_batch(cfg, prec):
    import torch
    from paper_1910_09142_gb300 import binding as b
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    p = b.params(**cfg, precision=getattr(b, prec), seed=6, chain_id=9)
    other = b.params(Lx=2, two_W=2, beta=0.2, tau=0.1, chi_max=12, cutoff=1e-8, precision=getattr(b, prec), seed=1)
    ctx = b.Context(b.query_memory(p) + (sms + 16) * b.query_memory(other) + (8 << 20))
    try:
        want = None
        for n, budget in [(1, 0), (1, 7), (sms // 12, 0), (sms // 3, 0), (sms // 3, 5), (sms - 1, 0), (sms + 8, 0)]:
            cid = ctx.init_chain(p)
            rest = [ctx.init_chain(other) for _ in range(n - 1)]
            ids = rest[: n // 2] + [cid] + rest[n // 2:]
            got = []
            for _ in range(2):
                left = ids
                while budget and left:
                    done = ctx.evolve_partial(left, budget)
                    left = [c for c, d in zip(left, done) if not d]
                if not budget:
                    ctx.evolve(ids)
                got += ctx.get_mps(cid) + [ctx.measure([cid], b.num_obs(p))]
                got += list(ctx.collapse([cid], b.num_env(p)))
                if rest:
                    ctx.collapse(rest, b.num_env(other))
            if want is None:
                want = got
            assert len(got) == len(want)
            assert all(np.array_equal(x, y) for x, y in zip(got, want)), (n, budget)
            for c in ids:
                ctx.free_chain(c)
    finally:
        ctx.close()
