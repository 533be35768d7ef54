"""A state that no split can keep a value of ends its chain with an error (GPU
tests): in a cluster of 8, 4 and 2 CTAs, one CTA, and half an SM; the other
chains of the batch go on."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["HM_FP64", "HM_MIXED", "HM_MIXED32"])
def test_zero_and_nan_states_report_an_error(prec):
    import torch
    from paper_1910_09142_gb300 import binding as b
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    p = b.params(Lx=2, two_W=0, beta=0.4, tau=0.1, chi_max=9, cutoff=1e-12, precision=getattr(b, prec), seed=3)
    ctx = b.Context((sms + 16) * b.query_memory(p) + (8 << 20))
    try:
        want = None
        for n in (1, sms // 12, sms // 6, sms // 3, sms - 1, sms + 8):
            for value in (0.0, np.nan):
                good = [ctx.init_chain(p) for _ in range(n - 1)]
                bad = ctx.init_chain(p)
                ctx.set_mps(bad, [np.full((1, 3, 1), value)] * 4)
                ctx.evolve(good[: n // 2] + [bad] + good[n // 2:])
                with pytest.raises(b.HmError) as err:
                    ctx.stats(bad)
                assert err.value.code == b.HM_ERR_NUMERIC
                obs = ctx.measure([bad] + good, b.num_obs(p))
                assert np.isnan(obs[0]).all()
                want = obs[1] if want is None and good else want
                assert all(np.array_equal(o, want) for o in obs[1:])
                for c in good + [bad]:
                    ctx.free_chain(c)
    finally:
        ctx.close()
