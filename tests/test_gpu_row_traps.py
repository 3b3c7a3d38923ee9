"""Row sweeps of complex64 that hold an instance's trap factors in registers
(rows of 64, 256 and 512 points): runs of consecutive rows that begin and end inside
an instance or cross several, ragged last tiles, instances with their own trap.
"""
import numpy as np
import pytest

import gpe_inputs as gi

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,batch", [((2, 512), 1), ((4, 512), 701), ((64, 512), 67), ((512, 4), 1), ((2, 256), 1203),
                                     ((256, 256), 5), ((2, 4, 256), 301), ((4, 8, 512), 97), ((2, 64), 2051),
                                     ((64, 64, 64), 3)],
                         ids=lambda v: "x".join(map(str, v)) if isinstance(v, tuple) else str(v))
def test_instances_with_their_own_traps_match_the_oracle(orc, n, batch):
    """Same bound as the batches of shorter rows: 2e-5 after 5 steps."""
    import torch
    import paper_2301_08275_gb300 as gpe
    nd = len(n)
    rng = np.random.default_rng(batch)
    g_each = rng.uniform(0, 80, size=batch)
    gam_each = rng.uniform(0.5, 3.0, size=(batch, 3))
    lo, length = (-6.0, -5.0, -4.0)[:nd], (12.0, 10.0, 8.0)[:nd]

    def spec(b):
        return gi.Spec(n=n, lo=lo, length=length, g=float(g_each[b]), dt=1e-3, gamma=tuple(gam_each[b][:nd]))

    base = [gi.random_field(spec(0), seed=200 + k, smooth=0.05) for k in range(min(batch, 8))]
    p = gpe.Plan(n, lo, length, g=1.0, dt=1e-3, gamma=gam_each[0][:nd], batch=batch, g_each=g_each, gamma_each=gam_each)
    x = torch.from_numpy(np.stack([base[b % len(base)] for b in range(batch)]).astype(np.complex64)).cuda()
    p.step_real(x, 5)
    torch.cuda.synchronize()
    out = x.cpu().numpy()
    p.close()
    for b in sorted({*range(0, batch, max(1, batch // 40)), batch - 1}):
        ref = orc.Problem(**spec(b).kwargs()).step_real(base[b % len(base)], 5)
        assert np.linalg.norm(out[b] - ref) < 2e-5 * np.linalg.norm(ref), b
