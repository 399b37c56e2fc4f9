"""Transforms of N = 2^4..2^8, several limbs to a CTA: limb counts that fill the
last CTA and that do not, against the oracle bit for bit, with the words behind
the last limb left alone."""
import numpy as np
import pytest

import synth
from oracle import ring as R

from gpu_common import dev, host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("log_n", range(4, 9))
@pytest.mark.parametrize("bits", [[50], [61, 53, 45]])
def test_every_remainder_of_limbs(log_n, bits):
    import paper_2601_15401_gb300 as G
    p = synth.make_params(log_n, bits, 1, 1)
    ctx = G.Context.from_params(p)
    g = synth.rng(230, log_n)
    for polys in (1, 2, 3, 4, 5, 9):
        x = np.stack([synth.uniform_residues(g, p.q, p.N) for _ in range(polys)])
        for call, form, rows in ((ctx.ntt, 0, R.ntt_rows), (ctx.intt, 1, R.intt_rows)):
            buf = dev(np.full((polys + 1, p.L, p.N), 7, np.uint64))
            call(G.Tuple(dev(x), polys, p.L, p.L, form), G.Tuple(buf, polys, p.L, p.L, 1 - form))
            ctx.check()
            got = host(buf)
            assert np.array_equal(got[:polys], np.stack([rows(a, p.q) for a in x])), polys
            assert (got[polys:] == 7).all(), polys
