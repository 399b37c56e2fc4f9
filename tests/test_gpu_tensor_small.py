"""Tensor products with single polynomials among the children, and of every
small unrolled shape, against the oracle: a single polynomial has no unrolled
kernel and takes the bounded one, with and without "tensor_fixed", on limbs
(every prime below 2^60) and as 128-bit products."""
import numpy as np
import pytest

import synth
from oracle import ckks as O

from gpu_common import dev, host

pytestmark = pytest.mark.gpu

NODES = [(1,), (1, 1), (2, 1), (1, 2), (3, 1), (1, 1, 1), (1, 2, 1), (2, 2, 1), (3, 3, 1), (1, 1, 1, 1), (13, 1),
         (2, 2), (3, 3), (2, 2, 2), (3, 2, 3)]


@pytest.mark.parametrize("bits", [[50, 45, 54], [61, 50, 45]])
def test_small_nodes_match_the_oracle(bits):
    import paper_2601_15401_gb300 as G
    p = synth.make_params(6, bits, 1, 3)
    ctx, octx = G.Context.from_params(p), O.Ctx(p)
    g = synth.rng(210, len(bits))
    for polys in NODES:
        tups = [np.stack([synth.uniform_residues(g, p.q, p.N) for _ in range(n)]) for n in polys]
        n_out = sum(polys) - len(polys) + 1
        want = O.tensor_product(octx, tups)
        for fixed in (1, 0):
            ctx.tune_set("tensor_fixed", fixed)
            # one polynomial more than the result has: it stays as it was
            buf = np.full((n_out + 1, p.L, p.N), 7, dtype=np.uint64)
            out = G.Tuple.wrap(dev(buf))
            ctx.tensor([G.Tuple.wrap(dev(t)) for t in tups], out)
            ctx.check()
            assert out.n_polys == n_out
            got = host(out.data)
            assert np.array_equal(got[:n_out], want), (polys, fixed)
            assert np.array_equal(got[n_out:], buf[n_out:]), (polys, fixed)
