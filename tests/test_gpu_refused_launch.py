"""A call whose launch CUDA refuses (more limbs than a grid dimension holds)
reports the error and leaves nothing behind: the next valid calls, on that
context and on another, succeed with the right residues, and the runtime holds
no error for the thread."""
import numpy as np
import pytest

import synth
from oracle import ring as R

from gpu_common import dev, host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("log_n", [4, 9])
def test_a_refused_transform_leaves_no_error_behind(log_n):
    import torch

    import paper_2601_15401_gb300 as G
    from paper_2601_15401_gb300._lib import CkksError
    p = synth.make_params(log_n, [50, 45], 1, 2)
    ctx, other = G.Context.from_params(p), G.Context.from_params(p)
    polys = 32768 if log_n > 4 else 65535       # times 2 limbs: above 65535
    big = torch.zeros((polys, 2, p.N), dtype=torch.uint64, device="cuda")
    x = synth.uniform_residues(synth.rng(220), p.q, p.N)
    for call in ("ntt", "intt"):
        with pytest.raises(CkksError) as e:
            getattr(ctx, call)(G.Tuple(big, polys, 2, 2, 0 if call == "ntt" else 1))
        assert e.value.code == -5
        for c in (other, ctx):
            t = G.Tuple(dev(x[None]), 1, 2, 2, 0)
            c.ntt(t)
            assert np.array_equal(host(t.data)[0], R.ntt_rows(x, p.q))
        other.check()
        torch.cuda.synchronize()
