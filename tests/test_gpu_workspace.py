"""A solver's first call on a gauge field, which makes its workspace."""
import numpy as np
import pytest

import synth
from gpu_helpers import to_dev

pytestmark = pytest.mark.gpu


def test_first_solve_of_a_large_batch_equals_the_second(sq):
    """The workspace's clears (about 1 GB here) end before its first use:
    with the launch shapes already tuned, nothing else stands between them.
    Unit links and rough solves keep it short."""
    import torch
    dims, nrhs = (16, 16, 16, 64), 32
    vol = int(np.prod(dims))
    eye = np.broadcast_to(np.eye(3, dtype=np.complex128), (vol, 4, 3, 3))
    fat, lng = to_dev(eye * synth.C1), to_dev(eye * synth.C3)
    b = torch.stack([to_dev(synth.gaussian_source(vol // 2, j)) for j in range(4)]).repeat(8, 1, 1)
    for k in range(3):
        gid = sq.gauge_load(dims, fat, lng)
        try:
            xs = [sq.cg_solve_multi(gid, b, [0.3] * nrhs, 1e-3)[0] for _ in range(2)]
            assert bool((xs[1].abs().sum(dim=(1, 2)) > 0).all())
            assert torch.equal(xs[0], xs[1]), k
        finally:
            sq.gauge_free(gid)
