"""The file that SQ_TUNE_CACHE names: the tuner's own lines are choices, a
user's lines force shapes."""
import numpy as np
import pytest

import oracle
import synth
from gpu_helpers import gauge

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize('prec', ['f32', 'i16', 'f64'])
def test_own_lines_leave_the_resident_form_on(tmp_path, monkeypatch, prec):
    """Multi-shift solves, sq_tuned_launch and sq_time_dslash tune and save the
    shapes of the kernels that one-system solves would launch; a later context on
    the same file runs these solves as one without a file does, bit for bit, and a
    line of the user's survives the file being written again."""
    from paper_1411_2223_gb300 import sq as sqm
    dims = (4, 6, 8, 10)
    fat, lng = gauge(dims, 0.25, 0)
    b = synth.gaussian_source(oracle.volume(dims) // 2, 7)
    user = 'dslash_v4:8x8x8x8:p1:r18:n1:m3 256 1'

    def solve(ctx):
        gid = ctx.gauge_load(dims, fat, lng)
        x, st = ctx.cg_solve(gid, b, 0.1, 1e-8, precision=prec)
        return x, (st['oe_block'], st['eo_block'])

    monkeypatch.delenv('SQ_TUNE_CACHE', raising=False)
    with sqm.Context(0) as ctx:
        want = solve(ctx)
    cache = tmp_path / 'tune.txt'
    cache.write_text(user + '\n')
    monkeypatch.setenv('SQ_TUNE_CACHE', str(cache))
    with sqm.Context(0) as ctx:
        gid = ctx.gauge_load(dims, fat, lng)
        ctx.cg_solve_multishift(gid, b, [0.1, 0.2], 1e-8, precision=prec)
        for mode in ('cg_oe', 'cg_eo'):
            shape = ctx.tuned_launch(gid, prec, 18, 1, mode)
    text = cache.read_text().splitlines()
    assert user in text and len(text) > 3
    with sqm.Context(0) as ctx:
        got = solve(ctx)
        gid = ctx.gauge_load(dims, fat, lng)
        assert ctx.tuned_launch(gid, prec, 18, 1, 'cg_eo') == shape
    assert got[1] == want[1]
    assert np.array_equal(got[0], want[0])
