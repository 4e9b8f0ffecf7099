"""The depthwise + pointwise block on tiles small enough for teams of depthwise warps: stage counts that
are not a multiple of the teams, several items per CTA, channel tiles that the warps of a lane
quarter take in turn, and planes at the limit of one team.  Against the oracle, every output."""
import zlib

import numpy as np
import pytest

from gpu_util import check_close
from test_gpu_dwpw import _block_tensors, _oracle_block, _run_block, hgc  # noqa: F401

pytestmark = pytest.mark.gpu

CASES = [
    # (id, n, c, h, w, k, stride, teams)
    ("7x7, one image, 12 stages with a channel tail, ragged channel tiles", 1, 712, 7, 7, 1000, 1, 4),
    ("7x7, three stages, four images per tile: one team", 40, 136, 7, 7, 512, 1, 1),
    ("14x14, five stages, four channel tiles", 2, 320, 14, 14, 512, 1, 2),
    ("14x14 -> 7x7 stride 2", 3, 192, 14, 14, 384, 2, 4),
    ("one row of 16 pixels", 2, 448, 1, 16, 256, 1, 2),
    ("32-channel stages, 6x10", 5, 32, 6, 10, 128, 1, 4),
    ("several items per CTA, weights that stay in the ring", 95, 24, 10, 14, 443, 1, 2),
    ("five items per CTA", 244, 24, 15, 10, 361, 1, 2),
]


@pytest.mark.parametrize("name,n,c,h,w,k,stride,teams", CASES, ids=[c[0] for c in CASES])
def test_block_with_teams(hgc, oracle, name, n, c, h, w, k, stride, teams):  # noqa: F811
    info = hgc.DwPwDesc(n, c, h, w, k, stride).plan_info()
    assert info["dw_teams"] == teams, info
    if "items per CTA" in name:
        assert info["tiles"] > info["grid"], info
    rng = np.random.default_rng(zlib.crc32(name.encode()))
    t = _block_tensors(rng, n, c, h, w, k)
    for y_nhwc in (True, False):
        ref = _oracle_block(oracle, n, c, h, w, k, stride, *t, True, y_nhwc)
        got = _run_block(hgc, n, c, h, w, k, stride, *t, True, y_nhwc, y_nhwc, True)
        check_close(got, ref, what=f"{name} nhwc={y_nhwc}")
