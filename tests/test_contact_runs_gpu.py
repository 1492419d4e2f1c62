"""The contact search's runs of cells where they break: rows that cross tiles, end at a
wall, wrap, or meet a last tile one cell wide, against the FP64 oracle (every pair)."""
import pytest

from tests.test_overlap_gpu import _check, _run
from tests.test_parity_gpu import make_case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rebin", [1, 4])
@pytest.mark.parametrize("deterministic", [False, True])
@pytest.mark.parametrize("q,n,periodic,npart",
                         [(9, (33, 20), (1, 1), 150), (9, (33, 17), (0, 1), 130),
                          (9, (65, 9), (1, 0), 130), (9, (64, 12), (1, 0), 170),
                          (19, (17, 18, 8), (1, 0, 1), 700), (15, (16, 9, 13), (1, 1, 0), 500),
                          (19, (34, 7, 9), (0, 1, 0), 600)])
def test_runs(q, n, periodic, npart, deterministic, rebin):
    c = make_case(q=q, n=n, periodic=periodic, tau=0.8, width=2, npart=npart, seed=11,
                  dia=(0.5, 0.8), rr=2.0, band=(0.1, 0.9), u_scale=2e-3, f0_eps=1e-3, e=0.8)
    got, ref = _run(c, 8, rebin=rebin, overlap="off", deterministic=deterministic)
    _check(got, ref, c["X"])
