"""Hidden widths besides the headline ones, in both precisions, on the GPU against the oracle stage by stage (needs a B200):
partial column tiles (384 is one and a half of 256), the smallest batches, row counts around the tiles' edges, boards whose
cell count is and is not a multiple of 64, batches on either side of the base-GEMM and tile-size rules."""
import pytest

from paper_2104_06272_b200.workloads import Workload, random_params
from tests import parity as par

pytestmark = pytest.mark.gpu

CASES = [
    # (H, precision, B, N, T)
    (384, 0, 3, 3, 2), (384, 0, 129, 11, 5), (384, 1, 77, 5, 4), (512, 0, 70, 8, 6), (512, 0, 2049, 7, 3), (768, 0, 33, 16, 3),
    (768, 1, 257, 6, 3), (1024, 0, 130, 9, 2), (1024, 0, 1025, 4, 2), (1024, 1, 9, 7, 3), (384, 0, 9500, 3, 2),
    # the warp-level kernels' widths: batches around a CTA's 32 envs and a dh1 tile's 64, one and several t-slices
    (32, 0, 33, 5, 3), (32, 1, 65, 4, 2), (96, 0, 2, 3, 4), (96, 0, 777, 7, 20), (96, 1, 64, 12, 5), (192, 0, 100, 6, 9),
    (192, 0, 5, 4, 55), (192, 1, 2100, 5, 3), (64, 0, 1500, 5, 9), (64, 1, 31, 6, 33),
]


@pytest.fixture(scope="module")
def bnd():
    from paper_2104_06272_b200 import binding

    return binding


@pytest.mark.parametrize("H,prec,B,N,T", CASES)
def test_width_one_iteration_stage_by_stage(bnd, H, prec, B, N, T):
    w = Workload(f"h{H}_p{prec}_b{B}", B=B, N=N, H=H, T=T, iters=1, precision=prec, episode_cap=4)
    an = bnd.Anakin(bnd.cfg_from_workload(w, debug_logits=1))
    an.reset(11)
    an.set(bnd.PARAMS, random_params(5, w.P, 0.15 if H <= 256 else 0.05))
    par.MARGINS.clear()
    try:
        par.check_iteration(an, bnd, w, 11)
        par.check_iteration(an, bnd, w, 11)
    finally:
        print(w.name, "worst error / bound:", {k: round(v, 3) for k, v in par.MARGINS.items()})
