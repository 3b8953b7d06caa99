"""Hidden widths besides the headline ones, in both precisions, on the GPU against the oracle stage by stage (needs a B200):
partial column tiles (384 is one and a half of 256), the smallest batches, row counts around the tiles' edges, boards whose
cell count is and is not a multiple of 64, batches on either side of the base-GEMM and tile-size rules."""
import numpy as np
import pytest

from oracle import binding as orc
from paper_2104_06272_b200.workloads import Workload, random_params
from tests import parity as par

pytestmark = pytest.mark.gpu

CASES = [
    # (H, precision, B, N, T)
    (384, 0, 3, 3, 2), (384, 0, 129, 11, 5), (384, 1, 77, 5, 4), (512, 0, 70, 8, 6), (512, 0, 2049, 7, 3), (768, 0, 33, 16, 3),
    (768, 1, 257, 6, 3), (1024, 0, 130, 9, 2), (1024, 0, 1025, 4, 2), (1024, 1, 9, 7, 3), (384, 0, 9500, 3, 2),
    (384, 1, 9500, 3, 2), (512, 1, 9473, 4, 2), (768, 0, 9490, 2, 2),
    # the warp-level kernels' widths: batches around a CTA's 32 envs and a dh1 tile's 64, one and several t-slices
    (32, 0, 33, 5, 3), (32, 1, 65, 4, 2), (96, 0, 2, 3, 4), (96, 0, 777, 7, 20), (96, 1, 64, 12, 5), (192, 0, 100, 6, 9),
    (192, 0, 5, 4, 55), (192, 1, 2100, 5, 3), (64, 0, 1500, 5, 9), (64, 1, 31, 6, 33),
    # width 64: several steps in a 128-row tile (rows left over, slices that end short), one env more than fits, a CTA that walks
    # 24 tiles (longer ones: LONG_SUMS below); boards of more than 128 cells there and at 128 and 256
    (64, 0, 1, 12, 5), (64, 0, 5, 16, 40), (64, 1, 64, 12, 7), (64, 0, 65, 5, 20), (64, 1, 129, 16, 3), (64, 0, 18945, 3, 17),
    (128, 0, 130, 16, 5), (128, 1, 77, 12, 9), (256, 0, 40, 12, 7), (256, 1, 300, 16, 4), (32, 1, 300, 16, 9), (192, 1, 70, 13, 6),
    # units of (128-env tile, slice) that do not come out even: more units than CTAs, a short last slice, 5 and 16 slices
    (128, 0, 2500, 5, 24), (128, 1, 1300, 5, 11), (256, 0, 6000, 5, 7), (256, 1, 1000, 4, 17), (256, 0, 100, 6, 33),
    # width 128 on boards of up to 128 cells (tiles of 64 envs, one kernel from the head outputs to dh1): batches around a tile's edge,
    # the largest board, several units a CTA with a short last tile, a CTA without a whole slice
    (128, 0, 1, 11, 3), (128, 1, 63, 2, 70), (128, 0, 64, 3, 9), (128, 0, 65, 11, 20), (128, 1, 9537, 8, 3), (128, 0, 19000, 6, 5),
    # the agent rows of W1 beside three CTAs per SM at width 64, and one step or one CTA short of it
    (64, 0, 14241, 3, 3), (64, 0, 14300, 9, 16), (64, 0, 14241, 3, 9), (64, 0, 14209, 11, 10), (64, 0, 14208, 5, 10),
    # just beyond one wave of the smaller-batch rollouts at H = 128 and 256
    (128, 0, 9473, 4, 2), (128, 1, 9500, 5, 3), (128, 0, 9480, 14, 2), (256, 0, 4737, 4, 2), (256, 1, 4800, 5, 3),
    # 16 and 32 envs per CTA, agent rows of W1 in shared memory and not
    (256, 0, 2368, 4, 2), (256, 0, 2369, 12, 2), (256, 1, 2500, 13, 2), (256, 0, 19, 13, 3), (256, 1, 33, 14, 3),
    (192, 0, 17, 16, 3), (192, 0, 2369, 3, 2), (128, 1, 2368, 16, 2), (128, 0, 2400, 5, 2), (96, 0, 2368, 5, 2), (96, 0, 2380, 5, 3), (96, 0, 4737, 3, 2),
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


@pytest.mark.parametrize("prec,B,T,passes", [(0, 148 * 128 + 77, 5, 60), (1, 148 * 128 + 77, 5, 60), (0, 148 * 64, 97, 20), (1, 148 * 64, 97, 20)])
def test_width_128_gradients_do_not_depend_on_timing(bnd, prec, B, T, passes):
    """Two handles in lockstep over many passes: the same bits.  Two to three units of 64 envs a CTA, some fifteen tiles; one unit of 97 tiles a
    CTA, where in fp32 both accumulators are emptied and restarted on the way.  (The warps of the fused backward kernel hand tiles on
    through mbarriers; one that read the agent plane's accumulator ahead of its last MMAs showed here in one pass of fifteen in bf16.)"""
    pair = []
    for _ in range(2):
        an = bnd.Anakin(bnd.make_cfg(B, 8, 128, T, precision=prec, episode_cap=4))
        an.reset(6)
        pair.append(an)
    for i in range(passes):
        grads = []
        for an in pair:
            an.run(1)
            grads.append(an.get(bnd.GRADS))
        assert (grads[0].view(np.uint32) == grads[1].view(np.uint32)).all(), f"pass {i}"


LONG_SUMS = [
    # (H, precision, B, N, T, bias of the value head).  Many rows a CTA: the accumulators of the backward kernels are emptied and
    # restarted on the way: the agent plane every 48 tiles of 128 rows at H = 256 and, on boards of more than 128 cells, 128, every 96 tiles
    # at 64; dW2 at 64 every 32; at H = 128 on smaller boards, in tiles of 64 rows, the agent plane every 96 and dW2 every 56.  However the
    # tiles are dealt out, one of the 148 CTAs (74 pairs at H = 256) has at least the mean of them.
    # The tensor core rounds toward zero, so a sum that is left in one accumulator is biased, most where nearly every MMA adds to
    # it: four cells, and a value head that is off by 3 (every row pulls the same way).
    (128, 0, 131072, 2, 96, 3.0), (64, 0, 131072, 2, 160, 3.0),
    (128, 0, 18945, 13, 49, 0.0), (256, 0, 30000, 3, 20, 3.0), (256, 0, 7000, 12, 70, 0.0),
    (64, 0, 18945, 3, 98, 0.0), (64, 0, 18945, 12, 98, 0.0), (64, 1, 18945, 5, 34, 0.0), (64, 1, 18945, 12, 34, 0.0),
    # one unit of T tiles a CTA: exactly one group of either accumulator, and one tile more
    (128, 0, 148 * 64, 3, 56, 0.0), (128, 0, 148 * 64, 3, 57, 0.0), (128, 0, 148 * 64, 3, 96, 0.0), (128, 0, 148 * 64, 3, 97, 0.0),
]


@pytest.mark.parametrize("H,prec,B,N,T,bias", LONG_SUMS)
def test_gradients_of_long_sums(bnd, H, prec, B, N, T, bias):
    """One whole update on the library's own trajectory, element by element against the oracle."""
    w = Workload(f"long_h{H}_p{prec}", B=B, N=N, H=H, T=T, iters=1, precision=prec)
    an = bnd.Anakin(bnd.cfg_from_workload(w, debug_logits=1))
    an.reset(11)
    theta = random_params(5, w.P, 0.15)
    theta[-1] = bias
    an.set(bnd.PARAMS, theta)
    st = par.gpu_state(an, bnd)
    an.rollout()
    an.gae()
    row = lambda which: an.get(which).reshape(T, B)  # noqa: E731
    par.MARGINS.clear()
    try:
        par.check_learn(an, bnd, w, st, dict(pos=row(bnd.TRAJ_POS), action=row(bnd.TRAJ_ACTION)), row(bnd.ADV), row(bnd.RET))
    finally:
        print(w.name, "worst error / bound:", {k: round(v, 3) for k, v in par.MARGINS.items()})
    assert an.status() == 0


def test_width_128_dw2_is_as_exact_as_sums_of_scattered_rows(bnd):
    """dW2 of 1.28 million rows against the oracle's sums in double.  The tensor core rounds every addition toward zero, by up to 2^-23 of what the
    accumulator holds; 3 * 3584 / 16 additions to sums that are on average half grown lose 672 * 2^-23 / 4 = 2e-5 at most where every term
    has the same sign.  Sums of 4096 rows that lie scattered over the batch gave 1.7e-5 here, of as many consecutive rows of the same envs
    1.9e-5."""
    B, N, T = 20000, 8, 64
    w = Workload("dw2_error", B=B, N=N, H=128, T=T, iters=1)
    an = bnd.Anakin(bnd.cfg_from_workload(w, debug_logits=1))
    an.reset(11)
    theta = random_params(5, w.P, 0.15)
    theta[-1] = 0.0
    an.set(bnd.PARAMS, theta)
    st = par.gpu_state(an, bnd)
    an.rollout()
    an.learn()
    traj = [an.get(which).reshape(T, B) for which in (bnd.TRAJ_POS, bnd.TRAJ_ACTION, bnd.ADV, bnd.RET)]
    gates = an.get(bnd.DEBUG_GATES).reshape(2, B * T, 4)
    want = orc.learn(N, 128, 0, theta, st["walls"], st["goal"], *traj, np.float32(w.value_coef), np.float32(w.entropy_coef), gates=(gates[0], gates[1]))[0]
    sl = orc.Dims(N, 128).slices()["W2"]
    want = want[sl].astype(np.float64)
    err = np.linalg.norm(an.get(bnd.GRADS)[sl] - want) / np.linalg.norm(want)
    print(f"2-norm of the error of dW2: {err:.2e}")
    assert err <= 1.75e-5 and an.status() == 0


@pytest.mark.parametrize("H,B,N", [(64, 606208, 12), (256, 303104, 12), (64, 4194304, 3), (32, 606208, 5), (1024, 65536, 16)])
def test_wall_plane_sums_are_not_biased(bnd, H, B, N):
    """fp32 sums over the envs on the tensor core, which rounds every addition toward zero.  Every row adds the same value here (all gates
    open, no policy gradient, returns off by a constant), so what the additions lose has one sign.  The leading 16-bit terms of the at most
    8192 rows of a split are equal numbers of 11 bits: 24 bits hold their sum, and it loses nothing as long as no other term goes into the
    same accumulator.  What is left: a value as two fp16 terms, 2^-22, and dh1 itself, 3 H / 16 MMAs each of which loses less than a unit in
    the last place, 2^-23, of a sum that is on average half grown.  Boards of two row tiles a plane, where a split has most rows, a batch of
    more than 128 such splits, three-term operands.  (With both terms in one accumulator: 6e-6 to 8e-6, 1e-4 in one of 128 splits.)"""
    an = bnd.Anakin(bnd.make_cfg(B, N, H, 1, entropy_coef=0.0))
    an.reset(7)
    rng = np.random.default_rng(3)
    sl = orc.Dims(N, H).slices()
    theta = np.zeros(an.P, np.float32)
    theta[sl["W1"]] = 0.1 * rng.standard_normal(3 * N * N * H) / N
    theta[sl["b1"]] = 2.0
    theta[sl["W2"]] = rng.uniform(0.5, 1.5, H * H) / H
    theta[sl["b2"]] = 1.0
    theta[sl["Wh"]].reshape(H, 5)[:, 4] = rng.uniform(0.5, 1.5, H) / H
    an.set(bnd.PARAMS, theta)
    an.rollout()
    value = an.get(bnd.TRAJ_VALUE)[:B]
    ret = (value + 64).astype(np.float32)  # (far off, so that rounding of the values themselves does not count)
    an.set(bnd.ADV, np.zeros(B, np.float32))
    an.set(bnd.RET, ret)
    an.update()
    assert an.status() == 0
    grads = an.get(bnd.GRADS)
    # in double: dL/dvalue of a row, down through open gates, times the number of rows of a bias, of a wall cell, of a goal cell
    d_out = 2 * float(bnd.make_cfg(B, N, H, 1).value_coef) * (value.astype(np.float64) - ret).mean()
    d_h1 = d_out * theta[sl["W2"]].reshape(H, H).astype(np.float64) @ theta[sl["Wh"]].reshape(H, 5)[:, 4]
    walls, goal = an.get(bnd.ENV_WALLS).reshape(B, -1), an.get(bnd.ENV_GOAL)
    cells = np.arange(N * N)
    n_wall = np.array([((walls[:, c >> 5] >> (c & 31)) & 1).sum() for c in cells])
    n_goal = np.bincount(goal, minlength=N * N)
    dW1 = grads[sl["W1"]].reshape(3, N * N, H)
    for name, got, want in (("b1", grads[sl["b1"]], d_h1), ("walls", dW1[0], np.outer(n_wall / B, d_h1)), ("goal", dW1[2], np.outer(n_goal / B, d_h1))):
        bias = (np.asarray(got, np.float64) - want).sum() / want.sum()
        print(f"H = {H}, {B} envs: {name} off by {bias:+.2e}")
        assert abs(bias) <= 2.0**-22 + 3 * H / 16 * 2.0**-24, name
        par.assert_close(got, want, par.RTOL_FP32, name)


@pytest.mark.parametrize("H,prec,B,T", [(32, 0, 40, 7), (64, 0, 33, 9), (96, 1, 70, 5), (128, 0, 65, 11), (128, 1, 200, 4), (256, 0, 127, 6), (256, 0, 300, 9),
                                        (256, 1, 129, 7), (384, 0, 70, 5), (32, 0, 3000, 17), (64, 0, 6000, 9), (96, 1, 3000, 16), (192, 0, 1500, 16),
                                        (192, 1, 5000, 3)])
def test_replayed_forward_pass_equals_the_rollouts_own(bnd, H, prec, B, T):
    """The update of a trajectory handed back through set() recomputes the forward pass in slices of steps (few envs), and must
    give the gradient of the update that reuses the rollout's activations."""
    w = Workload("replay", B=B, N=5, H=H, T=T, iters=1, precision=prec, episode_cap=6)
    grads = []
    for hand_back in (False, True):
        an = bnd.Anakin(bnd.cfg_from_workload(w))
        an.reset(3)
        an.set(bnd.PARAMS, random_params(5, w.P, 0.15 if H <= 256 else 0.05))
        an.rollout()
        if hand_back:
            an.set(bnd.TRAJ_POS, an.get(bnd.TRAJ_POS))
        an.learn()
        grads.append(an.get(bnd.GRADS))
        assert an.status() == 0
    par.assert_close(grads[1], grads[0], par.rtol_of(prec), "replayed gradient")


@pytest.mark.parametrize("B,H", [(3, 384), (130, 512), (77, 768), (1024, 1024)])
def test_acting_without_a_workspace_at_the_wide_widths(bnd, B, H):
    """One step's activations in the library's own scratch give the trajectory of the handle-based rollout."""
    import numpy as np
    import torch

    T, N = 5, 6
    cfg = bnd.make_cfg(B, N, H, T)
    an = bnd.Anakin(cfg)
    an.reset(7)

    def dev(which):
        x = an.get(which)
        return torch.from_numpy(x.view(np.int32) if x.dtype == np.uint32 else x).cuda()

    env = [dev(w) for w in (bnd.PARAMS, bnd.ENV_WALLS, bnd.ENV_START, bnd.ENV_GOAL, bnd.ENV_POS, bnd.ENV_TEP)]
    traj = [torch.zeros(n, dtype=t, device="cuda") for n, t in ((T * B, torch.uint8), (T * B, torch.int8), (T * B, torch.uint8),
                                                               (T * B, torch.float32), ((T + 1) * B, torch.float32), (T * B, torch.float32))]
    for call in range(2):
        assert bnd.rollout_noalloc(cfg, 7, call * T, T, *env, *traj) == bnd.OK
        an.rollout()
        for x, which in zip(traj, (bnd.TRAJ_POS, bnd.TRAJ_ACTION, bnd.TRAJ_DONE, bnd.TRAJ_REWARD, bnd.TRAJ_VALUE, bnd.TRAJ_LOGP)):
            want = an.get(which)
            if want.dtype == np.float32:
                par.assert_close(x.cpu().numpy(), want, 1e-5, "trajectory")
            else:
                assert (x.cpu().numpy() == want.reshape(-1)).all()
    assert an.status() == 0 and bnd.noalloc_status()[1] == 0
