"""The deferred-restart kernel with supplied actions and supplied start states: same bits as the general
kernel's per-lane shapes. Sizes around its 64-environment warps, horizons around the 32-step blocks in
which it reads actions, and one batch whose environments drift so far apart that the slowest ones
have to collect their actions themselves."""
import numpy as np
import pytest

from tests import gpu_helpers as H

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

RD = ("reward_stream", "done_bits")


@pytest.fixture(scope="module")
def cp():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2301_13062_b200 import binding, build
    build.build()
    binding.lib()
    torch.cuda.set_device(0)
    return binding


def rollout(cp, coop, n, T, kind=0, streams=(), limit=0, contracted=False, starts=None, given=None, spread=None, defer=0):
    from paper_2301_13062_b200 import inputs
    words = (n + 31) // 32
    shapes = {"done_bits": ((T, words), torch.int32), "reward_stream": ((T, n), torch.float32)}
    out = {"ep_return_sum": torch.full((n,), -1.0, device="cuda"),
           "ep_count": torch.full((n,), -1, dtype=torch.int32, device="cuda"),
           "totals": torch.zeros(2, dtype=torch.int64, device="cuda")}
    for name in streams:
        out[name] = torch.full(shapes[name][0], 7, dtype=shapes[name][1], device="cuda")
    weights = torch.from_numpy(inputs.per_env_linear_weights(n, 3)).cuda() if kind == 6 else inputs.policy_weights(kind, 3)
    kw = {"policy": cp.policy(kind, weights) if kind else None, "max_episode_steps": limit, "action_bits_in": given,
          "arithmetic": cp.CP_ARITH_CONTRACTED if contracted else cp.CP_ARITH_EXACT, "start_states_in": starts}
    cp.cp_tune("rollout_defer", defer)
    try:
        with H.rollout_shape(cp, {0: 0, 5: 2}.get(coop, 1), coop):
            if spread:
                planes = torch.from_numpy(inputs.random_states(n, 5, spread)).cuda()
                ep_len = torch.arange(n, dtype=torch.int32, device="cuda") % 37
                cp.cp_rollout_ex(T=T, state=cp.cp_wrap(planes, n, 9, t=11, env_offset=6), ep_len=ep_len, **kw, **out)
                out["planes"], out["ep_len"] = planes, ep_len
            else:
                out["final_state"] = torch.zeros(4, n, device="cuda")
                cp.cp_rollout_ex(n_envs=n, T=T, seed=9, t0=11, env_offset=6, **kw, **out)
    finally:
        cp.cp_tune("rollout_defer", 0)
    torch.cuda.synchronize()
    return {k: v.cpu().numpy() for k, v in out.items()}


def assert_same_bits(a, b):
    for k in a:
        assert np.array_equal(a[k].view(np.uint32) if a[k].dtype == np.float32 else a[k],
                              b[k].view(np.uint32) if b[k].dtype == np.float32 else b[k]), k


def action_rows(T, n):
    return torch.from_numpy(np.random.default_rng(2).integers(-2**31, 2**31, (T, (n + 31) // 32)).astype(np.int32)).cuda()


def start_rows(T, n):
    rng = np.random.default_rng(17)
    s = rng.uniform(-0.3, 0.3, (T, 4, n)).astype(np.float32)  # angles on both sides of the polynomial range
    s[:, 2, ::7] = rng.uniform(-3, 3, s[:, 2, ::7].shape)
    s[T // 2, 0, ::5] = np.inf
    s[T // 3, 3, ::5] = np.nan
    s[T // 3, 2, 1::5] = np.nan
    return torch.from_numpy(s).cuda()


@pytest.mark.parametrize("n", [1, 31, 33, 64, 65, 1000, 4099])
@pytest.mark.parametrize("T", [2, 12, 31, 32, 33, 65, 200, 300])
def test_supplied_actions(cp, n, T):
    bits = action_rows(T, n)
    for streams, limit, spread, contracted in (((), 0, None, False), (RD, 20, "wide", False), (RD, 0, None, True), ((), 9, "edge", False)):
        args = dict(streams=streams, limit=limit, spread=spread, given=bits, contracted=contracted)
        general = rollout(cp, 2, n, T, **args)
        for defer in (0, 2, 6):
            assert_same_bits(rollout(cp, 5, n, T, defer=defer, **args), general)


@pytest.mark.parametrize("kind,given", [(0, False), (0, True), (1, False), (6, False), (2, True)])
@pytest.mark.parametrize("n,T", [(1, 33), (65, 12), (1000, 200), (4099, 70)])
def test_supplied_starts(cp, kind, given, n, T):
    bits = action_rows(T, n) if given else None
    for streams, limit, spread, contracted in (((), 0, None, False), (RD, 20, "wide", False), (RD, 0, "edge", True)):
        args = dict(kind=kind, streams=streams, limit=limit, spread=spread, given=bits, starts=start_rows(T, n), contracted=contracted)
        general = rollout(cp, 2, n, T, **args)
        for defer in (0, 2, 6):
            assert_same_bits(rollout(cp, 5, n, T, defer=defer, **args), general)


@pytest.mark.parametrize("kind,given", [(0, False), (0, True), (1, False), (6, False)])
@pytest.mark.parametrize("theta", [0.3, 0.2, None])   # episodes of one step; of one to three; rows of either sort and of twenty steps
@pytest.mark.parametrize("n,T", [(65, 33), (4099, 200)])
def test_short_episodes_from_supplied_starts(cp, kind, given, theta, n, T):
    """The passes come closer together while episodes are short, and apart again."""
    rng = np.random.default_rng(8)
    s = rng.uniform(-0.05, 0.05, (T, 4, n)).astype(np.float32)
    s[:, 2] = theta if theta else np.array([0.3, 0.2, 0.0])[(np.arange(T) // 16) % 3][:, None]
    s[:, 3] = rng.uniform(0.1, 0.5, (T, n))
    bits = action_rows(T, n) if given else None
    for streams, limit, contracted in (((), 0, False), (RD, 2, False), (RD, 0, True)):
        args = dict(kind=kind, streams=streams, limit=limit, given=bits, starts=torch.from_numpy(s).cuda(), contracted=contracted)
        general = rollout(cp, 2, n, T, **args)
        for defer in (2, 6):
            assert_same_bits(rollout(cp, 5, n, T, defer=defer, **args), general)


@pytest.mark.parametrize("kind,given,starts", [(0, True, False), (0, True, True), (0, False, True), (1, False, True), (6, False, True)])
@pytest.mark.parametrize("n,T", [(70_001, 200), (47_361, 250)])
def test_what_a_caller_gets(cp, kind, given, starts, n, T):
    """Nothing forced: large enough for this kernel, which is told by the launch of its own that clears the done
    bits (actions alone with outputs take it from 66,304 environments on)."""
    bits = action_rows(T, n) if given else None
    rows = torch.rand(T, 4, n, generator=torch.Generator("cuda").manual_seed(5), device="cuda") * 0.1 - 0.05 if starts else None
    for streams, limit, spread in (((), 0, None), (RD, 0, "wide"), (RD, 11, None)):
        args = dict(kind=kind, streams=streams, limit=limit, spread=spread, given=bits, starts=rows)
        general = rollout(cp, 2, n, T, **args)
        before = cp.cp_launch_count()
        assert_same_bits(rollout(cp, 0, n, T, **args), general)
        cleared = streams == RD and limit != 11 and (starts or n > 66_304)
        assert cp.cp_launch_count() - before == (2 if cleared else 1)


@pytest.mark.parametrize("starts", [False, True])
def test_environments_far_apart(cp, starts):
    """Constant actions end an episode after ten steps; the recorded actions of a policy that balances end
    none. The first kind falls hundreds of steps behind the second in the same warp."""
    n, T = 130, 3000
    words = (n + 31) // 32
    balance = cp.policy(1, np.array([0, 0, 0, 0, 0.05, 0.1, 1.0, 0.5, 0, 0], np.float32))
    given = torch.zeros(T, words, dtype=torch.int32, device="cuda")
    cp.cp_rollout_ex(n_envs=n, T=T, seed=9, t0=11, env_offset=6, policy=balance, action_bits=given)
    every_third = [sum(1 << i for i in range(32) if (32 * w + i) % 3) for w in range(words)]
    given |= torch.tensor(np.array(every_third, np.uint32).view(np.int32)).cuda()     # the others always push right
    args = dict(given=given, starts=torch.zeros(T, 4, n, device="cuda") if starts else None, streams=RD)
    general = rollout(cp, 2, n, T, **args)
    assert_same_bits(rollout(cp, 5, n, T, **args), general)
    assert general["ep_count"][::3].max() <= 1 and general["ep_count"][1::3].min() > T // 15


@pytest.mark.parametrize("coop", [0, 5])
@pytest.mark.parametrize("n,T", [(100_003, 200), (4099, 40)])   # what a caller gets, and the kernel asked for
def test_done_bits_written_over_the_actions(cp, coop, n, T):
    """A recording's actions replaced by the done bits of the call that plays it."""
    bits = action_rows(T, n)
    apart, over = torch.zeros_like(bits), bits.clone()
    reward, ret = torch.empty(T, n, device="cuda"), [torch.empty(n, device="cuda") for _ in range(2)]
    for given, done, r in ((bits, apart, ret[0]), (over, over, ret[1])):
        with H.rollout_shape(cp, 0, coop):
            cp.cp_rollout_ex(n_envs=n, T=T, seed=9, action_bits_in=given, done_bits=done, reward_stream=reward, ep_return_sum=r)
    assert torch.equal(apart, over) and torch.equal(*ret)


@pytest.mark.parametrize("coop", [0, 5])
def test_rewards_written_over_the_start_states(cp, coop):
    """Reward row r lies over start states of row r / 4, read by the step before or not at all. Episodes of one
    step (x beyond its threshold), so that every row is read; x overwritten by a reward would not end them."""
    n, T = 50_001, 200
    starts = torch.from_numpy(np.random.default_rng(4).uniform(-0.05, 0.05, (T, 4, n)).astype(np.float32)).cuda()
    starts[:, 0] += 3.0
    got = []
    for over in (False, True):
        s = starts.clone()
        reward = s.view(-1)[:T * n].view(T, n) if over else torch.empty(T, n, device="cuda")
        done = torch.empty(T, (n + 31) // 32, dtype=torch.int32, device="cuda")
        final = torch.empty(4, n, device="cuda")
        with H.rollout_shape(cp, 0, coop):
            cp.cp_rollout_ex(n_envs=n, T=T, seed=9, start_states_in=s, done_bits=done, reward_stream=reward, final_state=final)
        got.append((done, final))
    assert torch.equal(got[0][0], got[1][0]) and torch.equal(got[0][1], got[1][1])
