"""Small batches under feedback policies or from supplied start states: the producer-assisted kernel
(linear policies, supplied starts) and the network kernel that spreads hidden units over lanes. Both
must give the bits of the general kernel's per-lane shape, which the other files pin to the oracle.
Sizes: around the 32 environments of a bit-plane word, odd warp tasks, and either side of the bounds
at which the network kernel takes more lanes or leaves the call (148 SMs: 2,368, 4,736, 9,472 and 14,208
environments). Horizons: around the 32-step hand-overs of both kernels."""
import numpy as np
import pytest

from tests import gpu_helpers as H

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

LINEAR, MLP, MLP32, MLP64, PER_ENV, DEEP = 1, 2, 4, 5, 6, 7
ALL = ("reward_stream", "done_bits", "action_bits", "trajectory")


@pytest.fixture(scope="module")
def cp():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2301_13062_b200 import binding, build
    build.build()
    binding.lib()
    torch.cuda.set_device(0)
    return binding


def policy_of(cp, kind, n, seed=3):
    from paper_2301_13062_b200 import inputs
    if kind == PER_ENV:
        return cp.policy(kind, torch.from_numpy(inputs.per_env_linear_weights(n, seed)).cuda())
    return cp.policy(kind, inputs.policy_weights(kind, seed))


def rollout(cp, coop, kind, n, T, streams=(), limit=0, contracted=False, starts=None, given=None, spread=None):
    from paper_2301_13062_b200 import inputs
    words = (n + 31) // 32
    shapes = {"done_bits": ((T, words), torch.int32), "action_bits": ((T, words), torch.int32),
              "reward_stream": ((T, n), torch.float32), "trajectory": ((T, 4, n), torch.float32)}
    out = {"ep_return_sum": torch.full((n,), -1.0, device="cuda"),
           "ep_count": torch.full((n,), -1, dtype=torch.int32, device="cuda"),
           "totals": torch.zeros(2, dtype=torch.int64, device="cuda")}
    for name in streams:
        out[name] = torch.full(shapes[name][0], 7, dtype=shapes[name][1], device="cuda")
    kw = {"policy": policy_of(cp, kind, n) if kind else None, "max_episode_steps": limit, "action_bits_in": given,
          "arithmetic": cp.CP_ARITH_CONTRACTED if contracted else cp.CP_ARITH_EXACT, "start_states_in": starts}
    with H.rollout_shape(cp, 1 if coop else 0, coop):
        if spread:  # a batch in the middle of its episodes
            planes = torch.from_numpy(inputs.random_states(n, 5, spread)).cuda()
            ep_len = torch.arange(n, dtype=torch.int32, device="cuda") % 37
            cp.cp_rollout_ex(T=T, state=cp.cp_wrap(planes, n, 9, t=11, env_offset=6), ep_len=ep_len, **kw, **out)
            out["planes"], out["ep_len"] = planes, ep_len
        else:
            out["final_state"] = torch.zeros(4, n, device="cuda")
            cp.cp_rollout_ex(n_envs=n, T=T, seed=9, t0=11, env_offset=6, **kw, **out)
    torch.cuda.synchronize()
    return {k: v.cpu().numpy() for k, v in out.items()}


def assert_same_bits(a, b):
    for k in a:
        assert np.array_equal(a[k].view(np.uint32) if a[k].dtype == np.float32 else a[k],
                              b[k].view(np.uint32) if b[k].dtype == np.float32 else b[k]), k


def start_rows(T, n):
    rng = np.random.default_rng(17)
    s = rng.uniform(-0.3, 0.3, (T, 4, n)).astype(np.float32)  # angles on both sides of the polynomial range
    s[:, 2, ::7] = rng.uniform(-3, 3, s[:, 2, ::7].shape)
    s[T // 2, 0, ::5] = np.inf
    s[T // 3, 3, ::5] = np.nan
    return torch.from_numpy(s).cuda()


@pytest.mark.parametrize("kind", [MLP, MLP32, MLP64, DEEP])
@pytest.mark.parametrize("n,T", [(1, 33), (31, 64), (33, 5), (1000, 4), (1184, 11), (1184, 40), (1185, 31), (2369, 32), (4737, 31),
                                 (9465, 65), (9472, 33), (9473, 33), (9473, 129), (14208, 129), (14209, 129)])
def test_networks(cp, kind, n, T):
    for streams, limit, spread in (((), 0, None), (ALL, 20, "wide"), (("done_bits",), 0, "edge"), (("trajectory",), 9, None),
                                   (("reward_stream", "done_bits"), 0, "edge")):
        args = dict(streams=streams, limit=limit, spread=spread)
        assert_same_bits(rollout(cp, 0, kind, n, T, **args), rollout(cp, 2, kind, n, T, **args))


@pytest.mark.parametrize("kind", [MLP, MLP32, MLP64, DEEP])
@pytest.mark.parametrize("n,T", [(97, 50), (1500, 50), (4097, 50), (9473, 64), (14208, 128), (14209, 128)])
def test_networks_contracted(cp, kind, n, T):
    for streams in ((), ALL, ("reward_stream", "done_bits")):
        args = dict(streams=streams, limit=15, contracted=True)
        assert_same_bits(rollout(cp, 0, kind, n, T, **args), rollout(cp, 2, kind, n, T, **args))


@pytest.mark.parametrize("kind", [MLP, MLP32, MLP64, DEEP])
@pytest.mark.parametrize("contracted", [False, True])
@pytest.mark.parametrize("n,T", [(4737, 33), (9473, 31), (9487, 97), (14209, 8), (18944, 64), (18961, 130), (28417, 65), (37889, 49), (56832, 66)])
def test_networks_by_two_lanes_and_one(cp, kind, contracted, n, T):
    """148 SMs: two lanes per environment up to 9,472 (4-16-2) and 28,416 (4-32-2), one up to 37,888 or 56,832, depending on
    network and outputs; sixteen or eight environments of the last warp or byte present."""
    for streams, limit, spread in (((), 0, "edge"), (ALL, 20, "wide"), (("reward_stream", "done_bits"), 0, None), (("action_bits",), 7, "edge")):
        args = dict(streams=streams, limit=limit, spread=spread, contracted=contracted)
        assert_same_bits(rollout(cp, 0, kind, n, T, **args), rollout(cp, 2, kind, n, T, **args))


@pytest.mark.parametrize("kind", [MLP, MLP32, MLP64, DEEP])
@pytest.mark.parametrize("contracted", [False, True])
@pytest.mark.parametrize("n,T", [(97, 50), (1500, 50), (4097, 50), (4737, 50), (4745, 17), (9473, 65), (14_209, 64), (18_961, 130)])
def test_networks_from_supplied_starts(cp, kind, contracted, n, T):
    """With four lanes per environment and, with outputs beyond 4,736 environments on 148 SMs, with two and one, whose lanes
    bring two and four components each; angles beyond the polynomial range, NaN and infinities among the start states."""
    for streams, limit in (((), 0), (ALL, 0), (ALL, 6), (("reward_stream", "done_bits"), 0)):
        args = dict(streams=streams, limit=limit, starts=start_rows(T, n), spread="edge", contracted=contracted)
        assert_same_bits(rollout(cp, 0, kind, n, T, **args), rollout(cp, 2, kind, n, T, **args))


@pytest.mark.parametrize("kind", [MLP, MLP32, MLP64, DEEP])
@pytest.mark.parametrize("n", [1, 8, 9, 17, 25, 1217])
def test_networks_in_place_with_warps_past_the_end(cp, kind, n):
    """A batch advanced in place whose last CTA has warps without environments: those read neither its states
    nor its episode lengths, which another warp rewrites. (That they do not is seen in the kernel; here that
    everything else is as before.)"""
    for streams in ((), ALL):
        args = dict(streams=streams, limit=60, spread="edge")
        assert_same_bits(rollout(cp, 0, kind, n, 70, **args), rollout(cp, 2, kind, n, 70, **args))


@pytest.mark.parametrize("kind", [LINEAR, PER_ENV])
@pytest.mark.parametrize("n,T", [(1, 15), (33, 32), (2049, 33), (4737, 16), (4801, 65)])
@pytest.mark.parametrize("contracted", [False, True])
def test_linear_policies(cp, kind, n, T, contracted):
    for streams, limit, spread in (((), 0, None), (ALL, 20, "wide"), (("reward_stream", "done_bits"), 0, "edge"),
                                   (("action_bits", "trajectory"), 9, None)):
        args = dict(streams=streams, limit=limit, spread=spread, contracted=contracted)
        assert_same_bits(rollout(cp, 4, kind, n, T, **args), rollout(cp, 2, kind, n, T, **args))
        assert_same_bits(rollout(cp, 0, kind, n, T, **args), rollout(cp, 2, kind, n, T, **args))


@pytest.mark.parametrize("kind", [0, LINEAR, PER_ENV, MLP])
@pytest.mark.parametrize("given", [False, True])
@pytest.mark.parametrize("n,T", [(1, 17), (33, 1), (1000, 16), (4801, 47), (2049, 97)])
def test_supplied_starts(cp, kind, given, n, T):
    bits = torch.from_numpy(np.random.default_rng(2).integers(-2**31, 2**31, (T, (n + 31) // 32)).astype(np.int32)).cuda()
    for streams, limit, spread in (((), 0, None), (ALL, 20, "wide"), (("reward_stream", "done_bits"), 0, None),
                                   (("done_bits",), 0, "edge")):
        args = dict(streams=streams, limit=limit, spread=spread, starts=start_rows(T, n), given=bits if given else None)
        general = rollout(cp, 2, kind, n, T, **args)
        for coop in (0, 4):  # what a caller gets; helper warps, which take such calls from 96 steps on
            assert_same_bits(rollout(cp, coop, kind, n, T, **args), general)


@pytest.mark.parametrize("given", [False, True])
@pytest.mark.parametrize("contracted", [False, True])
@pytest.mark.parametrize("n,T", [(31, 1), (4736, 2), (4735, 36), (4737, 35), (9472, 34), (9473, 37), (4700, 129)])
def test_hashed_and_given_actions_by_pairs_per_sm(cp, given, contracted, n, T):
    """148 SMs: three helper warps up to 4,736 environments, the cart's velocity a step behind up to 9,472, neither beyond;
    horizons around the hand-overs and the four steps of a trip."""
    bits = torch.from_numpy(np.random.default_rng(2).integers(-2**31, 2**31, (T, (n + 31) // 32)).astype(np.int32)).cuda()
    for streams, limit, spread in (((), 0, None), (("reward_stream", "done_bits"), 0, "wide"), ((), 9, "edge"),
                                   (("reward_stream", "done_bits"), 20, None), (ALL, 0, "edge")):
        args = dict(streams=streams, limit=limit, spread=spread, contracted=contracted, given=bits if given else None)
        assert_same_bits(rollout(cp, 0, 0, n, T, **args), rollout(cp, 2, 0, n, T, **args))


@pytest.mark.parametrize("kind", [0, LINEAR, PER_ENV, MLP, MLP64])
@pytest.mark.parametrize("coop", [0, 1, 2, 3])
@pytest.mark.parametrize("n,T", [(1, 5), (33, 7), (65, 3), (1000, 9), (57_001, 115), (160_001, 3)])
def test_outputs_together_equal_outputs_apart(cp, kind, coop, n, T):
    """The general kernel's instances for fixed combinations of outputs (with the action bits, all four) write what the
    instance that tests for each output writes, in every shape; the size before the last is one where all four stay tested, the last has two environments per thread."""
    words = (n + 31) // 32
    bits = torch.from_numpy(np.random.default_rng(4).integers(-2**31, 2**31, (T, words)).astype(np.int32)).cuda()
    for contracted, limit, given in ((False, 0, None), (True, 4, None), (False, 6, bits if kind == 0 else None)):
        args = dict(limit=limit, contracted=contracted, given=given, spread="edge")
        apart = rollout(cp, coop, kind, n, T, streams=("done_bits", "trajectory"), **args)
        apart |= rollout(cp, coop, kind, n, T, streams=("reward_stream", "action_bits"), **args)
        for streams in (ALL, ("reward_stream", "done_bits", "action_bits")):
            got = rollout(cp, coop, kind, n, T, streams=streams, **args)
            assert_same_bits(got, {k: apart[k] for k in got})


@pytest.mark.parametrize("n,T", [(250_003, 20), (250_003, 26), (450_003, 12)])
def test_own_policies_with_all_outputs_on_larger_batches(cp, n, T):
    """Contracted, more than 151,552 environments on 148 SMs: restarts per lane without tests of the outputs, per lane with them on
    rows off 32 bytes, by the warp on the shortest of those launches."""
    args = dict(streams=ALL, contracted=True, limit=9, spread="edge")
    general = rollout(cp, 2, PER_ENV, n, T, **args)
    for coop in (0, 1):
        assert_same_bits(rollout(cp, coop, PER_ENV, n, T, **args), general)
