"""The network policies' screen: most actions come from an estimate of the logits' difference, the rest from
the defined logits. The last layer scaled by 2^100 scales every logit exactly, so the actions stay, but puts
the estimate's bound at infinity: then every action comes from the defined logits. Both must give the same
bits, also where the logits nearly or always coincide, and from states that hold NaN and infinities."""
import numpy as np
import pytest

from tests import gpu_helpers as H
from tests.test_gpu_feedback_small import ALL, DEEP, MLP, MLP32, MLP64, assert_same_bits, cp, torch  # noqa: F401

pytestmark = pytest.mark.gpu


def weights(kind, apart):
    """The policy of a seed, its second logit's weights moved to within `apart` of the first's."""
    from paper_2301_13062_b200 import inputs
    w = inputs.policy_weights(kind, 11)
    h = {MLP: 16, MLP32: 32, MLP64: 64, DEEP: 16}[kind]
    last = w[w.size - 2 * h - 2:]
    rows, bias = last[:2 * h].reshape(2, h), last[2 * h:]
    rows[1] = rows[0] + np.float32(apart) * (rows[1] - rows[0])
    bias[1] = bias[0] + np.float32(apart) * (bias[1] - bias[0])
    return w, w.size - 2 * h - 2


def rollout(cp, coop, w, kind, n, T, streams, limit, contracted):  # noqa: F811
    from paper_2301_13062_b200 import inputs
    words = (n + 31) // 32
    shapes = {"done_bits": ((T, words), torch.int32), "action_bits": ((T, words), torch.int32),
              "reward_stream": ((T, n), torch.float32), "trajectory": ((T, 4, n), torch.float32)}
    out = {"ep_return_sum": torch.zeros(n, device="cuda"), "ep_count": torch.zeros(n, dtype=torch.int32, device="cuda")}
    for name in streams:
        out[name] = torch.zeros(shapes[name][0], dtype=shapes[name][1], device="cuda")
    planes = torch.from_numpy(inputs.random_states(n, 5, "edge")).cuda()
    planes[1, ::7] = float("nan")
    planes[3, 3::11] = float("inf")
    planes[0, 5::13] = float("-inf")
    ep_len = torch.arange(n, dtype=torch.int32, device="cuda") % 17
    with H.rollout_shape(cp, 1 if coop else 0, coop):
        cp.cp_rollout_ex(T=T, state=cp.cp_wrap(planes, n, 9, t=11, env_offset=6), ep_len=ep_len, policy=cp.policy(kind, w),
                         max_episode_steps=limit, arithmetic=cp.CP_ARITH_CONTRACTED if contracted else cp.CP_ARITH_EXACT, **out)
    torch.cuda.synchronize()
    return {k: v.cpu().numpy() for k, v in {**out, "planes": planes, "ep_len": ep_len}.items()}


@pytest.mark.parametrize("kind", [MLP, MLP32, MLP64, DEEP])
@pytest.mark.parametrize("contracted", [False, True])
@pytest.mark.parametrize("apart", [1.0, 1e-3, 0.0])
def test_estimates_decide_as_the_defined_logits_do(cp, kind, contracted, apart):  # noqa: F811
    w, last = weights(kind, apart)
    scaled = w.copy()
    scaled[last:] *= np.float32(2.0**100)
    # sizes: one environment, either side of a bit-plane word, and the kernel a caller gets for larger batches (148 SMs:
    # two lanes per environment at 4,737 for 4-16-2 and 4-32-2, which keeps them without outputs at 9,473; one lane at 9,473
    # for the others but 4-64-2, for that one at 14,209); coop 2 / 5: the general kernel and the deferred-restart kernel wherever it applies
    for coop, n, T, streams, limit in ((0, 1, 40, (), 0), (0, 33, 33, ALL, 20), (0, 1200, 35, (), 9), (2, 97, 40, ALL, 0),
                                       (2, 65, 40, (), 20), (5, 129, 45, (), 0), (0, 70_001, 14, (), 0),
                                       (0, 4737, 33, (), 9), (0, 4737, 33, ALL, 0), (0, 9473, 33, (), 0), (0, 9473, 33, ALL, 20),
                                       (0, 14_209, 33, (), 20), (0, 14_209, 33, ALL, 0),
                                       (5, 129, 45, ("reward_stream", "done_bits"), 20)):
        args = (kind, n, T, streams, limit, contracted)
        assert_same_bits(rollout(cp, coop, w, *args), rollout(cp, coop, scaled, *args))


def test_tanh_of_the_special_function_unit(cp):  # noqa: F811
    out = torch.zeros(3, dtype=torch.int64, device="cuda")
    cp.cp_selftest_screen(out)
    exact, contracted, odd = out.tolist()
    # every float32; 8.0e-6 is what the bound of the estimates rests on
    assert 7_000_000 < exact <= 8_000_000 and 7_000_000 < contracted <= 8_000_000 and odd == 0
