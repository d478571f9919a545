"""The four-environments-per-thread step for planes that do not start on 16 bytes: same bits as the
one-environment-per-thread step, around its tiles of 128 environments, with every optional argument,
in place and out of place."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def cp():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2301_13062_b200 import binding, build
    build.build()
    binding.lib()
    torch.cuda.set_device(0)
    yield binding
    binding.cp_tune("step_vec_min_envs", 262144)


def step(cp, min_envs, n, pad, given, limit, in_place, wanted, offset):
    from paper_2301_13062_b200 import inputs
    if (n + pad) % 4 == 0:
        offset = 1                                                  # or the float4 form would take the call
    z = np.concatenate([inputs.random_states(n - n // 3, 4, "wide"), inputs.random_states(n // 3, 5, "edge")], 1) if n > 3 \
        else inputs.random_states(n, 4, "edge")
    store = torch.zeros(4 * (n + pad) + 1, device="cuda")          # planes from the first float on, or from the second
    planes = store[offset:offset + 4 * (n + pad)].view(4, n + pad)
    planes[:, :n] = torch.from_numpy(z).cuda()
    out = planes if in_place else torch.full((4, n + pad), 7.0, device="cuda")
    action = torch.from_numpy(inputs.random_actions(n, 8)).cuda() if given else None
    reward, done = torch.full((n,), 7.0, device="cuda"), torch.full((n,), 7, dtype=torch.uint8, device="cuda")
    ep_len = torch.arange(n, dtype=torch.int32, device="cuda") % 50 if limit else None
    a = cp.cp_wrap(planes, n, 3, t=21, env_offset=5)
    b = a if in_place else cp.cp_wrap(out, n, 3)
    cp.cp_tune("step_vec_min_envs", min_envs)
    cp.cp_step_ex(a, action, b, reward if wanted else None, done if wanted else None, ep_len, limit)
    torch.cuda.synchronize()
    r = {"planes": out, "reward": reward, "done": done}
    if limit:
        r["ep_len"] = ep_len
    return {k: v.cpu().numpy().tobytes() for k, v in r.items()}


@pytest.mark.parametrize("n", [1, 2, 31, 33, 127, 128, 129, 255, 257, 4099])
@pytest.mark.parametrize("pad,offset", [(0, 1), (1, 0), (2, 0)])
@pytest.mark.parametrize("given,limit,in_place,wanted", [(False, 0, False, True), (True, 0, True, True),
                                                         (True, 40, False, True), (False, 40, True, False)])
def test_same_bits_as_one_environment_per_thread(cp, n, pad, offset, given, limit, in_place, wanted):
    assert step(cp, 1, n, pad, given, limit, in_place, wanted, offset) == \
        step(cp, 1 << 30, n, pad, given, limit, in_place, wanted, offset)
