"""cp_step_host on page-locked buffers (the kernel works on host memory, in pieces on large batches) gives what it gives on pageable
ones (copies), with and without actions, in place, at ragged sizes, from misaligned and overlapping buffers, and works on what
earlier work on the caller's stream has left in them."""
import ctypes

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
    return binding


def buffers(n, pinned, offset, form):
    from paper_2301_13062_b200 import inputs

    def make(count, dtype):
        t = torch.full((count + 4,), 7, dtype=dtype)
        return (t.pin_memory() if pinned else t)[offset:offset + count]

    z = torch.from_numpy(inputs.random_states(n, 6, "edge")).reshape(-1)
    planes = make(4 * n, torch.float32)
    planes.copy_(z)
    out = planes if form == "in place" else make(4 * n, torch.float32)
    reward, done = make(n, torch.float32), make(n, torch.uint8)
    if form == "overlap":  # reward lies in the input planes: only the copies' order is defined
        reward = planes[:n]
    action = make(n, torch.uint8)
    action.copy_(torch.from_numpy(inputs.random_actions(n, 3)))
    for t in (planes, out, reward, done, action):
        assert t.is_pinned() == pinned
    return planes, action, out, reward, done


@pytest.mark.parametrize("n", [1, 33, 4099, 70_001, 262_143, 262_145])
@pytest.mark.parametrize("offset", [0, 1])
@pytest.mark.parametrize("form", ["apart", "in place", "overlap"])
@pytest.mark.parametrize("given", [False, True])
def test_page_locked_equals_pageable(cp, n, offset, form, given):
    got = []
    for pinned in (True, False):
        planes, action, out, reward, done = buffers(n, pinned, offset, form)
        cp.cp_step_host(n, 9, 4, planes, action if given else None, out, reward, done)
        got.append([t.numpy().tobytes() for t in (planes, out, reward, done)])
    assert got[0] == got[1]


@pytest.mark.parametrize("n,offset,form", [(450_001, 0, "apart"), (800_003, 1, "in place"), (1_500_001, 1, "apart"), (1_536_000, 0, "in place")])
@pytest.mark.parametrize("given", [False, True])
def test_pieces_equal_pageable(cp, n, offset, form, given):
    """Three, four and six pieces, the last of them ragged, on rows that start anywhere between two lines."""
    got = []
    for pinned in (True, False):
        planes, action, out, reward, done = buffers(n, pinned, offset, form)
        cp.cp_step_host(n, 9, 4, planes, action if given else None, out, reward, done)
        got.append([t.numpy().tobytes() for t in (planes, out, reward, done)])
    assert got[0] == got[1]


@pytest.mark.parametrize("n", [70_001, 450_001, 1_500_001])
@pytest.mark.parametrize("own_stream", [False, True])
def test_reads_what_earlier_work_on_the_stream_writes(cp, n, own_stream):
    """Inputs that a copy on the current stream fills after 10 ms of other work there: one kernel on host memory, two and six
    pieces, whose copies in run on a stream that only an event orders after the caller's."""
    from paper_2301_13062_b200 import inputs
    planes, action, out, reward, done = buffers(n, False, 0, "apart")
    cp.cp_step_host(n, 9, 4, planes, action, out, reward, done)
    want = [t.numpy().tobytes() for t in (out, reward, done)]
    source = torch.from_numpy(inputs.random_states(n, 6, "edge")).reshape(-1).cuda()
    chosen = torch.from_numpy(inputs.random_actions(n, 3)).cuda()
    late, action, out, reward, done = buffers(n, True, 0, "apart")
    cp.cp_step_host(n, 9, 4, late, action, out, reward, done)   # whatever the library makes once
    late.zero_()
    action.zero_()
    torch.cuda.synchronize()
    with torch.cuda.stream(torch.cuda.Stream() if own_stream else torch.cuda.default_stream()):
        torch.cuda._sleep(20_000_000)
        late.copy_(source, non_blocking=True)
        action.copy_(chosen, non_blocking=True)
        cp.cp_step_host(n, 9, 4, late, action, out, reward, done)
    assert [t.numpy().tobytes() for t in (out, reward, done)] == want


def test_a_capturing_stream_is_refused_and_left_usable(cp):
    """A call that waits for its result cannot be captured: an error, as with pageable buffers, no work on the copy stream,
    and the next call outside the capture is as before."""
    n = 450_001
    planes, action, out, reward, done = buffers(n, True, 0, "apart")
    cp.cp_step_host(n, 9, 4, planes, action, out, reward, done)
    want = [t.numpy().tobytes() for t in (out, reward, done)]
    cudart, graph = ctypes.CDLL("libcudart.so.12"), ctypes.c_void_p()
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        assert cudart.cudaStreamBeginCapture(ctypes.c_void_p(s.cuda_stream), 1) == 0   # thread-local
        try:
            with pytest.raises(cp.CartpoleError):
                cp.cp_step_host(n, 9, 4, planes, action, out, reward, done)
        finally:
            assert cudart.cudaStreamEndCapture(ctypes.c_void_p(s.cuda_stream), ctypes.byref(graph)) != 0
        cudart.cudaGetLastError()
    out.zero_()
    cp.cp_step_host(n, 9, 4, planes, action, out, reward, done)
    assert [t.numpy().tobytes() for t in (out, reward, done)] == want
