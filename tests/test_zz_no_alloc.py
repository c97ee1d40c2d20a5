"""The linear entry point that allocates nothing (needs a B200).

Some users of this library run where device allocation is not allowed at call time: a serving
loop whose memory pool is fixed once at start-up, a plug-in that owns only the buffers it was
handed, code between the begin and end of a latency-critical section. spec_op_linear needs a
scratch buffer from its caller; spec_op_linear_static keeps that scratch inside the library.
This file checks, through the C ABI, that the second gives the first's result, twice in a row
(the built-in scratch still holds the first call's partial sums when the second call starts),
and that a problem larger than the built-in scratch is refused with a message.

Collected last on purpose: a run that stops at the first failure has then run everything else.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

TOL = 1e-5   # the tolerance of the stand-alone linear tests: max|a-b| / max|b|


@pytest.fixture(scope="module")
def torch():
    t = pytest.importorskip("torch")
    if not t.cuda.is_available():
        pytest.skip("no CUDA device")
    return t


def _operands(torch, M, N, K, seed, dtype):
    rng = np.random.default_rng(seed)
    x = torch.from_numpy(rng.standard_normal((M, K)).astype(np.float32)).cuda().to(dtype)
    w = torch.from_numpy((rng.standard_normal((N, K)) * 0.05).astype(np.float32)).cuda().to(dtype)
    return x, w


def test_static_scratch_linear_matches_caller_scratch_linear_twice(torch):
    from paper_2503_14153_b200 import spec_op_linear, spec_op_linear_static
    # two different problems back to back: the second starts with the first's leftovers in the scratch
    cases = [(64, 1000, 704, 3, 11), (32, 384, 256, 2, 12)]
    for M, N, K, ctas, seed in cases:
        x, w = _operands(torch, M, N, K, seed, torch.bfloat16)
        want = spec_op_linear(x, w, ctas)
        y = torch.full((M, N), float("nan"), dtype=torch.float32, device="cuda")   # caller-owned output
        before = torch.cuda.memory_stats()["allocation.all.allocated"]    # cumulative count of allocations
        torch.cuda.synchronize()
        free_before = torch.cuda.mem_get_info()[0]                        # what the driver says is free on the device
        got = spec_op_linear_static(x, w, y, ctas)
        assert torch.cuda.memory_stats()["allocation.all.allocated"] == before   # none came from torch's allocator
        if (M, N, K) != cases[0][:3]:
            # (the library links the CUDA runtime statically, so an allocation of its own would not show in torch's
            # counters: after the first call, which may load the kernels' code, the device's free memory must not move)
            assert torch.cuda.mem_get_info()[0] == free_before
        torch.cuda.synchronize()
        err = (got - want).abs().max().item() / want.abs().max().item()
        assert err <= TOL, (M, N, K, ctas, err)
    # the same problem again: identical bits both times
    x, w = _operands(torch, 64, 1000, 704, 11, torch.bfloat16)
    y1 = spec_op_linear_static(x, w, torch.empty((64, 1000), dtype=torch.float32, device="cuda"), 3).clone()
    y2 = spec_op_linear_static(x, w, torch.empty((64, 1000), dtype=torch.float32, device="cuda"), 3)
    assert torch.equal(y1, y2)


def test_static_scratch_linear_float32(torch):
    from paper_2503_14153_b200 import spec_op_linear, spec_op_linear_static
    x, w = _operands(torch, 13, 301, 688, 13, torch.float32)
    want = spec_op_linear(x, w)
    got = spec_op_linear_static(x, w, torch.empty((13, 301), dtype=torch.float32, device="cuda"))
    assert (got - want).abs().max().item() / want.abs().max().item() <= TOL


def test_static_scratch_linear_refuses_oversize(torch):
    from paper_2503_14153_b200 import SpecError, spec_op_linear_static
    from paper_2503_14153_b200.binding import STATIC_SCRATCH_FLOATS
    M, N, K, ctas = 64, 32768, 256, 4
    from paper_2503_14153_b200 import load_library
    assert load_library().spec_op_linear_scratch_floats(M, N, K, ctas) > STATIC_SCRATCH_FLOATS
    x, w = _operands(torch, M, N, K, 14, torch.bfloat16)
    y = torch.empty((M, N), dtype=torch.float32, device="cuda")
    with pytest.raises(SpecError) as ei:
        spec_op_linear_static(x, w, y, ctas)
    assert ei.value.code == -3 and "exceeds the built-in scratch" in str(ei.value)


def _call(lib, entry, x, w, y, scratch, stream):
    M, K, N = x.shape[0], x.shape[1], w.shape[0]
    args = [1, x.data_ptr(), w.data_ptr(), y.data_ptr(), M, N, K, 296]
    return getattr(lib, entry)(*args, *([scratch.data_ptr()] if entry == "spec_op_linear" else []), stream.cuda_stream)


@pytest.mark.parametrize("entry,most", [("spec_op_linear_static", 0), ("spec_op_linear", 1)])
def test_no_pinned_memory_for_a_thread(entry, most):
    """In a process of its own, three threads one after another: the entry without allocations makes no pinned memory either, in no
    thread, and the other entry one block in all, whatever the number of threads that call it."""
    import subprocess
    import sys
    code = f"""
import sys, threading
sys.path[:0] = {[p for p in sys.path if p]!r}
import torch
import test_zz_no_alloc as T
from paper_2503_14153_b200 import load_library
lib = load_library()
x, w = T._operands(torch, 64, 1000, 704, 15, torch.bfloat16)
y, scratch, stream = torch.zeros((64, 1000), device="cuda"), torch.empty(int(lib.spec_op_linear_scratch_floats(64, 1000, 704, 296)) + 4, device="cuda"), torch.cuda.Stream()
torch.cuda.synchronize()
for _ in range(3):
    t = threading.Thread(target=lambda: print(T._call(lib, {entry!r}, x, w, y, scratch, stream), lib.spec_debug_pinned_allocations()))
    t.start(); t.join()
"""
    out = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, timeout=300)
    assert out.stdout.split() == ["0", str(most)] * 3, out.stdout + out.stderr


def test_linear_from_many_threads(torch):
    """Sixteen threads on streams of their own, ten calls each: every call reports its own status and its own result."""
    import threading
    from paper_2503_14153_b200 import load_library
    lib = load_library()
    ops = [_operands(torch, 16, 500 + 8 * i, 256, 30 + i, torch.bfloat16) for i in range(16)]
    outs = [torch.zeros((16, w.shape[0]), device="cuda") for _, w in ops]
    scratch = [torch.empty(int(lib.spec_op_linear_scratch_floats(16, w.shape[0], 256, 296)) + 4, device="cuda") for _, w in ops]
    streams = [torch.cuda.Stream() for _ in ops]
    torch.cuda.synchronize()
    got = [[] for _ in ops]

    def work(i):
        torch.cuda.set_device(0)
        for _ in range(10):
            got[i].append(_call(lib, "spec_op_linear", *ops[i], outs[i], scratch[i], streams[i]))
    threads = [threading.Thread(target=work, args=(i,)) for i in range(16)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    for i, (x, w) in enumerate(ops):
        want = x.double() @ w.double().T
        assert got[i] == [0] * 10
        assert (outs[i] - want).abs().max().item() / want.abs().max().item() <= TOL
        assert (scratch[i][-4:].view(torch.int32) == 0).all()


@pytest.mark.parametrize("pinned", [1, 0])
def test_wait_that_runs_out_is_reported(torch, pinned):
    """A kernel's wait that runs out reaches the caller of a stand-alone operation, through the pinned word as through the caller's own:
    the code, the status in the caller's words, and a clean call after it, from which nothing of it remains."""
    from paper_2503_14153_b200 import load_library
    lib = load_library()
    stream = torch.cuda.Stream()
    x, w = _operands(torch, 16, 500, 256, 50, torch.bfloat16)
    y, scratch = torch.zeros((16, 500), device="cuda"), torch.zeros(int(lib.spec_op_linear_scratch_floats(16, 500, 256, 296)) + 4, device="cuda")
    words = scratch[-4:]
    torch.cuda.synchronize()
    for _ in range(2):
        assert lib.spec_debug_op_wait_timeout(1000, pinned, words.data_ptr(), stream.cuda_stream) == -6      # SPEC_E_TIMEOUT
        torch.cuda.synchronize()
        assert words.view(torch.int32)[:2].tolist() == [1, 99]
        assert _call(lib, "spec_op_linear", x, w, y, scratch, stream) == 0
        torch.cuda.synchronize()
        assert words.view(torch.int32)[0].item() == 0
        assert (y - x.double() @ w.double().T).abs().max().item() <= TOL * y.abs().max().item()
    assert lib.spec_debug_op_wait_timeout(0, pinned, words.data_ptr(), stream.cuda_stream) == -1
