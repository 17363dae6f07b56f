"""The CPython module behind the attention calls: broken preconditions raise before anything is launched, and
leave the interpreter usable (no GPU is present in this run)."""
import threading
import time

import pytest
import torch


@pytest.fixture(scope="module")
def pa():
    import paper_2503_03588_b200 as pa_

    return pa_


def _bf16(*shape):
    return torch.zeros(shape, dtype=torch.bfloat16)


def test_broken_preconditions_raise(pa):
    q, kc, lens = _bf16(1, 4, 128), _bf16(1, 64, 2, 128), torch.ones(1, dtype=torch.int32)
    with pytest.raises(AssertionError):
        pa.pa_decode(q, kc, kc, lens.long(), 5, 1)                     # lengths of another type
    with pytest.raises(AssertionError):
        pa.pa_decode(q.transpose(1, 2), kc, kc, lens, 5, 1)            # q not contiguous
    with pytest.raises(AssertionError):
        pa.pa_decode_paged(q, kc, kc, torch.zeros((1, 1), dtype=torch.int64), lens, 5, 1)
    with pytest.raises(AssertionError):
        pa.pa_prefill(_bf16(1, 64, 4, 256)[..., ::2], kc, kc, lens, lens)   # head_dim not contiguous
    with pytest.raises(AssertionError):
        pa.pa_prefill_backward(_bf16(1, 64, 4, 128), kc, kc, _bf16(1, 64, 4, 128).float(), lens, _bf16(1, 64, 4, 128), lens, lens)
    with pytest.raises(TypeError):
        pa.pa_decode(q, None, kc, lens, 5, 1)
    with pytest.raises(TypeError):
        pa.pa_decode(q, kc, kc, lens, "5", 1)
    with pytest.raises(OverflowError):
        pa.pa_decode(q, kc, kc, lens, 1 << 40, 1)


def test_library_errors_carry_status_and_message(pa):
    if torch.cuda.is_available():
        stream_error = pa.PaError
    else:
        stream_error = (pa.PaError, RuntimeError)  # (without a driver torch itself may refuse to name a stream)
    with pytest.raises(stream_error):
        pa.pa_decode(_bf16(1, 4, 96), _bf16(1, 64, 2, 96), _bf16(1, 64, 2, 96), torch.ones(1, dtype=torch.int32), 5, 1)


def test_errors_of_torch_keep_their_class(pa):
    """A C++ exception of torch comes out as the Python exception torch itself would raise."""
    with pytest.raises(RuntimeError) as expected:
        torch.empty(1, device="vulkan")
    with pytest.raises(type(expected.value)) as got:
        pa.pa_build_layout(1000, 64, 5, 1, device="vulkan")
    assert type(got.value) is type(expected.value) is NotImplementedError


@pytest.mark.parametrize("device", [0, None, "cuda", torch.device("cuda", 0), "nowhere", 1.5])
def test_devices_are_named_as_in_torch(pa, device):
    """Layouts take what torch.empty takes for a device (None: the default one), and raise what it raises."""
    def error_of(call):
        try:
            with torch.device("cuda"):
                call()
        except Exception as e:
            return type(e)

    expected = error_of(lambda: torch.empty(1, device=device))
    for build in (lambda d: pa.pa_build_layout(1000, 64, 5, 1, device=d),
                  lambda d: pa.pa_build_window_layout(1000, 64, 5, 1, device=d),
                  lambda d: pa.pa_build_tile_layout(1000, 128, 5, 1, 64, device=d)):
        assert error_of(lambda: build(device)) is expected


def test_no_output_type_is_no_type_error(pa):
    """o_dtype None stands for torch's default type, as in torch.empty."""
    q, kc, lens = _bf16(1, 4, 128), _bf16(1, 64, 2, 128), torch.ones(1, dtype=torch.int64)
    with pytest.raises(AssertionError):   # the lengths' type, which is looked at after the output has been made
        pa.pa_decode(q, kc, kc, lens, 5, 1, o_dtype=None)


def test_other_threads_run_while_an_output_is_allocated(pa, monkeypatch):
    """An allocation that takes long (here: 160 MB filled with a pattern) does not hold the interpreter lock."""
    if torch.cuda.is_available():
        pytest.skip("the call is made to end before its launch, which takes a machine without a GPU")
    monkeypatch.setattr(torch.utils.deterministic, "fill_uninitialized_memory", True)
    torch.use_deterministic_algorithms(True)
    ticks, stop = [], threading.Event()

    def tick():
        while not stop.is_set():
            ticks.append(time.perf_counter())
            time.sleep(0.001)

    thread = threading.Thread(target=tick)
    thread.start()
    try:
        t0 = time.perf_counter()
        with pytest.raises(RuntimeError):
            pa.pa_build_window_layout(40_000_000, 1, 1, 0, col_idx=torch.empty(1, dtype=torch.int32), device="cpu")
        t1 = time.perf_counter()
    finally:
        stop.set()
        thread.join()
        torch.use_deterministic_algorithms(False)
    inside = [t0] + [t for t in ticks if t0 < t < t1] + [t1]
    assert max(b - a for a, b in zip(inside, inside[1:])) < 0.5 * (t1 - t0), (t1 - t0, len(inside))


def test_the_module_is_rebuilt_for_another_torch_or_python(pa, monkeypatch):
    """Its file is as new as before, but it fits the versions it was built against only."""
    import importlib.util
    import os

    path = os.path.join(os.path.dirname(pa.__file__), "build.py")
    spec = importlib.util.spec_from_file_location("_powerattn_build_under_test", path)
    build = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(build)
    assert not build._calls_stale([])
    version = build._torch_version()
    for name, value in (("CALLS_STAMP", build.CALLS_STAMP + ".missing"), ("_torch_version", lambda: "2.99.0"),
                        ("_torch_dir", lambda: "/elsewhere/torch")):
        with monkeypatch.context() as m:
            m.setattr(build, "_torch_version", lambda: version)   # (else read from where torch is)
            m.setattr(build, name, value)
            assert build._calls_stale([]), name


def test_status_and_message_of_the_library(pa):
    """Sizes are checked on the host, before anything that needs a GPU."""
    for call, status, message in (
            (lambda: pa.pa_build_layout(0, 64, 5, 1), 1, "seq_len must be >= 1 (got 0)"),
            (lambda: pa.pa_build_window_layout(100, 64, 0, 1), 1, "a sliding-window layout needs window_blocks >= 1"),
            (lambda: pa.pa_build_tile_layout(100, 100, 5, 1, 64), 2, "block 100 is not a multiple of tile 64")):
        with pytest.raises(pa.PaError) as e:
            call()
        assert e.value.status == status and message in str(e.value)
