"""What the compiled marshalling module refuses before any library call (no GPU needed)."""
import ctypes
import subprocess
import sys
import threading

import numpy as np
import pytest
import torch


@pytest.fixture(scope="module")
def tq():
    from paper_2402_01798_b200 import binding
    binding.lib()
    return binding


def test_wrong_arguments_raise(tq):
    g = torch.zeros(2, 16)
    ws, st, hint = torch.zeros(8, dtype=torch.uint8), torch.zeros(128, dtype=torch.uint8), torch.zeros(16, dtype=torch.uint8)
    with pytest.raises(ValueError, match="CUDA tensor"):
        tq.tq_stats(g, stats_dev=st, workspace=ws)
    with pytest.raises(ValueError, match="CUDA tensor"):
        tq.tq_stats_hinted(g, hint, stats_dev=st, workspace=ws)
    with pytest.raises(TypeError):
        tq.tq_stats([1.0, 2.0], stats_dev=st, workspace=ws)
    p = tq.tq_params_from_levels([-1.0, -0.5, 0.5, 1.0])
    with pytest.raises(ValueError, match=r"\[N, words\] CUDA tensor"):
        tq.tq_decompress_aggregate(torch.zeros((1, 4), dtype=torch.int32), 16, [p], out=torch.zeros(16))
    with pytest.raises(ValueError, match="one Params per worker"):
        tq.tq_decompress_aggregate_rows([16, 32], 16, [p], out=torch.zeros(16))
    with pytest.raises(TypeError):
        tq._calls().params_device(st)                      # too few arguments


def test_library_status_comes_back(tq):
    """Addresses and numbers reach the library unchanged: its own argument checks answer."""
    with pytest.raises(tq.TqError) as e:
        tq.tq_params_batch(b"\0" * 64, 1, 5, tq.UNIFORM, 3.0)              # five levels
    assert e.value.status == tq.ERR_INVALID_ARG
    with pytest.raises(tq.TqError) as e:
        tq.tq_params_device(torch.zeros(64, dtype=torch.uint8), 1, 4, -1, 3.0, params_dev=torch.zeros(176, dtype=torch.uint8), stream=0)
    assert e.value.status == tq.ERR_INVALID_ARG
    p = tq.tq_params_from_levels([-1.0, 1.0])
    with pytest.raises(tq.TqError) as e:
        tq.tq_decompress_aggregate_rows([20], 16, [p], out=torch.zeros(16), stream=0)      # a row off its 16-byte boundary
    assert e.value.status == tq.ERR_ALIGNMENT


def test_packed_rows_outside_the_gpu_and_with_more_dimensions(tq):
    """The fused update and the device-parameter calls read packed rows wherever the GPU can, pinned host memory included, and a
    row may be folded ([N, 2, 4]): such a block reaches the library, whose own checks answer."""
    buf = torch.zeros(20, dtype=torch.int32)
    rows = buf[(-buf.data_ptr() // 4) % 4 + 1:][:16]                                           # four bytes off a 16-byte boundary
    out, params = torch.zeros(16), torch.zeros(2 * 176, dtype=torch.uint8)
    p = tq.tq_params_from_levels([-1.0, -0.5, 0.5, 1.0])
    for packed in (rows.view(2, 8), rows.view(2, 2, 4)):
        for call in (lambda: tq.tq_decompress_aggregate_device_params(packed, 16, params, 4, out=out, stream=0),
                     lambda: tq.tq_decompress_aggregate_segments(packed, [(0, 16)], params, 4, out=out, stream=0),
                     lambda: tq.tq_decompress_aggregate_apply(packed, 16, [p, p], out, None, lr=0.1, stream=0)):
            with pytest.raises(tq.TqError) as e:
                call()
            assert e.value.status == tq.ERR_ALIGNMENT


@pytest.mark.parametrize("rows", [64, 65, 1000])
def test_weights_of_more_rows_than_the_library_takes(tq, rows):
    """One weight per row, a list too short (zeros follow) and one too long.  More than 64 rows are the library's to refuse, without a
    weight written beyond the 64 that the binding keeps; with 64 the misaligned rows are what it refuses."""
    packed = torch.zeros(4 * rows + 8, dtype=torch.int32)
    packed = packed[(-packed.data_ptr() // 4) % 4 + 1:][:4 * rows].view(rows, 4)
    out, params = torch.zeros(16), torch.zeros(176 * rows, dtype=torch.uint8)
    p = tq.tq_params_from_levels([-1.0, -0.5, 0.5, 1.0])
    for weights in ([0.5] * rows, [], (0.5,) * (rows - 1), torch.ones(rows)):
        for call in (lambda: tq.tq_decompress_aggregate_device_params(packed, 16, params, 4, weights=weights, out=out, stream=0),
                     lambda: tq.tq_decompress_aggregate_segments(packed, [(0, 16)], params, 4, weights=weights, out=out, stream=0),
                     lambda: tq.tq_decompress_aggregate_apply(packed, 16, [p] * rows, out, None, lr=0.1, weights=weights, stream=0),
                     lambda: tq.tq_decompress_aggregate_rows([8] * rows, 16, [p] * rows, weights=weights, out=out, stream=0)):
            with pytest.raises(tq.TqError) as e:
                call()
            assert e.value.status == (tq.ERR_ALIGNMENT if rows == 64 else tq.ERR_INVALID_ARG)
    for call in (lambda w: tq.tq_decompress_aggregate_device_params(packed, 16, params, 4, weights=w, out=out, stream=0),
                 lambda w: tq.tq_decompress_aggregate_apply(packed, 16, [p] * rows, out, None, lr=0.1, weights=w, stream=0)):
        with pytest.raises(IndexError):
            call([0.5] * (rows + 1))
        with pytest.raises(TypeError):
            call([0.5, None])


@pytest.mark.gpu
def test_weights_of_more_rows_than_the_library_takes_in_a_block(tq):
    """As above for the call that asks for a CUDA block."""
    p = tq.tq_params_from_levels([-1.0, 1.0])
    with pytest.raises(tq.TqError) as e:
        tq.tq_decompress_aggregate(torch.zeros((65, 4), dtype=torch.int32, device="cuda"), 16, [p] * 65, weights=[0.1] * 65)
    assert e.value.status == tq.ERR_INVALID_ARG


def test_other_threads_run_while_the_library_works(tq, tmp_path):
    """A call may last: a launch waits for room in a full queue, the parameter design of 64 records takes its time.  With a library
    function that sleeps 0.2 s in place of each of the library's, another thread goes on meanwhile."""
    (tmp_path / "slow.c").write_text("#include <unistd.h>\nint slow(void) { usleep(200000); return 0; }\n")
    subprocess.run(["gcc", "-shared", "-fPIC", "-o", str(tmp_path / "slow.so"), str(tmp_path / "slow.c")], check=True)
    slow = ctypes.CDLL(str(tmp_path / "slow.so"))
    native, at = tq._calls(), lambda f: ctypes.cast(f, ctypes.c_void_p).value
    buf, p = torch.zeros(1024, dtype=torch.int32), tq.params_array([tq.tq_params_from_levels([-1.0, 1.0])])
    packed, seg = buf.view(1, 1024), tq.segments_array([(0, 16)])
    calls = {"params_batch": (buf, 1, 16, 1, 3.0, 1, 0.0, p), "params_device": (buf, 1, 16, 1, 3.0, 1, 0.0, buf, 0),
             "decompress_aggregate_rows": ([buf], 16, p, None, buf, 0), "decompress_aggregate_apply": (packed, 16, p, [1.0], buf, None, 0.1, 0.9, 0.0, 0),
             "decompress_aggregate_device_params": (packed, 16, buf, 2, None, buf, 0), "decompress_aggregate_segments": (packed, seg, buf, 2, None, buf, 0)}
    ticks, stop = [0], threading.Event()

    def count():
        while not stop.wait(0.002):
            ticks[0] += 1

    other = threading.Thread(target=count)
    other.start()
    native.bind([at(slow.slow)] * len(tq._NATIVE))
    try:
        for name, args in calls.items():
            before = ticks[0]
            assert getattr(native, name)(*args) == tq.OK
            assert ticks[0] - before >= 10, name
    finally:
        native.bind([at(getattr(tq.lib(), name)) for name in tq._NATIVE])
        stop.set()
        other.join()


def test_stream_handles(tq):
    """A raw handle may be anything that int() takes: numpy integers, the handle objects of other libraries."""
    class Handle:
        def __int__(self):
            return 0

    p, out = tq.tq_params_from_levels([-1.0, 1.0]), torch.zeros(16)
    for stream in (0, np.int64(0), np.uint64(0), Handle()):
        with pytest.raises(tq.TqError) as e:
            tq.tq_decompress_aggregate_rows([20], 16, [p], out=out, stream=stream)
        assert e.value.status == tq.ERR_ALIGNMENT
    with pytest.raises(TypeError):
        tq.tq_decompress_aggregate_rows([20], 16, [p], out=out, stream=object())


def test_objects_with_an_address(tq):
    """Buffers that are not typed by a tensor: whatever has a data_ptr(), a storage for one."""
    class Buffer:
        def __init__(self, at):
            self.data_ptr = lambda: at

    p, t = tq.tq_params_from_levels([-1.0, 1.0]), torch.zeros(64)
    for call in (lambda: tq.tq_decompress_aggregate_rows([Buffer(20)], 16, [p], out=t, stream=0),
                 lambda: tq.tq_decompress_aggregate_rows([16], 16, [p], out=Buffer(16), stream=0),
                 lambda: tq.tq_params_device(Buffer(4), 1, 4, 0, 3.0, params_dev=t.untyped_storage(), stream=0)):
        with pytest.raises(tq.TqError) as e:
            call()
        assert e.value.status == tq.ERR_ALIGNMENT
    for bad in (object(), "text", 1.5):
        with pytest.raises(TypeError):
            tq.tq_decompress_aggregate_rows([bad], 16, [p], out=t, stream=0)


def test_records_and_weights_of_the_fused_update(tq):
    """The fused update takes the records of a larger job for its first rows, but not too few; weights are what float() takes."""
    p, t = tq.tq_params_from_levels([-1.0, 1.0]), torch.zeros(64)
    packed = torch.zeros(9, dtype=torch.int32)
    packed = packed[(-packed.data_ptr() // 4) % 4 + 1:][:4].view(1, 4)                        # misaligned: the library's check answers
    for params, weights in (([p], None), ([p, p, p], None), ((tq.Params * 2)(p, p), [np.float32(1)]), ([p], ["0.5"]), ([p], torch.ones(1)), ([p], (w for w in [1]))):
        with pytest.raises(tq.TqError) as e:
            tq.tq_decompress_aggregate_apply(packed, 16, params, t, None, lr=0.1, weights=weights, stream=0)
        assert e.value.status == tq.ERR_ALIGNMENT
    with pytest.raises(ValueError, match="one Params per worker"):
        tq.tq_decompress_aggregate_apply(packed, 16, [], t, None, lr=0.1, stream=0)
    with pytest.raises(ValueError):
        tq.tq_decompress_aggregate_apply(packed, 16, [p], t, None, lr=0.1, weights=["half"], stream=0)


def test_host_calls_do_without_the_compiled_module(tq, monkeypatch):
    """The parameter design and the sizes go through ctypes; only a call of a round asks for the module, and says what to do."""
    monkeypatch.setattr(tq, "_native", None)
    monkeypatch.setattr(tq, "_lib", None)
    monkeypatch.delattr("paper_2402_01798_b200._tq_python")
    monkeypatch.setitem(sys.modules, "paper_2402_01798_b200._tq_python", None)                # an import fails
    assert tq.tq_params_from_levels([-1.0, 1.0]).bits == 1 and tq.tq_packed_words(100, 3) == 12
    with pytest.raises(RuntimeError, match="paper_2402_01798_b200.build"):
        tq.tq_params_batch(b"\0" * 64, 1, 4, tq.UNIFORM, 3.0)


def test_module_of_another_torch(tq, monkeypatch, tmp_path):
    """torch's C++ interface changes between versions: a module of another one is refused, and built again by the next build."""
    from paper_2402_01798_b200 import build
    monkeypatch.setattr(tq, "_native", None)
    monkeypatch.setattr(build, "NATIVE_TORCH", str(tmp_path / "version"))
    ran = []
    monkeypatch.setattr(build, "_run", lambda cmd, verbose, what: (ran.append(what), open(cmd[cmd.index("-o") + 1], "w").close()))
    monkeypatch.setattr(build.os, "replace", lambda a, b: build.os.unlink(a))
    (tmp_path / "version").write_text("1.0.0")
    with pytest.raises(RuntimeError, match="torch 1.0.0"):
        tq.tq_params_batch(b"\0" * 64, 1, 4, tq.UNIFORM, 3.0)
    build.build_native()
    assert len(ran) == 1 and build.native_torch() == torch.__version__
    build.build_native()
    assert len(ran) == 1
    with pytest.raises(tq.TqError):
        tq.tq_params_batch(b"\0" * 64, 1, 4, tq.UNIFORM, 3.0)
