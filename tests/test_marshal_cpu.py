"""The marshalling module's own checks: what it refuses before the library is called, and how it calls (no GPU needed)."""
import collections
import ctypes
import re
import subprocess
import threading
import time

import pytest
import torch


@pytest.fixture(scope="module")
def B():
    from paper_2507_12000_b200 import build

    build.build()
    from paper_2507_12000_b200 import binding

    return binding


def _out(n=1):
    return {"accept_len": torch.zeros(n, dtype=torch.int32), "p_row": torch.zeros(n, 8), "token": torch.zeros(n, dtype=torch.int32)}


def test_refusals(B):
    tl, ws = torch.zeros(1, 2, 8), torch.zeros(256, dtype=torch.uint8)
    with pytest.raises(AssertionError):  # not a CUDA tensor
        B.dssd_edge_verify(tl, None, None, None, 1.0, out=_out(), workspace=ws)
    with pytest.raises(TypeError):       # not a tensor
        B.dssd_edge_verify([1.0], None, None, None, 1.0, out=_out(), workspace=ws)
    with pytest.raises(AssertionError):
        B.dssd_device_resample(torch.zeros(1, 8), None, torch.zeros(1, dtype=torch.int32), torch.zeros(1), 0, out=_out(), workspace=ws)
    with pytest.raises(TypeError):       # wrong number of arguments
        B._marshal.edge_verify(tl)
    with pytest.raises(KeyError):        # a required output is missing
        B.dssd_round_host({"target_logits": tl, "uniforms_rs": torch.zeros(1)}, 1.0, ws, out={}, stream=0)
    with pytest.raises(TypeError):       # half precision logits are no payload of this library
        B.dssd_round_host({"target_logits": tl.half(), "uniforms_rs": torch.zeros(1)}, 1.0, ws, out=_out(), stream=0)


def test_statuses_come_through(B):
    host = {"target_logits": torch.zeros(1, 1, 8), "uniforms_rs": torch.zeros(1)}
    with pytest.raises(B.DssdError) as e:  # temperature 0 is refused by the library itself
        B.dssd_round_host(host, 0.0, torch.zeros(256, dtype=torch.uint8), out=_out(), stream=0)
    assert e.value.status == B.DSSD_ERR_INVALID_ARG


@pytest.fixture()
def slow_library(B, tmp_path):
    """In the library's place one whose every entry point takes 0.2 s, notes its last argument and succeeds."""
    calls = re.findall(r"X\((dssd_\w+)\)", open(B._PKG + "/csrc/marshal.cpp").read())
    src = tmp_path / "slow.c"
    host = ("const void *target_logits, int dtype, const void *a, const void *b, const void *c, const void *d, const void *e, float T, "
            "int B, int gamma, int V, void *f, void *g, void *h, void *i, void *j, void *arena, unsigned long bytes, void *stream")
    src.write_text("#include <unistd.h>\nvoid *last_stream;\n" + "".join(
        f"int {n}({host}) {{ last_stream = stream; usleep(200000); return 0; }}\n" if n == "dssd_round_host" else
        f"int {n}(void) {{ usleep(200000); return 0; }}\n" for n in calls))
    so = tmp_path / "libslow.so"
    subprocess.run(["gcc", "-shared", "-fPIC", "-o", str(so), str(src)], check=True)
    slow = ctypes.CDLL(str(so))
    B._marshal.bind(slow._handle)
    yield slow
    B._marshal.bind(B.lib._handle)


@pytest.mark.parametrize("topk", [False, True])
def test_other_threads_run_during_a_call(B, slow_library, topk):
    host = {"target_logits": torch.zeros(1, 1, 8), "uniforms_rs": torch.zeros(1)}
    arena, out = torch.zeros(256, dtype=torch.uint8), _out()
    started, stop, during = threading.Event(), threading.Event(), []

    def count():
        started.set()
        while not stop.is_set():
            during.append(time.monotonic())
            time.sleep(0.002)

    t = threading.Thread(target=count)
    t.start()
    started.wait()
    begin = time.monotonic()
    if topk:
        B.dssd_round_host_topk(host, 1.0, 4, arena, out=out, stream=0)
    else:
        B.dssd_round_host(host, 1.0, arena, out=out, stream=0)
    end = time.monotonic()
    stop.set()
    t.join()
    # a thread that waits for the lock may run once on either side of the call, and no more
    assert end - begin > 0.19
    assert sum(begin + 0.02 < x < end - 0.02 for x in during) > 5


class _Handle:
    """A stream as other packages wrap it: converts to the integer."""

    def __int__(self):
        return 0x1234


@pytest.mark.parametrize("stream,value", [(0x1234, 0x1234), (_Handle(), 0x1234), (0, None)])
def test_streams(B, slow_library, stream, value):
    host = {"target_logits": torch.zeros(1, 1, 8), "uniforms_rs": torch.zeros(1)}
    B.dssd_round_host(host, 1.0, torch.zeros(256, dtype=torch.uint8), out=_out(), stream=stream)
    assert ctypes.c_void_p.in_dll(slow_library, "last_stream").value == value
    with pytest.raises((TypeError, AttributeError)):
        B.dssd_round_host(host, 1.0, torch.zeros(256, dtype=torch.uint8), out=_out(), stream=object())


def test_mappings_other_than_dict(B, slow_library):
    """Anything with [] and get: tensors that only the mapping's answer holds live until the call returns."""
    class Made(collections.UserDict):
        def __getitem__(self, name):
            return super().__getitem__(name).clone()

    host = Made(target_logits=torch.zeros(1, 1, 8), uniforms_rs=torch.zeros(1))
    out = collections.UserDict(_out())
    assert B.dssd_round_host(host, 1.0, torch.zeros(256, dtype=torch.uint8), out=out, stream=0) is out
    with pytest.raises(KeyError):
        B.dssd_round_host(host, 1.0, torch.zeros(256, dtype=torch.uint8), out=collections.UserDict(), stream=0)
    with pytest.raises((TypeError, AttributeError)):
        B.dssd_round_host(host, 1.0, torch.zeros(256, dtype=torch.uint8), out=[1], stream=0)
