"""The host side of the library (csrc/api.cu) against fakes of the CUDA runtime and of the kernel launchers
(host_runtime_fake.cpp): what a call launches, keeps and reports, without a GPU."""
import ctypes as C
import os
import subprocess

import pytest

from paper_2507_19608_b200 import _build
from paper_2507_19608_b200 import binding as B

HERE = os.path.dirname(os.path.abspath(__file__))
CUDA_INCLUDE = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(_build._nvcc()))), "include")
LAUNCH_FAILURE = 719


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("fake") / "fake.so")
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-fvisibility=hidden", "-Wl,-Bsymbolic", "-DNVTX_NO_IMPL",
                    "-DDELTA_BUILDING_LIB", "-I", CUDA_INCLUDE, "-o", so, "-x", "c++", os.path.join(_build.CSRC, "api.cu"),
                    os.path.join(HERE, "host_runtime_fake.cpp")], check=True)
    lib = C.CDLL(so)
    for name in ("delta_last_cuda_error", "fake_log"):
        getattr(lib, name).restype = C.c_char_p
    return lib


class Host:
    """A state over the fake runtime, and host buffers nothing reads."""

    def __init__(self, lib, H=32, H_kv=8, T=1024, source=B.DELTA_SRC_QUERY, dtype="bf16", Bn=1):
        self.lib, self.T, self.cfg = lib, T, B.make_config(Bn, H, H_kv, 64, T + 64, dtype, source=source)
        lib.fake_clear()
        lib.fake_device(0)
        n = C.c_size_t()
        assert lib.delta_state_workspace_bytes(C.byref(self.cfg), C.byref(n)) == 0
        self.st = C.c_void_p()
        assert lib.delta_state_init(C.byref(self.cfg), C.c_void_p(1 << 40), n, None, C.byref(self.st)) == 0
        self.buf = C.c_void_p(1 << 44)
        self.call_log()

    def prefill_host(self):
        n = C.c_size_t()
        assert self.lib.delta_prefill_staging_bytes(C.byref(self.cfg), self.T, C.byref(n)) == 0
        return self.lib.delta_attn_prefill_host(self.st, self.buf, self.buf, self.buf, self.buf, self.buf, n, self.T,
                                                C.c_float(0.3), 64, None)

    def prefill(self):
        c = self.cfg
        return self.lib.delta_attn_prefill(self.st, *[self.buf] * 4, self.T, c.H, c.H_kv, c.d, C.c_float(0.3), 64, None)

    def decode(self):
        return self.lib.delta_attn_decode_step(self.st, *[self.buf] * 6, C.c_float(0.3), 64, None)

    def reset(self):
        assert self.lib.delta_state_reset(self.st, None) == 0

    def call_log(self, nvtx=False):
        log = self.lib.fake_log().decode().splitlines()
        self.lib.fake_clear()
        return [x for x in log if nvtx or not x.startswith(("push", "pop"))]


@pytest.mark.parametrize("name", ["chain", "attn", "finish", "memcpy", "synchronize"])
def test_host_prefill_reports_the_error_of_the_failed_call(fake, name):
    h = Host(fake)
    fake.fake_fail(name.encode(), LAUNCH_FAILURE)
    assert h.prefill_host() == B.DELTA_ERR_CUDA
    assert fake.delta_last_cuda_error() == b"fakeError: code 719"
    assert h.call_log()[-1] == "synchronize"        # nothing of the call is left in flight
    assert fake.delta_state_position(h.st) == 0


def test_host_prefill_opens_an_nvtx_range(fake):
    h = Host(fake)
    assert h.prefill_host() == 0
    log = h.call_log(nvtx=True)
    assert log[0] == "push delta_attn_prefill_host" and log[-1] == "pop"
    assert sum(x.startswith("push") for x in log) == sum(x == "pop" for x in log)


def test_streams_of_the_host_prefill_are_kept_per_device(fake):
    """Six devices in turn, twice: the second round makes and destroys nothing."""
    h = Host(fake)
    for turn in range(2):
        for dev in range(10, 16):
            fake.fake_device(dev)
            h.reset()
            assert h.prefill_host() == 0
            log = h.call_log()
            assert log.count(f"stream_create dev={dev}") == (2 if turn == 0 else 0)
            assert not any("destroy" in x for x in log)


def test_host_prefill_on_a_capturing_stream_touches_nothing(fake):
    """The call synchronises, so it cannot be captured: refused before a pooled stream joins the capture."""
    h = Host(fake)
    fake.fake_capturing(1)
    status = h.prefill_host()
    fake.fake_capturing(0)
    assert status == B.DELTA_ERR_CUDA and h.call_log() == []
    assert fake.delta_last_cuda_error() == b"fakeError: code 900"       # cudaErrorStreamCaptureUnsupported
    assert h.prefill_host() == 0


@pytest.mark.parametrize("packed", [0, 1])
def test_only_a_step_behind_a_step_may_fetch_ahead_of_its_wait(fake, packed):
    """The first step behind a prefill must take what the prefill's last kernel wrote behind its wait for it."""
    h = Host(fake, source=B.DELTA_SRC_KEY)
    assert fake.delta_state_set_key_cache(h.st, packed) == 0
    for _ in range(2):
        assert h.prefill() == 0
        assert [h.decode() for _ in range(3)] == [0, 0, 0]
        assert [x[-1] for x in h.call_log() if x.startswith("decode_mma")] == ["0", "1", "1"]
        h.reset()


@pytest.mark.parametrize("source,dtype,packed,forced,reported,launched", [
    (B.DELTA_SRC_QUERY, "bf16", 0, -1, 1, "decode_mma"), (B.DELTA_SRC_QUERY, "bf16", 0, 0, 0, "decode"),
    (B.DELTA_SRC_KEY, "bf16", 0, -1, 1, "decode_mma"), (B.DELTA_SRC_KEY, "bf16", 0, 0, 0, "decode_key"),
    (B.DELTA_SRC_KEY, "bf16", 1, -1, 1, "decode_mma"), (B.DELTA_SRC_KEY, "bf16", 1, 0, 1, "decode_mma"),
    (B.DELTA_SRC_QUERY, "f32", 0, -1, 0, "decode_f32"), (B.DELTA_SRC_QUERY, "f32", 0, 0, 0, "decode")])
def test_the_reported_decode_kernel_is_the_one_that_runs(fake, source, dtype, packed, forced, reported, launched):
    h = Host(fake, source=source, dtype=dtype)
    if packed:
        assert fake.delta_state_set_key_cache(h.st, 1) == 0
    assert fake.delta_state_set_decode_kernel(h.st, forced) == 0
    assert h.prefill() == 0
    h.call_log()
    assert fake.delta_state_decode_kernel(h.st) == reported
    assert h.decode() == 0
    assert [x.split()[0] for x in h.call_log()] == [launched]


@pytest.mark.parametrize("Bn,H,H_kv,dtype,parts", [(1, 32, 8, "bf16", [16] * 2), (3, 20, 5, "bf16", [12, 16, 16, 16]),
                                                   (1, 8, 8, "f32", [4, 4])])
def test_a_call_in_parts_takes_the_form_of_the_whole_call(fake, Bn, H, H_kv, dtype, parts):
    """The attention kernels round by their form; the host-buffer call cuts a batch and must not change it."""
    h = Host(fake, H=H, H_kv=H_kv, Bn=Bn, dtype=dtype)
    assert h.prefill_host() == 0
    assert [x for x in h.call_log() if x.startswith("attn")] == [f"attn heads={n} form_heads={Bn * H}" for n in parts]


def test_compressed_cache_bytes_are_zero_before_a_prefill(fake):
    """The fill words on the device are an earlier prompt's, or unset, until a prefill has written them."""
    h = Host(fake, source=B.DELTA_SRC_KEY)
    assert fake.delta_state_set_key_cache(h.st, 1) == 0
    packed, dense = C.c_uint64(7), C.c_uint64(7)
    fake.fake_fill(0x5a)
    status = fake.delta_key_cache_bytes(h.st, C.byref(packed), C.byref(dense), None)
    fake.fake_fill(-1)
    assert (status, packed.value, dense.value) == (0, 0, 0)
