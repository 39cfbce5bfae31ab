"""Stream and event handling of the runtime, on the CPU: the host object linked
with a CUDA runtime that runs nothing but keeps the order of launches, event
records and event waits (fake_cuda.cpp)."""
import ctypes as C
import os
import subprocess

import pytest

from paper_2608_00573_gb300 import binding as B
from paper_2608_00573_gb300 import build as BUILD
from paper_2608_00573_gb300 import workload as W
from tests.oracle_helpers import small_cfg

HERE = os.path.dirname(os.path.abspath(__file__))


class Stream:
    """What the binding reads of a torch stream."""

    def __init__(self, fake, ptr=0x500, priority=0):
        self.cuda_stream = ptr
        fake.fake_stream(C.c_void_p(ptr), priority)


@pytest.fixture(scope="module")
def fake_path(tmp_path_factory):
    BUILD.build()
    out = str(tmp_path_factory.mktemp("fake") / "libtrimmoe_fake.so")
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(BUILD.nvcc()))), "include")
    subprocess.check_call(["g++", "-shared", "-fPIC", "-std=c++17", "-Wl,-Bsymbolic", "-I", inc,
                           os.path.join(HERE, "fake_cuda.cpp"), os.path.join(BUILD.BUILD, "trimmoe.o"), "-o", out, "-ldl"])
    return out


@pytest.fixture
def fake(fake_path, monkeypatch):
    monkeypatch.setattr(B, "LIB_PATH", fake_path)
    monkeypatch.setattr(B, "_lib", None)
    L = B.lib()
    L.fake_launch_name.restype = C.c_char_p
    L.fake_launch_stream.restype = C.c_void_p
    L.fake_launch_stream.argtypes = L.fake_launch_name.argtypes = [C.c_int]
    L.fake_reset()
    return L


def engine(cfg, **kw):
    small = W.make_small_weights(cfg, calib={"exit_bias": [1.0] * cfg.N})
    tables = W.make_tables(cfg, small["W_r"], calib={"theta": [0.6] * cfg.N})
    eng = B.Engine(cfg, tables, small, W.make_expert_weights_host(cfg), T_max=cfg.T, device="cpu", **kw)
    return eng, eng.tokens_to_device(W.make_tokens(cfg))


def launches(fake):
    return [(fake.fake_launch_name(i).decode(), fake.fake_launch_stream(i)) for i in range(fake.fake_launches())]


def shared_cfg(**kw):
    return small_cfg(**{**dict(name="streams", N=2, d=256, E=4, k=2, F=128, F_sh=256, T=40, M=4, H=2, seed=71), **kw})


@pytest.mark.parametrize("profile", [1, 2])
def test_replayed_launch_times_are_all_read(fake, profile):
    """Replays in a row without a host wait, then another batch size: every GEMM
    launch that is counted is timed, and reading the times leaves no error for
    the next launch to report."""
    eng, tok = engine(shared_cfg(), profile=profile, graphs=True)
    st = Stream(fake)
    for T in (40, 24, 40):
        for _ in range(5):          # plain, then replays of both instances
            eng.forward(tok, T=T, stream=st)
    s = eng.stats()
    assert s["n_gemm_up"] == s["n_gemm_down"] == 15 * 4
    assert s["ms_gemm_up"] + s["ms_gemm_down"] == s["n_gemm_up"] + s["n_gemm_down"]
    eng.close()


@pytest.mark.parametrize("profile", [0, 1, 2])
def test_timed_launches_do_not_overlap(fake, profile):
    """With profiling every GEMM launch is on the caller's stream, so that the
    times of the launches add up; without, the shared expert's two run beside
    the routed ones."""
    cfg = shared_cfg()
    eng, tok = engine(cfg, profile=profile)
    st = Stream(fake)
    eng.layer_step(1, tok, stream=st)
    on = [s == st.cuda_stream for name, s in launches(fake) if name == "gemm"]
    assert len(on) == 4 and on.count(False) == (0 if profile else 2)
    eng.close()


@pytest.mark.parametrize("what", ["launch", "record"])
def test_failed_call_leaves_no_work_behind_on_the_side_stream(fake, what):
    """Whichever launch or event record of a layer step fails, the caller's stream
    (or the host) has waited for everything that the call put on the side stream:
    the look-ahead tables beside the router, the shared expert's GEMMs beside the
    routed ones."""
    eng, tok = engine(shared_cfg(N=3, T=600))
    st = Stream(fake)
    eng.layer_step(1, tok, stream=st)
    names = launches(fake)
    side = [name for name, s in names if s != st.cuda_stream]
    assert sorted(side) == ["gemm", "gemm", "tables"] and fake.fake_unordered(C.c_void_p(st.cuda_stream)) == 0
    failures = 0
    for n in range(len(names) + 1):
        fake.fake_reset()
        getattr(fake, f"fake_fail_{what}")(n)
        try:
            eng.layer_step(1, tok, stream=st)
        except B.TrimmoeError:
            failures += 1
        assert fake.fake_unordered(C.c_void_p(st.cuda_stream)) == 0, (what, n)
    assert failures == (len(names) if what == "launch" else 4)
    fake.fake_reset()
    eng.layer_step(1, tok, stream=st)
    eng.close()


def test_side_stream_has_the_callers_priority(fake):
    """The shared expert's GEMMs and the tables beside the router keep the
    priority of the stream that the call came on, also when a program changes
    between streams; the default streams have the default priority."""
    eng, tok = engine(shared_cfg(N=3, T=600))
    for ptr, prio in ((0x500, 0), (0x600, -5), (0x700, -2), (0x800, -5), (0x500, 0)):
        st = Stream(fake, ptr, prio)
        fake.fake_reset()
        eng.layer_step(1, tok, stream=st)
        side = [s for name, s in launches(fake) if s != ptr]
        assert len(side) == 3 and {fake.fake_priority(C.c_void_p(s)) for s in side} == {prio}
    for ptr in (0, 1, 2):       # the default stream, legacy and per thread
        fake.fake_reset()
        eng.layer_step(1, tok, stream=type("S", (), {"cuda_stream": ptr})())
        side = [s for name, s in launches(fake) if s not in (ptr, None)]
        assert len(side) == 3 and {fake.fake_priority(C.c_void_p(s)) for s in side} == {0}
    eng.close()
