"""The library's host code on a fake CUDA runtime (fake_cudart.cpp), without a
GPU: the order of what it puts on its streams, and what it does when a call
fails or another device is current.  Kernels do not run here."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

import paper_2001_09792_gb300 as rg
from paper_2001_09792_gb300 import _build

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def fake_lib(tmp_path_factory):
    _build.build()
    objs = [os.path.join(_build.OUT, s.replace(".cu", ".o")) for s in _build.SOURCES]
    if not all(os.path.exists(o) for o in objs):
        _build.build(force=True)
    out = str(tmp_path_factory.mktemp("fake") / "librg_fake.so")
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(_build.nvcc()))), "include")
    subprocess.run(["g++", "-shared", "-fPIC", "-O1", "-std=c++17", "-w", "-fno-gnu-unique", f"-I{inc}",
                    os.path.join(HERE, "fake_cudart.cpp"), *objs, "-o", out, "-Wl,-Bsymbolic", "-Wl,--no-undefined",
                    "-lpthread"], check=True)
    L = ctypes.CDLL(out)
    L.fake_log.restype = L.fake_kernels.restype = ctypes.c_char_p
    L.fake_stream.restype = L.fake_cleared.restype = ctypes.c_void_p
    L.rg_last_error.restype = ctypes.c_char_p
    return L


class Host:
    """The library on the fake runtime, with meshes in host memory."""

    def __init__(self, L):
        self.L = L
        self.scenes = []

    def stream(self, prio=0):
        return ctypes.c_void_p(self.L.fake_stream(prio))

    def log(self):
        return self.L.fake_log().decode().splitlines()

    def scene(self, flags=0):
        h = ctypes.c_void_p()
        desc = rg.rg_scene_desc((ctypes.c_float * 3)(0, 0, 0), 0.1, flags)
        assert self.L.rg_scene_create(ctypes.byref(h), ctypes.byref(desc)) == 0
        self.scenes.append(h)
        return h

    def destroy(self, h):
        self.scenes.remove(h)
        assert self.L.rg_scene_destroy(h) == 0

    def blas(self, h, nt=12, flags=0, stream=None):
        v, i = np.zeros((8, 3), np.float32), np.zeros((nt, 3), np.uint32)
        bid = ctypes.c_uint32()
        return self.L.rg_blas_build(h, v.ctypes.data_as(ctypes.c_void_p), 8, i.ctypes.data_as(ctypes.c_void_p), nt, flags,
                                    ctypes.byref(bid), stream)

    def renderable(self, flags=0):
        """A scene of one mesh and instance with a material and a light."""
        h = self.scene(flags)
        assert self.blas(h) == 0
        inst = np.zeros((1, 16), np.float32)
        assert self.L.rg_tlas_build(h, inst.ctypes.data_as(ctypes.c_void_p), 1, None) == 0
        mat = rg.rg_material(0, (ctypes.c_float * 3)(1, 1, 1), 1.0)
        light = rg.rg_light((ctypes.c_float * 3)(0, 1, 0), (ctypes.c_float * 3)(1, 1, 1))
        assert self.L.rg_scene_set_materials(h, ctypes.byref(mat), 1) == 0
        assert self.L.rg_scene_set_lights(h, ctypes.byref(light), 1) == 0
        return h

    def render(self, h, stream=None, size=512, depth=2):
        """The status of one frame, and what it put on the streams."""
        at = len(self.log())
        r = self.L.rg_render(h, ctypes.byref(rg.rg_camera()), size, size, depth, ctypes.c_void_p(1 << 20), stream)
        return r, self.log()[at:]


def launches(log):
    """The streams of a log's kernel launches, in order."""
    return [line.split()[2] for line in log if line.startswith("launch ")]


@pytest.fixture
def host(fake_lib):
    fake_lib.cudaSetDevice(0)
    fake_lib.fake_reset()
    H = Host(fake_lib)
    yield H
    for h in list(H.scenes):
        H.destroy(h)
    fake_lib.fake_finish()
    fake_lib.cudaSetDevice(0)


def test_growing_the_blas_table_waits_for_builds_on_other_streams(host):
    """The table of BLAS descriptors is copied when it grows; a build on another
    stream writes its descriptor and root box there, so the copy comes after
    it."""
    h, a, b = host.scene(), host.stream(), host.stream()
    assert [host.blas(h, stream=a) for _ in range(16)] == [0] * 16
    assert "devsync" not in host.log()   # (the first table holds 16)
    at = len(host.log())
    assert host.blas(h, stream=b) == 0
    new = host.log()[at:]
    copy = next(k for k, line in enumerate(new) if line.startswith(f"copy s{b.value // 16} "))
    assert "devsync" in new[:copy]


def test_scene_creation_waits_for_its_clear(host):
    """The clear of the status word is queued on the default stream; calls on
    streams that do not wait for that one come after it all the same."""
    host.scene()
    log = host.log()
    assert "streamsync s0" in log[log.index("memset s0"):]


def test_shared_scene_creation_waits_for_its_copies(host):
    h = host.scene()
    light = rg.rg_light((ctypes.c_float * 3)(0, 1, 0), (ctypes.c_float * 3)(1, 1, 1))
    assert host.L.rg_scene_set_lights(h, ctypes.byref(light), 1) == 0
    at = len(host.log())
    out = ctypes.c_void_p()
    assert host.L.rg_scene_create_shared(ctypes.byref(out), h) == 0
    host.scenes.append(out)
    new = host.log()[at:]
    last_copy = max(k for k, line in enumerate(new) if line == "copy s0")
    assert "streamsync s0" in new[last_copy:]


@pytest.mark.parametrize("call", ["materials", "lights", "sync", "reset"])
def test_calls_wait_for_their_copies_and_clears(host, call):
    """What a call writes to the scene through the default stream is in place
    when it returns: the next one may come on a stream that does not wait."""
    h = host.scene()
    status = host.L.fake_cleared()   # (the scene's status word, its error code first)
    mat = rg.rg_material(0, (ctypes.c_float * 3)(1, 1, 1), 1.0)
    light = rg.rg_light((ctypes.c_float * 3)(0, 1, 0), (ctypes.c_float * 3)(1, 1, 1))
    at = len(host.log())
    if call == "materials":
        assert host.L.rg_scene_set_materials(h, ctypes.byref(mat), 1) == 0
    elif call == "lights":
        assert host.L.rg_scene_set_lights(h, ctypes.byref(light), 1) == 0
    elif call == "sync":
        ctypes.c_int.from_address(status).value = rg.RG_ERR_STACK
        assert host.L.rg_sync(h) == rg.RG_ERR_STACK and host.L.rg_sync(h) == 0
    else:
        assert host.L.rg_reset_stats(h) == 0
    new = host.log()[at:]
    write = "memset s0" if call in ("sync", "reset") else "copy s0"
    last = max(k for k, line in enumerate(new) if line == write)
    assert "streamsync s0" in new[last:]


def test_server_lanes_are_set_up_on_their_own_streams(host):
    """A lane's stream waits for no other, so its first step finds the lane's
    status, ring and header only if they were written there."""
    srv = ctypes.c_void_p()
    at = len(host.log())
    assert host.L.rg_server_create(ctypes.byref(srv), ctypes.byref(rg.rg_server_desc())) == 0
    new = host.log()[at:]
    assert host.L.rg_server_destroy(srv) == 0
    lanes = {line.split()[1] for line in new if line.startswith("stream ")}
    writes = [line.split()[1] for line in new if line.startswith(("memset ", "copy "))]
    assert lanes and len(writes) >= 3 * len(lanes) and set(writes) == lanes


@pytest.mark.parametrize("flags", [rg.RG_BLAS_SAH, rg.RG_BLAS_SAH | rg.RG_MORTON63])
def test_sah_builds_on_a_second_device(host, flags):
    """The large shared memory of the SAH blocks is allowed per device."""
    for dev in (0, 1, 0):
        host.L.cudaSetDevice(dev)
        h = host.scene()
        for nt in (64, 2000):  # a block per segment; the levels above it in one block
            assert host.blas(h, nt, flags) == 0, host.L.rg_last_error()
    assert any("k_sah_rest" in line for line in host.log())


@pytest.mark.parametrize("flags", [rg.RG_MORTON30, rg.RG_BLAS_SAH])
def test_blas_build_is_refused_on_a_capturing_stream(host, flags):
    """A captured build would leave the descriptor to the graph's first launch,
    while the scene takes the BLAS as built; nothing is put into the graph."""
    h, s = host.scene(), host.stream()
    assert host.blas(h, stream=s) == 0
    host.L.fake_set_capturing(s, 1)
    at = len(host.log())
    assert host.blas(h, flags=flags, stream=s) == rg.RG_ERR_CUDA
    assert host.log()[at:] == []
    host.L.fake_set_capturing(s, 0)
    assert host.blas(h, flags=flags, stream=s) == 0


def test_failed_frame_leaves_nothing_behind_the_callers_stream(host):
    """When a launch of one band fails, the caller's stream still waits for
    every band that has work queued."""
    h, s = host.renderable(), host.stream()
    own = f"s{s.value // 16}"
    r, log = host.render(h, s)
    assert r == 0 and len(set(launches(log))) == 4
    host.L.fake_finish()
    for k in range(1, len(launches(log)) + 1):
        host.L.fake_fail_launch(k)
        r, part = host.render(h, s)
        host.L.fake_fail_launch(0)
        host.L.fake_finish()
        assert r == rg.RG_ERR_CUDA
        for band in set(launches(part)) - {own}:
            last = max(i for i, line in enumerate(part) if line.startswith("launch ") and line.split()[2] == band)
            rec = next(i for i, line in enumerate(part) if i > last and line.startswith("record ") and line.endswith(band))
            assert f"wait {own} {part[rec].split()[1]}" in part[rec:]


def test_bands_run_at_the_priority_of_the_callers_stream(host):
    h = host.renderable()
    prio = {f"s{st.value // 16}": p for p, st in ((p, host.stream(p)) for p in (-3, 0, -3, 2))}
    log = []
    for name in prio:
        r, part = host.render(h, ctypes.c_void_p(int(name[1:]) * 16))
        host.L.fake_finish()
        assert r == 0
        log += part
        made = {f[1]: int(f[5]) for f in (line.split() for line in log if line.startswith("stream "))}
        assert {made[b] for b in set(launches(part)) - {name}} == {prio[name]}


def streams_used(log):
    return len(set(launches(log)))


def test_bands_give_way_to_other_frames_in_flight(host):
    """A frame is banded unless two or more frames of other scenes, sharing
    their BLAS or not, are still running on its device; a scene's own earlier
    frame, a finished one and one of a destroyed scene do not count."""
    a, b, c = host.renderable(), host.renderable(), host.renderable()
    shared = ctypes.c_void_p()
    assert host.L.rg_scene_create_shared(ctypes.byref(shared), a) == 0
    host.scenes.append(shared)
    inst = np.zeros((1, 16), np.float32)
    assert host.L.rg_tlas_build(shared, inst.ctypes.data_as(ctypes.c_void_p), 1, None) == 0
    host.L.fake_finish()
    st = {id(h): host.stream() for h in (a, b, c, shared)}
    used = lambda h: streams_used(host.render(h, st[id(h)])[1])
    assert [used(shared), used(shared), used(a)] == [4, 4, 4]   # its own frames, then one other
    assert [used(b), used(c)] == [1, 1]                          # two and three others
    host.L.fake_finish()
    assert [used(c), used(b)] == [4, 4]
    assert used(a) == 1
    host.destroy(b)
    assert used(a) == 4                                          # c's alone
    assert not [line for line in host.log() if "capture mode" in line]  # (a query would end another thread's capture)
    host.L.fake_finish()


def test_frames_on_a_capturing_stream_are_one_pipeline(host):
    """No streams of the scene's own join a caller's capture, and no event
    recorded in one is asked for later."""
    h, s = host.renderable(), host.stream()
    assert host.render(h, s)[0] == 0   # (sizes the queues)
    host.L.fake_finish()
    host.L.fake_set_capturing(s, 1)
    r, log = host.render(h, s)
    host.L.fake_set_capturing(s, 0)
    assert r == 0 and streams_used(log) == 1
    assert not [line for line in log if line.startswith(("record ", "wait "))]


@pytest.mark.parametrize("w,h", [(3, 1048560), (3, 1048561), (1, 1 << 24), (33, 2097121), (1 << 24, 1)])
def test_fxaa_of_long_images_fits_the_grid(host, w, h):
    """Every size that rg_fxaa's argument check takes is launched."""
    assert host.L.rg_fxaa(ctypes.c_void_p(1 << 20), w, h, ctypes.c_void_p(1 << 40), None) == 0
    assert len(launches(host.log())) == 1


def test_every_query_kernel_is_one_whose_counter_is_cleared(host):
    """Queries clear their work counter where they launch the per-lane kernels;
    no whole-warp instantiation of a query mode exists that could be reached
    with a stale one."""
    names = host.L.fake_kernels().decode().split()
    query = [n for n in names if any(f"k_trace{k}ILi{m}E" in n for k in ("_lane", "_warp", "8_lane", "8") for m in (0, 1))]
    assert query and all("_lane" in n for n in query), query


def test_last_scene_of_a_device_gives_the_temporaries_back(host):
    """What the pool of temporaries keeps goes back, down to 16 MiB, when the last
    scene of its device is destroyed, not before, and not another device's."""
    scenes = {}
    for dev in (0, 0, 1):
        host.L.cudaSetDevice(dev)
        h = host.scene()
        assert host.blas(h) == 0
        scenes.setdefault(dev, []).append(h)
    trims = lambda: [line for line in host.log() if line.startswith("trim ")]
    host.destroy(scenes[0].pop())
    assert trims() == []
    host.destroy(scenes[0].pop())
    assert trims() == ["trim d0 16777216"]
    host.destroy(scenes[1].pop())
    assert trims() == ["trim d0 16777216", "trim d1 16777216"]


def test_allocations_take_the_kept_temporaries_before_they_fail(host):
    h = host.scene()
    assert host.blas(h) == 0
    for k in range(1, 4):   # of a server: of a scene and of its queues the same function
        host.L.fake_fail_malloc(k)
        at = len(host.log())
        srv = ctypes.c_void_p()
        assert host.L.rg_server_create(ctypes.byref(srv), ctypes.byref(rg.rg_server_desc())) == 0
        assert "trim d0 0" in host.log()[at:]
        assert host.L.rg_server_destroy(srv) == 0
    host.L.fake_fail_malloc(1)
    host.scene()
    host.L.fake_fail_malloc(0)


def test_frames_queued_on_one_stream_are_not_in_flight_together(host):
    """Frames of several scenes on one stream run one after another: each is
    banded, and together they count as one frame for the other streams."""
    scenes, s, t = [host.renderable() for _ in range(4)], host.stream(), host.stream()
    host.L.fake_finish()
    assert [streams_used(host.render(h, s)[1]) for h in scenes[:3]] == [4, 4, 4]
    assert streams_used(host.render(scenes[3], t)[1]) == 4     # one other stream
    assert streams_used(host.render(scenes[0], s)[1]) == 4
    host.L.fake_finish()
