"""CPU tests of the C ABI: the library loads, exports every symbol the header
declares, the host planner matches the oracle bit for bit, and host-checkable
argument errors are reported before anything touches a GPU."""
import ctypes
import os
import re

import numpy as np
import pytest

import oracle
import workloads as wl

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HEADER = os.path.join(ROOT, "include", "rf.h")


@pytest.fixture(scope="module")
def rf():
    import paper_2606_06309_gb300 as rf
    if not os.path.exists(rf.lib_path()):
        from paper_2606_06309_gb300 import build
        build.build()
    rf.load()
    return rf


def _declared():
    src = open(HEADER).read()
    src = re.sub(r"/\*.*?\*/", "", src, flags=re.S)
    return sorted(set(re.findall(r"\b(rf_[a-z_0-9]+)\s*\(", src)))


def test_exports_every_declared_symbol(rf):
    names = _declared()
    assert set(names) == set(rf.EXPORTS), names
    lib = ctypes.CDLL(rf.lib_path())
    for n in names:
        assert hasattr(lib, n), n


def test_status_strings(rf):
    assert rf.rf_status_str(0) == "RF_OK"
    assert rf.rf_status_str(5) == "RF_ERR_DEVICE_TIMEOUT"
    assert rf.rf_status_str(99) == "RF_ERR_UNKNOWN"
    assert rf.rf_version() >= 100


@pytest.mark.parametrize("name", list(wl.WORKLOADS))
def test_planner_matches_oracle(rf, name):
    w = wl.get(name)
    got = rf.rf_plan_build(w.F, w.S, w.is_key, w.stride, w.T_w)
    want = oracle.schedule(w.F, w.S, w.is_key, w.stride, w.T_w)
    np.testing.assert_array_equal(got["mask"], want["mask"])
    np.testing.assert_array_equal(got["cur_slot"], want["cur_slot"])
    for k in ("alpha", "beta", "dt"):
        np.testing.assert_array_equal(got[k], want[k].astype(np.float32), err_msg=k)


@pytest.mark.parametrize("T_w", [0, 3, 8])
def test_planner_warmup_and_sigma(rf, T_w):
    F, S = 7, 12
    is_key = [1, 0, 0, 1, 0, 0, 1]
    stride = wl.progressive_stride(S, 3)
    sig = np.array([(1 - s / S) ** 1.5 for s in range(S + 1)])  # non-uniform schedule
    got = rf.rf_plan_build(F, S, is_key, stride, T_w, sig)
    want = oracle.schedule(F, S, is_key, stride, T_w, sigma=sig)
    np.testing.assert_array_equal(got["mask"], want["mask"])
    for k in ("alpha", "beta", "dt"):
        np.testing.assert_array_equal(got[k], want[k].astype(np.float32), err_msg=k)


def test_planner_rejects_bad_args(rf):
    with pytest.raises(rf.RFError):
        rf.rf_plan_build(3, 4, [1, 0, 0], [2, 0, 2, 2], 0)       # stride < 1
    with pytest.raises(rf.RFError):
        rf.rf_plan_build(3, 4, [1, 0, 0], [2] * 4, 5)            # T_w > S
    with pytest.raises(rf.RFError):
        rf.rf_plan_build(3, 2, [1, 0, 0], [2] * 2, 0, [1.0, 0.5, 0.1])  # sigma_S != 0


def test_device_calls_reject_bad_args_on_host(rf):
    """Checks that happen before any CUDA call: null pointers, sizes, head dim."""
    lib = rf.load()
    P = 256  # any non-null, 16-byte aligned value; never dereferenced
    assert lib.rf_schedule_compact(None, 4, 8, P, P, P, P, None) == 1
    assert lib.rf_schedule_compact(P, 0, 8, P, P, P, P, None) == 1
    assert lib.rf_project(P, P, P, P, P, 4, 6, None) == 3            # E % 4 != 0
    assert lib.rf_step(P, P, None, P, P, P, 4, 8, None) == 1
    assert lib.rf_project(P, P, P, P, P, 4, 0, None) == 0            # E = 0: nothing to do
    assert lib.rf_step(P, P, P, P, P, P, 4, 0, None) == 0
    args = [P, None, P, P, P, 256, 256, 4, 64, 2, 96, P, P, 0.1, None, 0, None, None]
    assert lib.rf_attn(*args) == 2                                   # d = 96 unsupported
    args[10] = 128
    args[13] = -1.0
    assert lib.rf_attn(*args) == 1                                   # scale <= 0
    args[13] = 0.1
    args[5] = 100
    assert lib.rf_attn(*args) == 1                                   # row stride < H*d
    args[5] = 260
    assert lib.rf_attn(*args) == 3                                   # row stride % 8 != 0
    args[5] = 256
    args[2] = P + 2
    assert lib.rf_attn(*args) == 3                                   # misaligned Q
    args[2] = P
    args[14], args[15] = P + 16, 1 << 30
    assert lib.rf_attn(*args) == 3                                   # workspace not 256-aligned
    args[14], args[15] = P, -1
    assert lib.rf_attn(*args) == 1                                   # negative workspace size
    assert lib.rf_attn_workspace_bytes(96) == -1
    margs = [P, None, P, P, P, 256, 256, 4, 64, 2, 128, P, P, 0.1, None, None, 0, None, None]
    assert lib.rf_attn_block_masked(*margs) == 1                      # null block mask
    margs[14] = P
    margs[7], margs[8] = 4097, 128
    assert lib.rf_attn_block_masked(*margs) == 2                      # 4097 key blocks


def test_noalloc_rejects_bad_args_before_any_device_work(rf):
    """rf_attn_noalloc returns rf_attn's argument errors before it looks up its scratch array
    or enqueues the counter reset: no CUDA call happens, so this runs without a GPU."""
    lib = rf.load()
    P = 256
    base = [P, None, P, P, P, 256, 256, 4, 64, 2, 128, P, P, 0.1, None, None]
    cases = ((0, None, 1),      # null output
             (11, None, 1),     # null active list
             (10, 96, 2),       # head dim 96
             (13, 0.0, 1),      # softmax scale 0
             (5, 100, 1),       # row stride < H*d
             (6, 260, 3),       # output row stride % 8 != 0
             (7, 0, 1))         # no frames
    for i, v, want in cases:
        args = list(base)
        args[i] = v
        assert lib.rf_attn_noalloc(*args) == want, (i, v)


def test_pipeline_rejects_bad_args_on_host(rf):
    """The host-fed pipeline's argument checks run before any allocation or CUDA call."""
    lib = rf.load()
    P = 256
    out = ctypes.c_void_p(12345)
    pa = [4, 8, 2, 128, 64, 3, P, P, P, P, P, P, P, P, 3, None, None, None, ctypes.byref(out)]
    bad = list(pa)
    bad[18] = None
    assert lib.rf_pipeline_create(*bad) == 1                          # no handle to write
    bad = list(pa)
    bad[6] = None
    assert lib.rf_pipeline_create(*bad) == 1 and out.value is None    # null plan; handle cleared
    for i in (12, 13):
        bad = list(pa)
        bad[i] = None
        assert lib.rf_pipeline_create(*bad) == 1                      # no initial keys/values
    bad = list(pa)
    bad[3] = 96
    assert lib.rf_pipeline_create(*bad) == 2                          # d = 96 unsupported
    bad = list(pa)
    bad[4] = 66
    assert lib.rf_pipeline_create(*bad) == 3                          # E % 4 != 0
    for depth in (1, 9):
        bad = list(pa)
        bad[14] = depth
        assert lib.rf_pipeline_create(*bad) == 1                      # depth outside 2..8
    assert lib.rf_pipeline_step(None, 0, P, P, P, P, P, P, None, 0.1) == 1
    assert lib.rf_pipeline_sync(None, None) == 1
    assert lib.rf_pipeline_bytes(None, None, None, None) == 1
    lib.rf_pipeline_destroy(None)                                     # a no-op


def test_python_binding_raises_with_status(rf):
    """The binding turns a non-zero status into RFError carrying it, with the status name and
    the library's last-error text in the message (host-side checks; no GPU is touched)."""
    plan = rf.rf_plan_build(3, 4, [1, 0, 1], [2] * 4, 0)
    z2 = np.zeros((2, 3, 16), np.float32)
    kv = np.zeros((24, 2, 64), np.uint16)                               # bf16 bits
    with pytest.raises(rf.RFError) as e:
        rf.rf_pipeline_create(3, 8, 2, 96, 16, plan, z2, kv, kv, 3, 0, 0, 0)   # head dim 96
    assert e.value.status == 2 and "rf_pipeline_create" in str(e.value)
    with pytest.raises(rf.RFError) as e:
        rf.rf_pipeline_create(3, 8, 2, 64, 18, plan, z2, kv, kv, 3, 0, 0, 0)   # E % 4 != 0
    assert e.value.status == 3
    with pytest.raises(rf.RFError) as e:
        rf.rf_pipeline_create(3, 8, 2, 64, 16, plan, z2, kv, kv, 1, 0, 0, 0)   # depth 1
    assert e.value.status == 1
    assert rf.rf_status_str(2) and rf.rf_status_str(99)


def test_header_is_a_c_abi(rf, tmp_path):
    """include/rf.h compiles as C (gcc -std=c11, warnings as errors) and a C program linked
    against librf.so builds a plan and reads statuses through it; no GPU is used."""
    import shutil
    import subprocess
    gcc = shutil.which("gcc")
    if gcc is None:
        pytest.skip("no C compiler")
    exe = tmp_path / "plan_smoke"
    lib_dir = os.path.dirname(rf.lib_path())
    cmd = [gcc, "-std=c11", "-Wall", "-Wextra", "-Werror", "-I", os.path.join(ROOT, "include"),
           os.path.join(ROOT, "tests", "c_abi", "plan_smoke.c"), "-L", lib_dir, "-lrf",
           f"-Wl,-rpath,{lib_dir}", "-o", str(exe)]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.startswith("ok"), (r.returncode, r.stdout, r.stderr)


def test_attention_schedules(tmp_path):
    """The schedule arithmetic of the attention kernel over 14,000 random launches on grids of 1 to
    1024 CTAs (tests/c_abi/sched_check.cpp says what is checked)."""
    import shutil
    import subprocess
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no C++ compiler")
    exe = tmp_path / "sched_check"
    cmd = [gxx, "-O2", "-std=c++17", "-Wall", "-Wextra", "-Werror", "-I",
           os.path.join(ROOT, "paper_2606_06309_gb300", "csrc"),
           os.path.join(ROOT, "tests", "c_abi", "sched_check.cpp"), "-o", str(exe)]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.startswith("ok"), (r.returncode, r.stdout, r.stderr)


def _scene_proxies(F=21, E=960, starts=(0, 4, 9, 13, 17), noise=0.3, seed=0):
    rng = np.random.default_rng(seed)
    base = rng.standard_normal((len(starts), E))
    scene = np.searchsorted(np.array(starts), np.arange(F), side="right") - 1
    return base[scene] + noise * rng.standard_normal((F, E))


@pytest.mark.parametrize("seed", range(8))
def test_keyframe_select_host_matches_oracle(rf, seed):
    """Algorithm 1 on the host over inner products equals the oracle working on the
    proxies directly, over random thresholds, budgets and tolerances."""
    rng = np.random.default_rng(100 + seed)
    P = _scene_proxies(seed=seed, noise=float(rng.uniform(0.1, 1.5)))
    G = P @ P.T
    for _ in range(20):
        M = int(rng.integers(1, 22))
        tau, dtau = float(rng.uniform(-0.2, 1.0)), float(rng.uniform(-0.3, 0.3))
        up, down = float(rng.uniform(0, 4)), float(rng.uniform(0, 4))
        got = rf.rf_keyframe_select(G, M, tau, dtau, up, down)
        keys, _ = oracle.keyframe_select(P, M, tau, dtau, up, down)
        assert np.flatnonzero(got).tolist() == keys, (M, tau, dtau, up, down)


def test_keyframe_select_scene_starts(rf):
    P = _scene_proxies()
    got = rf.rf_keyframe_select(P @ P.T, 8, 0.5, 0.0, 1.0, 1.0)
    assert np.flatnonzero(got).tolist() == [0, 4, 9, 13, 17]
    with pytest.raises(rf.RFError):
        rf.rf_keyframe_select(np.zeros((3, 3)), 2, 0.5, 0.0, 1, 1)   # zero-norm frames


def test_bench_traffic_figures_belong_to_the_current_kernel():
    """bench.py reports roofline.traffic only while rf_attn.cu (without comments) hashes to the
    key its ncu capture was taken with; the committed figures are those of the current kernel."""
    import os
    import sys
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    sys.path.insert(0, root)
    import bench
    sha = bench._code_sha(os.path.join(root, "paper_2606_06309_gb300", "csrc", "rf_attn.cu"))
    for name, entry in bench.ATTN_TRAFFIC.items():
        assert entry["code_sha256_rf_attn_cu"] == sha, name
        assert entry["bytes_per_launch"] > 0


def test_plan_row_addresses():
    """stepcore._row is t[s].data_ptr() without the view: every step, negative steps, strided
    plans, and the same error past the ends."""
    import torch

    from paper_2606_06309_gb300.stepcore import _row
    for t in (torch.zeros(7, 5, dtype=torch.uint8), torch.zeros(7, 5),
              torch.zeros(9, 12)[1:8, 3:8], torch.zeros(14, 5)[::2]):
        for s in range(-7, 7):
            assert _row(t, s) == t[s].data_ptr(), s
        assert _row(t, np.int64(3)) == t[3].data_ptr()
        for s in (7, -8):
            with pytest.raises(IndexError):
                _row(t, s)


def _host_step_core(cls, **kw):
    """A step core of host tensors, for tests that replace every call of the library."""
    from paper_2606_06309_gb300.stepcore import upload_plan
    plan = upload_plan(3, 2, [1, 0, 1], [1, 1], 0, "cpu")
    return cls(3, 4, 8, 1, 64, plan, "cpu", split_kv=False, **kw)


@pytest.mark.parametrize("part", ["compact", "project", "project_kv", "attn", "step"])
@pytest.mark.parametrize("how", ["subclass", "object", "class"])
def test_run_calls_replaced_parts(rf, monkeypatch, part, how):
    """StepCore.run takes the fused call only where all five parts are its own: a part replaced in a
    subclass, on the object or on the class itself is called, with run's own arguments."""
    import torch

    from paper_2606_06309_gb300 import stepcore
    calls = []
    for name in ("rf_schedule_compact", "rf_project", "rf_project_kv", "rf_attn", "rf_step",
                 "rf_step_core"):
        monkeypatch.setattr(stepcore, name, lambda *a, name=name, **k: calls.append(name))
    inner = getattr(stepcore.StepCore, part)

    def outer(self, *a, **k):
        calls.append((part, a[-1]))
        return inner(self, *a, **k)

    cls = stepcore.StepCore
    if how == "subclass":
        cls = type("Sub", (cls,), {part: outer})
    elif how == "class":
        monkeypatch.setattr(cls, part, outer)
    core = _host_step_core(cls)
    if how == "object":
        setattr(core, part, outer.__get__(core))
    x = torch.zeros(12, 1, 64, dtype=torch.bfloat16)

    class Stream:
        cuda_stream = 0

    stream = Stream()
    core.run(0, torch.zeros(3, 8), x, x, x, x, 0.1, stream=stream)
    want = ["rf_schedule_compact", "rf_project", "rf_project_kv", "rf_attn", "rf_step"]
    at = ["compact", "project", "project_kv", "attn", "step"].index(part)
    want.insert(at, (part, stream))
    assert calls == want
    assert core.launches_per_step == 5


def test_run_of_the_class_itself_is_one_call(rf, monkeypatch):
    import torch

    from paper_2606_06309_gb300 import stepcore
    calls = []
    monkeypatch.setattr(stepcore, "rf_step_core", lambda *a: calls.append(a))
    x = torch.zeros(12, 1, 64, dtype=torch.bfloat16)
    for cls in (stepcore.StepCore, type("Sub", (stepcore.StepCore,), {"more": lambda self: 1})):
        core = _host_step_core(cls)
        core.run(1, torch.zeros(3, 8), x, x, x, x, 0.1, stream=7)
        assert core.launches_per_step == 2
    assert len(calls) == 2 and all(a[-1] == 7 for a in calls)


@pytest.mark.parametrize("status", [1, 2, 3, 4])
def test_run_repeats_a_refused_step_only(rf, monkeypatch, status):
    """An argument that the fused call refuses is left to the call at fault; a failed CUDA call, after
    which some of the step may have been enqueued, is raised with nothing repeated."""
    import torch

    from paper_2606_06309_gb300 import stepcore
    calls = []
    for name in ("rf_schedule_compact", "rf_project", "rf_project_kv", "rf_attn", "rf_step"):
        monkeypatch.setattr(stepcore, name, lambda *a, name=name: calls.append(name))

    def fused(*a):
        raise rf.RFError("rf_step_core", status)

    monkeypatch.setattr(stepcore, "rf_step_core", fused)
    core = _host_step_core(stepcore.StepCore)
    x = torch.zeros(12, 1, 64, dtype=torch.bfloat16)
    if status == 4:
        with pytest.raises(rf.RFError, match="rf_step_core failed"):
            core.run(0, torch.zeros(3, 8), x, x, x, x, 0.1, stream=0)
        assert calls == []
    else:
        core.run(0, torch.zeros(3, 8), x, x, x, x, 0.1, stream=0)
        assert calls == ["rf_schedule_compact", "rf_project", "rf_project_kv", "rf_attn", "rf_step"]
