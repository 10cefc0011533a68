"""The C-ABI library loads without a GPU and exports every symbol that include/kda.h declares;
argument errors that are detected before any CUDA call are reported with the right status."""
import ctypes
import os
import re

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def lib():
    from paper_2510_26692_b200 import build, api
    build.build()
    return api.load()


def declared_functions():
    text = open(os.path.join(ROOT, "include", "kda.h")).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    names = re.findall(r"\b(kda_[a-z0-9_]+)\s*\(", text)
    return sorted(set(names))


def test_header_symbols_exported(lib):
    names = declared_functions()
    assert "kda_chunk_fwd" in names and "kda_decode_step" in names and len(names) >= 10
    for n in names:
        assert hasattr(lib, n), "symbol %s declared in kda.h is not exported" % n


def test_unsupported_and_invalid_arguments(lib):
    import paper_2510_26692_b200 as K
    one = ctypes.c_void_p(256)
    # unsupported head size / chunk / dtype: rejected before any launch, no fallback
    rc = lib.kda_chunk_fwd(one, one, one, one, one, None, one, one, None, None, 1, 64, 2, 64, 64,
                           64, 1.0, K.KDA_BF16, one, 1 << 30, None)
    assert rc == 2 and "supported" in K.kda_last_error()
    rc = lib.kda_chunk_fwd(one, one, one, one, one, None, one, one, None, None, 1, 64, 2, 128, 128,
                           32, 1.0, K.KDA_BF16, one, 1 << 30, None)
    assert rc == 2
    rc = lib.kda_decode_step(one, one, one, one, one, one, None, one, 4, 2, 128, 64, 1.0,
                             K.KDA_BF16, None)
    assert rc == 2
    # misaligned pointer
    rc = lib.kda_chunk_fwd(ctypes.c_void_p(260), one, one, one, one, None, one, one, None, None, 1,
                           64, 2, 128, 128, 64, 1.0, K.KDA_BF16, one, 1 << 30, None)
    assert rc == 1 and "aligned" in K.kda_last_error()
    # cu_seqlens given on one side only
    rc = lib.kda_chunk_fwd(one, one, one, one, one, None, one, one, one, None, 1, 64, 2, 128, 128,
                           64, 1.0, K.KDA_BF16, one, 1 << 30, None)
    assert rc == 1
    # non-monotone / wrong-ended cu_seqlens (host copy is validated before any launch)
    bad = (ctypes.c_int32 * 3)(0, 80, 64)
    rc = lib.kda_chunk_fwd(one, one, one, one, one, None, one, one, one,
                           ctypes.cast(bad, ctypes.c_void_p), 2, 64, 2, 128, 128, 64, 1.0,
                           K.KDA_BF16, one, 1 << 30, None)
    assert rc == 1 and "decreases" in K.kda_last_error()
    bad2 = (ctypes.c_int32 * 3)(0, 10, 60)
    rc = lib.kda_chunk_fwd(one, one, one, one, one, None, one, one, one,
                           ctypes.cast(bad2, ctypes.c_void_p), 2, 64, 2, 128, 128, 64, 1.0,
                           K.KDA_BF16, one, 1 << 30, None)
    assert rc == 1
    # workspace too small / missing
    rc = lib.kda_chunk_fwd(one, one, one, one, one, None, one, one, None, None, 1, 64, 2, 128, 128,
                           64, 1.0, K.KDA_BF16, one, 1024, None)
    assert rc == 3 and "workspace" in K.kda_last_error()
    rc = lib.kda_chunk_fwd(one, one, one, one, one, None, one, one, None, None, 1, 64, 2, 128, 128,
                           64, 1.0, K.KDA_BF16, None, 0, None)
    assert rc == 3
    # q missing although o is requested
    rc = lib.kda_chunk_fwd(None, one, one, one, one, None, one, one, None, None, 1, 64, 2, 128, 128,
                           64, 1.0, K.KDA_BF16, one, 1 << 30, None)
    assert rc == 1


def test_workspace_queries(lib):
    import paper_2510_26692_b200 as K
    lo = K.kda_chunk_fwd_min_workspace_bytes(4096, 1, 32)
    hi = K.kda_chunk_fwd_workspace_bytes(4096, 1, 32)
    assert 0 < lo <= hi
    assert K.kda_chunk_fwd_workspace_bytes(1 << 20, 1, 32) <= (8 << 30)
    assert K.kda_chunk_fwd_workspace_bytes(4096, 1, 32, dk=64) == 0
    assert K.kda_chunk_fwd_host_workspace_bytes(4096, 1, 32) > hi
    assert K.kda_decode_step_host_workspace_bytes(256, 32) > 0


def test_missing_library_fails_loudly(monkeypatch):
    from paper_2510_26692_b200 import api
    monkeypatch.setattr(api, "_lib", None)
    monkeypatch.setattr(api, "_LIB_PATH", "/nonexistent/libkda_b200.so")
    with pytest.raises(ImportError):
        api.kda_version()


def test_per_device_table(lib):
    """What the library caches per device lives in one slot per device ordinal behind a mutex; the
    self-test exercises the table without any CUDA call.  Also from several threads at once."""
    import threading
    lib.kda_selftest_device_table.restype = ctypes.c_int
    assert lib.kda_selftest_device_table() == 0
    out = []
    ts = [threading.Thread(target=lambda: out.append(lib.kda_selftest_device_table())) for _ in range(8)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    # (the lock probe may find the mutex taken by a sibling thread: code 5 is not a table fault)
    assert all(c in (0, 5) for c in out) and 0 in out


def test_chunk_path_switch(lib):
    import paper_2510_26692_b200 as K
    for mode in (2, 1, 0):
        K.kda_set_chunk_path(mode)
    assert lib.kda_set_chunk_path(3) == 1 and lib.kda_set_chunk_path(-1) == 1


def _plan(lib, chunks, H, avail, n_sm):
    arr = (ctypes.c_int32 * len(chunks))(*chunks)
    out = (ctypes.c_int64 * 4)()
    lib.kda_selftest_fused_plan.restype = ctypes.c_int
    lib.kda_selftest_fused_plan.argtypes = [ctypes.c_void_p, ctypes.c_int, ctypes.c_int,
                                            ctypes.c_int64, ctypes.c_int, ctypes.c_void_p]
    rc = lib.kda_selftest_fused_plan(ctypes.cast(arr, ctypes.c_void_p), len(chunks), H, avail, n_sm,
                                     ctypes.cast(out, ctypes.c_void_p))
    assert rc == 0
    return tuple(out)


def test_fused_schedule_plan(lib):
    """Host side of the fused prefill kernel: clusters, engines and ring depth of a call within the constraints that the
    kernel relies on, and every (sequence, head) pair dealt out exactly once."""
    import random
    rng = random.Random(7)
    lib.kda_selftest_fused_job.restype = ctypes.c_int64
    cases = [([64], 32, 1024, 148), ([3, 11, 1, 5, 0, 14, 4, 3, 2, 0, 7], 5, 40, 148),
             ([5, 4], 40, 1024, 148), ([1], 1, 2, 148), ([9] * 7, 3, 7, 148), ([2, 2], 2, 1000, 8),
             ([4000, 20], 32, 5, 148), ([1] * 300, 32, 888, 148), ([3], 2, 3, 3)]
    for _ in range(200):
        n = rng.randint(1, 12)
        cases.append(([rng.randint(0, 20) for _ in range(n)], rng.randint(1, 70),
                      rng.randint(2, 1200), rng.choice([3, 4, 16, 132, 148, 160, 400])))
    for chunks, H, avail, n_sm in cases:
        n_clusters, size, n_eng, depth = _plan(lib, chunks, H, avail, n_sm)
        what = (chunks, H, avail, n_sm, n_clusters, size, n_eng, depth)
        J = len(chunks) * H
        assert size in (3, 4) and 1 <= n_clusters <= min(J, n_sm // size), what
        assert 2 <= n_eng <= 2 * (size - 1) and 1 <= depth <= 4, what
        assert n_clusters * n_eng * depth <= avail, what                        # the rings fit the workspace
        assert depth == 4 or n_clusters * n_eng * (depth + 1) > avail, what     # and no room is left unused
        jobs = []
        for c in range(n_clusters):
            r = 0
            while lib.kda_selftest_fused_job(n_clusters, c, r) < J:
                jobs.append(lib.kda_selftest_fused_job(n_clusters, c, r))
                r += 1
            # (a cluster stops at its first round without a job: there is none after it)
            assert lib.kda_selftest_fused_job(n_clusters, c, r + 1) >= J, what
        assert sorted(jobs) == list(range(J)), what
    assert _plan(lib, [4], 2, 64, 2)[0] == 0      # no cluster of three CTAs


def test_side_entry_points_reject_bad_arguments(lib):
    """Layer wrap, backward pass and DPLR comparison: argument errors found before any CUDA call."""
    import paper_2510_26692_b200 as K
    one = ctypes.c_void_p(256)
    f32, sz, i64, i32 = ctypes.c_float, ctypes.c_size_t, ctypes.c_int64, ctypes.c_int
    # kda_dplr_chunk_fwd: head size, misaligned pointer, cu_seqlens on one side only
    rc = lib.kda_dplr_chunk_fwd(one, one, one, one, one, one, None, one, one, None, None, 1, 64, 2, 64, 128, 64,
                                1.0, one, 1 << 30, None)
    assert rc == 2
    rc = lib.kda_dplr_chunk_fwd(one, one, one, ctypes.c_void_p(260), one, one, None, one, one, None, None, 1, 64, 2,
                                128, 128, 64, 1.0, one, 1 << 30, None)
    assert rc == 1 and "aligned" in K.kda_last_error()
    rc = lib.kda_dplr_chunk_fwd(one, one, one, one, one, one, None, one, one, one, None, 1, 64, 2, 128, 128, 64, 1.0,
                                one, 1 << 30, None)
    assert rc == 1
    assert lib.kda_dplr_chunk_fwd_workspace_bytes(4096, 1, 2, 128, 128, 64) >= \
        lib.kda_dplr_chunk_fwd_min_workspace_bytes(4096, 1, 2, 128, 128, 64) > 0
    assert lib.kda_dplr_chunk_fwd_workspace_bytes(4096, 1, 2, 64, 128, 64) == 0
    # kda_chunk_bwd: chunk length, missing gradient output, workspace too small
    args = [one] * 6 + [one, one] + [one] * 5 + [one, None, None]
    rc = lib.kda_chunk_bwd(*args, 1, 64, 2, 128, 128, 32, 1.0, K.KDA_BF16, one, 1 << 30, None)
    assert rc == 2
    bad = list(args)
    bad[9] = None      # dk
    rc = lib.kda_chunk_bwd(*bad, 1, 64, 2, 128, 128, 64, 1.0, K.KDA_BF16, one, 1 << 30, None)
    assert rc == 1 and "NULL" in K.kda_last_error()
    rc = lib.kda_chunk_bwd(*args, 1, 64, 2, 128, 128, 64, 1.0, K.KDA_BF16, one, 4096, None)
    assert rc == 3
    assert lib.kda_chunk_bwd_workspace_bytes(4096, 1, 32, 128, 128, 64) > 4096 * 32 * 128 * 4 * 12
    # kda_layer_fwd: decay-function parameters are required; y needs its gate and weight
    largs = [one] * 6 + [None, one, one]
    rc = lib.kda_layer_fwd(*largs, 1e-6, 1e-5, None, one, one, None, None, 1, 64, 2, 128, 128, 64, 1.0, one,
                           1 << 30, None)
    assert rc == 1 and "A_log" in K.kda_last_error()
    largs = [one] * 5 + [None, one, one, one]
    rc = lib.kda_layer_fwd(*largs, 1e-6, 1e-5, None, one, one, None, None, 1, 64, 2, 128, 128, 64, 1.0, one,
                           1 << 30, None)
    assert rc == 1 and "g_o" in K.kda_last_error()
    assert lib.kda_layer_fwd_workspace_bytes(4096, 1, 32, 128, 128, 64) >= \
        lib.kda_layer_fwd_min_workspace_bytes(4096, 1, 32, 128, 128, 64) > 0


def test_wait_limit_from_environment(lib):
    """KDA_WAIT_LIMIT_MS bounds every device-side wait; read once per process, so checked in children."""
    import subprocess
    import sys
    lib.kda_wait_limit_ns.restype = ctypes.c_uint64
    assert lib.kda_wait_limit_ns() == 1_000_000_000      # (this process: variable not set)
    code = ("import ctypes; from paper_2510_26692_b200 import api; l = api.load(); "
            "l.kda_wait_limit_ns.restype = ctypes.c_uint64; print(l.kda_wait_limit_ns())")
    for val, want in (("250", 250_000_000), ("0", 1_000_000_000), ("junk", 1_000_000_000), ("9999999", 1_000_000_000)):
        env = dict(os.environ, KDA_WAIT_LIMIT_MS=val)
        out = subprocess.run([sys.executable, "-c", code], cwd=ROOT, env=env, capture_output=True, text=True)
        assert out.returncode == 0, out.stderr
        assert int(out.stdout.strip().splitlines()[-1]) == want, (val, out.stdout)


def _calls():
    """The entry points with a native marshalling, and their arguments with None and a host tensor for every pointer."""
    import torch
    import paper_2510_26692_b200 as K
    def of(x, ws):
        return {
            "kda_decode_step": [x] * 8 + [0, 2, 128, 128, 1.0, K.KDA_BF16],
            "kda_decode_multi": [x] * 8 + [0, 1, 2, 128, 128, 1.0, K.KDA_BF16],
            "kda_layer_decode_step": [x] * 9 + [1e-6, 1e-5, x, x, x, 0, 2, 128, 128, 1.0],
            "kda_chunk_fwd": [x] * 10 + [0, 0, 2, 128, 128, 64, 1.0, K.KDA_BF16, ws],
            "kda_layer_fwd": [x] * 9 + [1e-6, 1e-5] + [x] * 5 + [0, 0, 2, 128, 128, 64, 1.0, ws],
            "kda_chunk_bwd": [x] * 16 + [0, 0, 2, 128, 128, 64, 1.0, K.KDA_BF16, ws]}
    return of(None, torch.zeros(1024, dtype=torch.uint8)), of(torch.zeros(4, dtype=torch.bfloat16), None)


def test_binding_raises_and_never_ends_the_process(lib):
    """Without a GPU, with host tensors, and with element types out of range: a Python exception each time (in a child
    process: a C++ exception behind the interpreter's back would end it)."""
    import subprocess
    import sys
    code = ("import sys; sys.path.insert(0, 'tests'); import torch, test_abi, paper_2510_26692_b200 as K\n"
            "none, host = test_abi._calls()\n"
            "at = dict(kda_decode_step=13, kda_decode_multi=14, kda_chunk_fwd=17, kda_chunk_bwd=23)   # element types\n"
            "for n in none:\n"
            "    for args, want in ((none[n], (RuntimeError, AssertionError, ValueError)), (host[n], (ValueError, TypeError, AttributeError))):\n"
            "        for dt in (1, 2 ** 40, 2 ** 70, -2 ** 70):\n"
            "            a = list(args)\n"
            "            if n in at: a[at[n]] = dt\n"
            "            if torch.cuda.is_available() and args is none[n]: continue\n"
            "            try: getattr(K, n)(*a)\n"
            "            except want: continue\n"
            "            raise SystemExit('%s returned' % n)\n"
            "print('done')\n")
    r = subprocess.run([sys.executable, "-c", code], cwd=ROOT, capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.strip().endswith("done"), (r.returncode, r.stdout[-500:], r.stderr[-500:])


def test_binding_host_tensors_are_refused(lib):
    """All six entry points name the first tensor that is not on the GPU."""
    import paper_2510_26692_b200 as K
    import torch
    for n, args in _calls()[1].items():
        a = [torch.zeros(4, dtype=torch.uint8) if x is None else x for x in args]
        with pytest.raises(ValueError, match="live on"):
            getattr(K, n)(*a)


def test_marshalling_of_another_torch_is_refused(lib, monkeypatch, tmp_path):
    """The native marshalling is compiled against torch's C++ headers: after an upgrade of torch it is built anew, and
    not called before that."""
    import torch
    from paper_2510_26692_b200 import api, build
    assert build.marshal_fits()
    monkeypatch.setattr(torch, "__version__", "0.0.1")
    assert not build.marshal_fits()
    monkeypatch.setattr(api, "_lib", None)
    with pytest.raises(ImportError, match="another Python or torch"):
        api.kda_version()
    built = []
    monkeypatch.setattr(build, "_build_marshal", lambda: built.append(1))
    build.build()
    assert built
