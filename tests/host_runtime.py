"""The library's host code on a fake CUDA runtime (fake_cudart.cpp): the objects
of the built library linked with it, loaded beside the real one."""
import ctypes
import os
import shutil
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))


def load(out_dir):
    """The library with the fake runtime, built into out_dir."""
    from paper_1105_5804_gb300 import build
    build.build()
    objs = [os.path.join(build.OUT_DIR, os.path.basename(s)[:-3] + ".o") for s in build.sources()]
    include = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build._nvcc()))), "include")
    so = os.path.join(str(out_dir), "libswccl_fake.so")
    cmd = [shutil.which("g++") or "g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-I", include,
           os.path.join(HERE, "fake_cudart.cpp")] + objs + ["-o", so]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    L = ctypes.CDLL(so)
    vp, i32, u64 = ctypes.c_void_p, ctypes.c_int, ctypes.c_uint64
    for name, args, res in [
            ("sw_last_error", [], ctypes.c_char_p), ("sw_create_threshold", [i32, i32, u64, u64, i32, vp], vp),
            ("sw3_create", [i32, i32, i32, i32, u64, u64, i32, vp], vp),
            ("sw_batch_create_ws", [i32, vp, vp, vp, vp, i32, i32, vp, ctypes.c_int64, vp], vp),
            ("sw_batch_device_bytes", [i32, vp, vp], ctypes.c_int64),
            ("sw_batch_stream", [vp], vp), ("fake_stream", [i32], vp), ("fake_capture", [vp, i32], None),
            ("fake_capture_valid", [vp], i32), ("fake_counts", [vp], None), ("fake_set_device", [i32], None),
            ("sw_sweep", [vp, i32], i32), ("sw3_sweep", [vp, i32], i32), ("sw_batch_sweep", [vp, i32], i32),
            ("sw_sweep_io", [vp, vp, i32, vp, vp], i32), ("sw_set_timing", [vp, i32], i32),
            ("sw3_set_timing", [vp, i32], i32), ("sw_set_mode", [vp, i32], i32),
            ("sw_set_update", [vp, i32, i32, u64], i32), ("sw_batch_set_graph", [vp, i32], i32),
            ("sw_get_info", [vp, vp], i32), ("sw3_get_info", [vp, vp], i32), ("sw_batch_info", [vp, vp], i32),
            ("sw_phase_times", [vp, vp, vp], i32), ("sw_observables", [vp, vp, i32, vp], i32),
            ("sw_destroy", [vp], i32), ("sw3_destroy", [vp], i32), ("sw_batch_destroy", [vp], i32),
            ("cudaStreamSynchronize", [vp], i32), ("cudaGetLastError", [], i32),
            ("ccl_label_noalloc", [vp, vp, i32, i32, i32, vp], i32), ("ccl_label", [vp, vp, i32, i32, i32, vp], i32)]:
        f = getattr(L, name)
        f.argtypes, f.restype = args, res
    return L
