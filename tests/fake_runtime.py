"""libsfft's objects linked against a CUDA runtime that runs on the host alone (fake_cudart.cpp): what the
host code allocates, launches and orders between streams, and what it does when one of those calls fails."""
import ctypes
import glob
import os
import subprocess

from paper_1201_2501_gb300 import build, sfft

HERE = os.path.dirname(os.path.abspath(__file__))
LAUNCH_FN = ctypes.CFUNCTYPE(None, ctypes.c_char_p, ctypes.POINTER(ctypes.c_void_p))


def load(folder):
    build.build()
    so = os.path.join(str(folder), "libsfft_fake.so")
    cuda = os.path.dirname(os.path.dirname(build._nvcc())) or "/usr/local/cuda"
    subprocess.run(["g++", "-std=c++17", "-O1", "-fPIC", "-shared", "-I", os.path.join(cuda, "include"), "-o", so,
                    os.path.join(HERE, "fake_cudart.cpp"), *sorted(glob.glob(os.path.join(build.BUILD, "*.o"))),
                    "-Wl,-z,defs", "-Wl,-Bsymbolic", "-lpthread"], check=True)
    L = ctypes.CDLL(so)
    L.fake_log.restype = ctypes.c_char_p
    L.fake_bytes.restype = ctypes.c_size_t
    L.sfft_last_error.restype = ctypes.c_char_p
    return L


def plan(L, n, k, mode=sfft.SFFT_EXACT, batch=1, **fields):
    """(status, handle) of sfft_plan_create with the defaults and `fields`."""
    p = sfft.SfftParams()
    L.sfft_params_default(ctypes.byref(p), ctypes.c_uint64(n), k, mode)
    for name, v in fields.items():
        setattr(p, name, v)
    h = ctypes.c_void_p()
    return L.sfft_plan_create(ctypes.byref(p), batch, ctypes.byref(h)), h


def log(L):
    return [line.split() for line in L.fake_log().decode().splitlines()]


def unordered(calls, st):
    """The launches of a call's log that work queued on stream `st` afterwards would not wait for."""
    events, behind, launches = {}, {}, []  # per event and stream: the launches it follows
    for what, *args in calls:
        if what == "launch":
            launches.append(args[0])
            behind.setdefault(args[1], set()).add(len(launches) - 1)
        elif what == "record":
            events[args[0]] = set(behind.get(args[1], ()))
        elif what == "wait":
            behind.setdefault(args[0], set()).update(events.get(args[1], ()))
    return [launches[i] for i in range(len(launches)) if i not in behind.get(st, ())]
