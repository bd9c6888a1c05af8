"""Answers kept per device (device_cache.h, no GPU): a second device is asked for itself, and an answer that
could not be had is asked for again."""
import ctypes
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
OUT = os.path.join(ROOT, "tests", "shim", "_build")


def test_answers_are_per_device():
    os.makedirs(OUT, exist_ok=True)
    so = os.path.join(OUT, "libdevice_cache_shim.so")
    src = os.path.join(ROOT, "tests", "shim", "device_cache_shim.cpp")
    subprocess.run(["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-o", so, src], check=True)
    lib = ctypes.CDLL(so)
    asked = ctypes.c_int(0)
    for device, now, answer, count in [(0, 1, 1, 1), (0, 0, 1, 1), (1, 0, 0, 2), (1, 1, 0, 2),
                                       (2, -1, 0, 3), (2, 1, 1, 4), (2, -1, 1, 4), (0, -1, 1, 4)]:
        assert lib.dc_get(device, now, ctypes.byref(asked)) == answer
        assert asked.value == count
