"""Builds sweep_host.cpp, the library's host-compilable code, with the host compiler."""
import ctypes
import os
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1903_00227_gb300", "csrc")


def host_library(where) -> ctypes.CDLL:
    so = os.path.join(str(where), "sweep_host.so")
    subprocess.check_call(["g++", "-O1", "-w", "-std=gnu++17", "-DWRS_CHECK=1", "-shared", "-fPIC", "-I", CSRC, "-o", so,
                           os.path.join(HERE, "sweep_host.cpp")])
    return ctypes.CDLL(so)
