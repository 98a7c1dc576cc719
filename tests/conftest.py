import ctypes
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)


def pytest_configure(config):
    config.addinivalue_line("markers", "gpu: needs a CUDA device (runs on a B200 box)")


@pytest.fixture(scope="session")
def oracle():
    import oracle as _oracle
    _oracle.build()
    return _oracle


@pytest.fixture(scope="session")
def rules(tmp_path_factory):
    """The index arithmetic of csrc/rules.cuh compiled for the host; undefined behaviour ends the process."""
    lib = str(tmp_path_factory.mktemp("rules") / "librules.so")
    subprocess.run(["g++", "-std=c++17", "-O2", "-Wall", "-Werror", "-ffp-contract=off", "-fsanitize=undefined",
                    "-fno-sanitize-recover=undefined", "-fPIC", "-shared",
                    "-I", os.path.join(ROOT, "paper_2507_04123_b200", "csrc"),
                    "-o", lib, os.path.join(ROOT, "tests", "rules_shim.cpp")], check=True)
    so = ctypes.CDLL(lib)
    u32, u64 = ctypes.c_uint32, ctypes.c_uint64
    so.clamp.restype, so.clamp.argtypes = u32, [u32]
    so.fits.restype, so.fits.argtypes = ctypes.c_int, [u64, u32, u32, u32, u32]
    so.ranked.restype, so.ranked.argtypes = u32, [u32, u32]
    so.ticket.restype, so.ticket.argtypes = u64, [u32, u32]
    so.tile_frames.restype, so.tile_frames.argtypes = ctypes.c_int64, [ctypes.c_int64, ctypes.c_int64]
    for f in (so.first_word, so.words_of_frame):
        f.restype, f.argtypes = u32, [u32, u32, u32]
    so.most_words.restype, so.most_words.argtypes = u32, [u32, u32]
    so.four_bits.restype, so.four_bits.argtypes = u32, [u32]
    so.frame_notes.argtypes = [u64, u64, ctypes.c_int, ctypes.c_int]
    so.notes.argtypes = [u64, u64, ctypes.c_int, ctypes.c_int]
    so.frames_log.argtypes = [u64, ctypes.c_int]
    so.frames_in_group.argtypes = [u64, ctypes.c_int]
    so.rows_aside.argtypes = [u64, u64, ctypes.c_int]
    so.rows_stay.argtypes = [u64, u64]
    return so
