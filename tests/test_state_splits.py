"""The state kernel's splits and clusters, from the header that the library decides by, compiled for the host: every split has tokens, the workspace
holds them, clusters only where they all fit at once, and the side of the line that was measured as the faster one.
"""
from __future__ import annotations

import ctypes
import os
import subprocess

import pytest

from paper_2211_10526_b200 import build

SMS = 148
FIT = (0, 296, 148, 93, 71, 56, 45, 37, 33)   # clusters of P CTAs that a B200 holds at once

SOURCE = """
#include "state_splits.cuh"
using namespace castling::tc;
extern "C" int splits(int planes, int tiles, int sms, int narrow, const int* fit, int* clustered) {
    const StateSplits s = state_splits(planes, tiles, sms, narrow != 0, [&](int P) { return fit[P]; });
    *clustered = s.clustered;
    return s.P;
}
extern "C" int most(int planes, int tiles, int sms) { return most_splits(planes, tiles, sms); }
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("splits")
    (d / "splits.cpp").write_text(SOURCE)
    subprocess.run([os.environ.get("CXX", "g++"), "-std=c++17", "-shared", "-fPIC", "-I", build.CSRC, str(d / "splits.cpp"), "-o", str(d / "splits.so")], check=True)
    return ctypes.CDLL(str(d / "splits.so"))


def split(lib, planes, tiles, narrow=False, fit=FIT):
    clustered = ctypes.c_int()
    P = lib.splits(planes, tiles, SMS, int(narrow), (ctypes.c_int * 9)(*fit), ctypes.byref(clustered))
    return P, bool(clustered.value)


def test_splits_are_not_empty_and_fit(lib):
    for planes in [*range(1, 330), 768, 3072]:
        for tiles in [*range(1, 70), 94, 128, 160, 255, 256, 512, 1000]:
            most = lib.most(planes, tiles, SMS)
            for narrow in (False, True):
                P, clustered = split(lib, planes, tiles, narrow)
                per = -(-tiles // P)
                assert 1 <= P <= most and (P - 1) * per < tiles
                assert planes * most <= 2 * SMS or most == 1
                if clustered:
                    assert 2 <= P <= 8 and planes < FIT[P]
                P, clustered = split(lib, planes, tiles, narrow, (0,) * 9)   # a device that does not say
                assert (P, clustered) == (most, False)


# planes, tiles of 128 rows, width 32 or not: the faster of a cluster and memory by more than 1 % (B200, from a graph)
@pytest.mark.parametrize("planes,tiles,narrow,clustered", [
    (1, 5, False, True), (1, 64, False, True), (1, 94, False, False), (1, 160, False, False), (3, 160, False, False), (6, 128, False, False), (9, 160, False, False),
    (16, 8, False, True), (16, 128, False, True), (18, 128, False, True), (24, 64, False, True), (37, 16, False, False), (37, 12, False, True),
    (42, 12, False, True), (42, 32, False, False), (49, 32, False, False), (49, 9, False, True), (64, 12, False, True), (66, 6, False, True),
    (72, 4, False, False), (72, 32, False, False), (74, 18, False, False), (88, 3, False, False), (87, 18, False, False), (84, 12, False, True), (92, 9, False, False), (96, 12, False, False), (98, 3, False, False),
    (100, 6, False, True), (128, 6, False, True),
    (9, 64, True, False), (16, 64, True, False), (16, 32, True, True), (16, 4, True, True), (49, 15, True, True), (64, 15, True, False), (64, 16, True, False),
    (74, 4, True, False), (92, 12, True, False), (98, 64, True, False), (37, 32, True, False), (37, 12, True, True)])
def test_the_faster_side(lib, planes, tiles, narrow, clustered):
    assert split(lib, planes, tiles, narrow)[1] == clustered
