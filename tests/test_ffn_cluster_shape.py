"""Split and shared-memory layout of the clustered feed-forward kernel, over its whole range of shapes, on the host: the header is
compiled by itself."""
import ctypes
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
FIELDS = ["M", "K", "Hid", "N2", "CS", "NC", "T", "BH", "RP", "stage_bytes", "slot_bytes", "slots_off", "bars_off", "J", "Tp",
          "kblocks", "stages", "wait_copies", "w2_off"]
SOURCE = """
#include "ffn_cluster_shape.h"
using namespace ago::ffn_cluster;
extern "C" int plan(FfnClusterShape* q) {      // M, K, Hid, N2 given -> bytes of shared memory, 0: no split
  q->kblocks = q->K / kBK;
  q->RP = std::min(kBM, (q->M + 15) / 16 * 16);
  if (!choose_split(q, (q->M + kBM - 1) / kBM, kResident)) return 0;
  return layout(q);
}
extern "C" int loads_of_one_stage() { return kLoadsOfOneStage; }
extern "C" int clusters(int row_blocks, int J, int resident) { return launched_clusters(row_blocks, J, resident); }
"""


class Shape(ctypes.Structure):
    _fields_ = [(n, ctypes.c_int) for n in FIELDS]


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("shape")
    src, so = d / "shape.cpp", d / "shape.so"
    src.write_text(SOURCE)
    subprocess.check_call(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I" + os.path.join(ROOT, "paper_2212_01005_b200", "csrc"),
                           str(src), "-o", str(so)])
    return ctypes.CDLL(str(so))


def shapes(lib):
    rows = [1, 16, 17, 40, 64, 80, 100, 112, 113, 128, 200, 256, 300, 511, 700, 1000, 1500, 2500, 3001, 4500, 12288]
    for m in rows:
        for k in (64, 128, 192, 320, 768, 1024, 2048):
            for hid in (128, 256, 384, 512, 640, 768, 1024, 1536, 1920, 2048, 3072, 4096):
                for n2 in (128, 192, 256, 384, 512, 576, 768, 1024):
                    q = Shape(M=m, K=k, Hid=hid, N2=n2)
                    smem = lib.plan(ctypes.byref(q))
                    if smem:
                        yield q, smem


def test_split_row_blocks_get_one_cluster_per_part(lib):
    # a cluster has room for one part only; fewer clusters than parts may be resident where a process has a share of the device
    for resident in (1, 7, 15, 33, 45, 74):
        for row_blocks in (1, 2, 5, 16, 37):
            for j in (2, 3, 6, 24):
                assert lib.clusters(row_blocks, j, resident) == row_blocks * j
            assert lib.clusters(row_blocks, 1, resident) == min(row_blocks, resident)
    assert any(q.J > 1 for q, _ in shapes(lib))


def test_staged_sums_stay_off_what_is_still_copied(lib):
    # the buffers of the staged sums lie over the ring; where they are larger the kernel waits for the copies out of the slots
    # behind it. They never reach the barriers.
    waits = {}
    for q, _ in shapes(lib):
        staging = min(2, q.NC // 64) * q.RP * 256 if q.J > 1 and q.RP >= 64 else 0
        assert staging <= q.bars_off, list(getattr(q, n) for n in FIELDS)
        past = staging > q.stages * q.stage_bytes
        assert bool(q.wait_copies) == past, list(getattr(q, n) for n in FIELDS)
        waits[(q.M, q.K, q.Hid, q.N2)] = past
    assert waits[(300, 64, 2048, 256)] and waits[(1000, 128, 512, 384)]
    assert not waits[(511, 768, 3072, 768)]


def test_ring_has_the_stages_that_two_producers_need(lib):
    short = 0
    for q, _ in shapes(lib):
        loads = q.kblocks if q.w2_off else q.Tp * (q.kblocks + q.CS * (q.BH // 64))      # of a part or row block
        assert q.stages >= 2 or q.stages == 1 and q.w2_off and loads <= lib.loads_of_one_stage(), list(getattr(q, n) for n in FIELDS)
        short += q.stages < 3
    assert short > 0


def test_layout_and_kernel_agree_on_whole_row_blocks(lib):
    # 128 rows in tiles of 128 hidden units: the kernel takes W2 through the ring, so nothing is set aside for it and the ring has
    # all that the tiles' slots leave
    for q, smem in shapes(lib):
        assert smem <= 227 * 1024
        if q.RP == 128 and q.BH == 128:
            assert q.w2_off == 0 and q.stage_bytes == 32768, list(getattr(q, n) for n in FIELDS)
            assert q.stages == min(16, (227 * 1024 - 1024 - 512 - q.CS * 32768) // 32768)
