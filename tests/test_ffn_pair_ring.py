"""Ring stages of the paired feed-forward kernel: every producer takes part in every stage, on the host (the header is compiled by
itself). A producer that a stage does not wait for may fall two phases behind the barrier it waits on, whose phases it tells apart by
one bit; the wait then never ends."""
import ctypes
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SOURCE = """
#include "ffn_pair_ring.h"
extern "C" int stages(int kblocks) { return ago::ffn_pair::g1_stages(kblocks); }
extern "C" int bytes(int kb, int kblocks, int leader) { return ago::ffn_pair::g1_stage_bytes(kb, kblocks, leader != 0); }
extern "C" int stage_bytes() { return ago::ffn_pair::kFStageBytes; }
"""


def test_every_stage_waits_for_the_producers_of_both_ctas(tmp_path):
    src, so = tmp_path / "ring.cpp", tmp_path / "ring.so"
    src.write_text(SOURCE)
    subprocess.check_call(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I" + os.path.join(ROOT, "paper_2212_01005_b200", "csrc"),
                           str(src), "-o", str(so)])
    lib = ctypes.CDLL(str(so))
    for kblocks in range(1, 65):
        n = lib.stages(kblocks)
        assert n % 2 == 0 and kblocks <= n <= kblocks + 1
        for kb in range(n):
            lead, mate = lib.bytes(kb, kblocks, 1), lib.bytes(kb, kblocks, 0)
            assert 0 < mate <= lib.stage_bytes(), (kblocks, kb)      # the leading CTA takes part by its arrival
            assert lead == (mate if kb < kblocks else 0), (kblocks, kb)
            assert mate % 16 == 0
