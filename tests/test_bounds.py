"""Index rules of the streaming kernels (csrc/rs_bounds.cuh), on the host (no
GPU): the header is compiled with the host compiler and every case is run.
"""
import ctypes
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1701_05913_gb300", "csrc")

SRC = """
#include "rs_bounds.cuh"
extern "C" int wave_chunk_step(int q, int nch, int nslots, int steps) { return rs_wave_chunk_step(q, nch, nslots, steps); }
extern "C" int part_place(int e, int nrow) { return rs_part_place(e, nrow); }
extern "C" int part_lost() { return RS_PART_LOST; }
"""


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    d = tmp_path_factory.mktemp("bounds")
    (d / "b.cpp").write_text(SRC)
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(d / "b.cpp"), "-o", str(d / "b.so")],
                   check=True)
    return ctypes.CDLL(str(d / "b.so"))


@pytest.mark.parametrize("steps", [1, 2, 4, 8, 16])
@pytest.mark.parametrize("nslots", [2, 4])
def test_wave_producer_copies_every_chunk_of_a_unit_once_and_no_other(rules, nslots, steps):
    """The wavefront sweeps' producer: as the consumer's step c advances it
    copies chunks while their step has come.  Units of fewer chunks than slots,
    as many and more."""
    for nch in range(1, 4 * nslots + 1):
        issued = []
        for c in range(nch * steps):
            while c >= rules.wave_chunk_step(len(issued), nch, nslots, steps):
                q = len(issued)
                assert q < nch, (nch, q)
                # the slot's chunk before has been left
                assert q < nslots or c >= (q - nslots + 1) * steps
                issued.append(q)
            # the consumer's own chunk is on its way when it gets there
            assert len(issued) > c // steps, (nch, c)
        assert len(issued) == nch


@pytest.mark.parametrize("nrow", [1, 2, 31, 1000, 65534])
def test_part_sweep_takes_its_rows_and_none_that_is_lost(rules, nrow):
    for e in range(0x10000):
        assert bool(rules.part_place(e, nrow)) == (e < nrow)
        assert not rules.part_place(e | rules.part_lost(), nrow)
