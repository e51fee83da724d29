"""Which phase of a stage's barrier ends when the last chunk issued into it has landed (pipe_phase.h,
compiled for the host), against a model of the ring: chunks issued in order, each into a stage whose
chunk before it has landed, up to one per stage still in flight when the issuing stops.  A wait for a
parity ends when the phase of that parity is the one completed last, which is also so before the
first phase for parity 1; a wait on any other parity than the function's would return at once with a
copy in flight, or never."""
import ctypes
import itertools
import os
import subprocess

import pytest

from paper_2607_05272_gb300 import build as B


@pytest.fixture(scope="module")
def last_parity(tmp_path_factory):
    d = tmp_path_factory.mktemp("pipe")
    src, out = d / "p.cpp", str(d / "p.so")
    src.write_text('#include "%s"\nextern "C" int f(unsigned i, unsigned S, unsigned s) '
                   '{ return simx::last_parity(i, S, s); }\n' % os.path.join(B.CSRC, "pipe_phase.h"))
    subprocess.run(["g++", "-shared", "-fPIC", "-std=c++17", "-o", out, str(src)], check=True)
    return ctypes.CDLL(out).f


def test_the_last_chunk_of_every_stage_is_waited_for(last_parity):
    def ends(completed, parity):
        return completed % 2 != parity   # the phase of this parity is the one before the current

    for S in (1, 2, 3, 5, 8):
        for issued in range(0, 4 * S + 2):
            per = [len(range(st, issued, S)) for st in range(S)]   # chunks issued into each stage
            for late in itertools.product((0, 1), repeat=min(S, 3)):
                for st in range(S):
                    parity = last_parity(issued, S, st)
                    if per[st] == 0:
                        assert parity == -1
                        continue
                    in_flight = st < len(late) and late[st]
                    assert ends(per[st] - in_flight, parity) == (not in_flight)


def test_a_resident_policy_fills_phase_0_only(last_parity):
    """Where the whole policy is issued once (S chunks of S stages), every wait is for parity 0."""
    for S in range(1, 9):
        assert all(last_parity(S, S, st) == 0 for st in range(S))
