"""The packets between the blocks of a resident launch, on the CPU: every way in
which a packet's store and the receiver's load can cross.

A vector access is as many accesses as it has elements, in no stated order; an
element arrives as a whole.  The element width is read from the accesses in
``packets.cuh``.
"""
import itertools
import os
import re

import pytest

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1907_00908_gb300", "csrc",
                   "packets.cuh")


def _words(op):
    """32-bit words of an element of the packet's store (st) or load (ld)."""
    with open(SRC) as f:
        got = re.findall(op + r"\.volatile\.global\.v([24])\.[ub](32|64) ", f.read())
    assert len(got) == 1 and int(got[0][0]) * int(got[0][1]) == 128
    return int(got[0][1]) // 32


def _taken(store, load):
    """Every packet (re, im) that a receiver can take for the new one."""
    new, old = ("re", "stamp", "im", "stamp"), ("old re", "old stamp", "old im", "old stamp")
    n_st, n_ld = 4 // store, 4 // load
    for order in itertools.permutations(range(n_st)):            # place of each element in the order of arrival
        for when in itertools.product(range(n_st + 1), repeat=n_ld):   # arrivals before each element of the load
            got = [new[w] if order[w // store] < when[w // load] else old[w] for w in range(4)]
            if got[1] == "stamp" and got[3] == "stamp":
                yield got[0], got[2]


def test_a_packet_with_both_stamps_holds_both_values():
    taken = set(_taken(_words("st"), _words("ld")))
    assert taken == {("re", "im")}


@pytest.mark.parametrize("store,load", [(1, 1), (1, 2), (2, 1)])
def test_narrower_elements_would_not_do(store, load):
    assert len(set(_taken(store, load))) > 1
