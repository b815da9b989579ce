"""The ABI structs of one energy call hold what the general ones of a context hold (host only)."""
import ctypes as C
import dataclasses

import numpy as np
import pytest

from paper_1702_01770_gb300 import inputs, phast

BASE = inputs.System("c", np.array([4, 5], np.int32), np.array([0, 1, 1, 0, 0, 1, 0, 1, 1], np.uint8), 12.5, k_bend=0.3, k_tors=-0.5,
                     k_lj_intra=3.0, k_lj_inter=2.0, C=(1.0, -0.5, 0.25, 0.5), k_fene=-20.0, fene_r0=0.9, fene_R=0.4, C_F=(1.0, 2.0, 3.0, 4.0))


@pytest.mark.parametrize("change", [{}, dict(C=(1.0, -0.5, -0.5)), dict(C_F=()), dict(C=[1, 0, 0, 1], box_L=7, k_bend=1),
                                    dict(C=np.array([1.0, 2.0, 3.0, 4.0], np.float32), box_L=0.0, sphere_R=np.float32(8.0)),
                                    dict(chain_len=[4, 5], seq=[0, 1] * 4 + [1]), dict(chain_len=np.array([9], np.int64), seq=np.ones(18, np.uint8)[::2])],
                         ids=["full", "three", "none", "ints", "numpy", "lists", "strided"])
def test_structs_of_a_call_match_the_general_ones(change):
    s = dataclasses.replace(BASE, **change)
    one, many = phast._CallStructs(s), phast._Structs([s])
    a, b = one.sys, many.sys[0]
    assert a.n_chains == b.n_chains == len(s.chain_len) and (a.box_L, a.sphere_R) == (b.box_L, b.sphere_R)
    assert a.chain_len[:a.n_chains] == b.chain_len[:a.n_chains] == [int(v) for v in s.chain_len]
    n = int(np.sum(s.chain_len))
    assert a.seq[:n] == b.seq[:n] == [int(v) for v in s.seq]
    assert C.string_at(C.addressof(one.ff), C.sizeof(one.ff)) == C.string_at(C.addressof(many.ff[0]), C.sizeof(one.ff))
