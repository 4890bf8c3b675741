"""Both slot widths of the hash set, at the edges of the code spaces that choose them."""
import numpy as np
import pytest
import torch

from oracle import nezha_oracle as O
from paper_2511_18793_b200 import synth

pytestmark = pytest.mark.gpu


def _key_that_maps_to_all_ones():
    """The 32-bit key whose image under the narrow form's bijection is the free slots' value: the finalizer inverted."""
    m = 0xFFFFFFFF
    m ^= m >> 16
    m = m * pow(0xC2B2AE35, -1, 1 << 32) & 0xFFFFFFFF
    m ^= (m >> 13) ^ (m >> 26)
    m = m * pow(0x85EBCA6B, -1, 1 << 32) & 0xFFFFFFFF
    return m ^ (m >> 16)


def _unpack(key, T):
    out = []
    for t in T:
        out.append(key % t)
        key //= t
    return out


@pytest.mark.parametrize("T,n,load_factor", [((256,) * 4, 40_000, 0.5),      # exactly 2^32 keys: the largest narrow space
                                             ((1024, 1024, 1024, 5), 40_000, 0.5),   # the next size up: wide
                                             ((256,) * 4, 30_000, 0.95), ((1024,) * 4, 30_000, 0.95),   # long walks
                                             ((3, 5, 7), 100, 0.5), ((2,), 1, 0.5)])                     # a few buckets
def test_membership_in_both_slot_widths(T, n, load_factor):
    from gpu_helpers import Case
    rng = np.random.default_rng(n + len(T))
    space = int(np.prod([int(t) for t in T], dtype=object))
    cat = np.stack([rng.integers(0, t, size=n) for t in T], axis=1).astype(np.int32)
    special = _key_that_maps_to_all_ones()
    probes = np.concatenate([cat, np.stack([rng.integers(0, t, size=50_000) for t in T], axis=1).astype(np.int32)])
    for with_special in (False, True):
        if special < space:
            tup = np.asarray([_unpack(special, T)], dtype=np.int32)
            cat = cat[~(cat == tup).all(axis=1)]
            cat = np.concatenate([cat, tup, tup]) if with_special else cat        # (twice: a duplicate of it counts once)
            probes = np.concatenate([probes, tup])
        w = synth.scaled(synth.WORKLOADS["tiny"], L=len(T), T=T, n_items=len(cat), batch=1, beam=2, n_hist=1, load_factor=load_factor)
        case = Case(w, catalog=cat, hist=np.zeros((1, 1, len(T)), dtype=np.int32))
        assert case.n_unique == len({tuple(r) for r in cat.tolist()})
        keys = case.eng.pack(torch.from_numpy(probes).cuda())
        assert np.array_equal(keys.cpu().numpy().view(np.uint64), O.pack_keys(probes, T))
        assert np.array_equal(case.eng.probe(keys).cpu().numpy().astype(bool), O.ValidSet(cat, T).contains(probes))
        # raw keys outside the code space, among them ones that agree with a member in their low 32 bits
        raw = np.concatenate([O.pack_keys(cat[:100], T) + np.uint64(1 << 32) * np.uint64(1 + (space >> 32)),
                              np.asarray([2 ** 64 - 1, 2 ** 64 - 2, space], dtype=np.uint64)])
        assert not case.eng.probe(torch.from_numpy(raw.view(np.int64)).cuda()).any().item()
        case.eng.close()
