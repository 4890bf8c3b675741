"""The catalogue's build by parts of the prefix map's longest region: both code loads, whole and partial last parts, repeated
items, walks over the ends of parts, a rebuild, and a code outside its codebook.
The launch count tells which build ran."""
import numpy as np
import pytest
import torch

from oracle import nezha_oracle as O
from paper_2511_18793_b200 import synth

pytestmark = pytest.mark.gpu


# Load factors low enough that the longest region is the direct one; at 0.95 the hash set's walks run over the ends of its parts.
# (63, 61, 59, 37): 8,389,269 prefixes of one word in 1,025 parts, the last of 661 prefixes.  256^3: the most parts, 8,192.
# (128, 128, 64): the smallest region, 16 MB in 256 parts.  1,572,864: the fewest items.
@pytest.mark.parametrize("T,n,load_factor", [((63, 61, 59, 37, 50), 1_600_000, 0.25), ((63, 61, 59, 37, 50), 4_100_000, 0.95),
                                             ((256,) * 4, 1_600_000, 0.1),
                                             ((256,) * 4, 2_013_000, 0.03),   # 8,192 + 4,096 counters: 48 KB to the byte
                                             ((240, 256, 256, 250), 1_572_864, 0.1),
                                             ((128, 128, 64, 16), 1_572_864, 0.5), ((128, 128, 64, 16), 1_572_863, 0.5)])
def test_build_by_parts(T, n, load_factor):
    from gpu_helpers import Case
    rng = np.random.default_rng(n)
    cat = np.stack([rng.integers(0, t, size=n) for t in T], axis=1).astype(np.int32)
    cat[1000:60_000, 1:] = cat[0, 1:]                                     # popular prefixes, items that repeat
    cat[60_000:90_000] = cat[:30_000]
    cat[-1] = np.asarray(T) - 1                                           # the last bit of the region, and of all keys
    w = synth.scaled(synth.WORKLOADS["tiny"], L=len(T), T=T, n_items=n, batch=2, beam=64, n_hist=3, load_factor=load_factor)
    case = Case(w, catalog=cat, hist=cat[rng.integers(0, n, size=(2, 3))]).prefill()
    keys_cat = O.pack_keys(cat, T)
    V = O.ValidSet(cat, T)
    prefixes = [np.unique(O.pack_keys(cat[:, : lv + 1], T[: lv + 1])) for lv in range(len(T))]
    near = cat[:300_000].copy()
    near[:, -1] = rng.integers(0, T[-1], size=len(near))                  # prefixes that exist, mostly with other last codes
    probes = np.concatenate([cat, near, np.stack([rng.integers(0, t, size=300_000) for t in T], axis=1).astype(np.int32)])
    want = V.contains(probes)
    keys = case.eng.pack(torch.from_numpy(probes).cuda())
    case.eng.profile_read()
    case.eng.build_hashset()
    # eight launches by parts; one, for the whole catalogue, just below the least number of items
    assert case.eng.profile_read()["hash"]["launches"] == (1 if n == 1_572_863 else 8)
    case.eng.set_option(4, 1)                                             # the filter at every level reads every region
    for _ in range(2):
        assert case.n_unique == len(np.unique(keys_cat))
        assert np.array_equal(case.eng.probe(keys).cpu().numpy().astype(bool), want)
        beams = case.eng.decode(w.beam, mode=2, trace=True)["trace"]["beams"].cpu().numpy()
        for lv in range(w.L):
            # the beams of a level: as many as fit of all valid extensions of the level's before, and each of them valid
            parents = prefixes[lv] % np.uint64(np.prod(T[:lv], dtype=np.int64))
            for b in range(w.batch):
                got = beams[lv, b][beams[lv, b, :, 0] >= 0]
                before = beams[lv - 1, b][beams[lv - 1, b, :, 0] >= 0]
                reach = np.isin(parents, O.pack_keys(before[:, :lv], T[:lv])).sum() if lv else len(parents)
                assert len(got) == min(w.beam, reach) and V.contains_prefix(got[:, : lv + 1]).all()
        case.n_unique = case.eng.build_hashset()                          # the same tables once more
    case.eng.close()


def test_bad_code_is_reported():
    from gpu_helpers import Case
    from paper_2511_18793_b200 import binding
    T, n = (63, 61, 59, 37, 50), 1_600_000
    rng = np.random.default_rng(1)
    cat = np.stack([rng.integers(0, t, size=n) for t in T], axis=1).astype(np.int32)
    w = synth.scaled(synth.WORKLOADS["tiny"], L=5, T=T, n_items=n, batch=1, beam=2, n_hist=1, load_factor=0.25)
    case = Case(w, catalog=cat, hist=cat[:1][None])
    case.eng.catalog[777, 2] = 59
    with pytest.raises(binding.NezhaError):
        case.eng.build_hashset()
    case.eng.catalog[777, 2] = 58
    cat[777, 2] = 58
    assert case.eng.build_hashset() == len(np.unique(O.pack_keys(cat, T)))
    case.eng.close()
