"""What the batched calls take as items: any sequence of mappings, as long as it has a length."""
import collections

import numpy as np
import pytest
import torch

from paper_2410_16926_b200 import pvq


class Lazy(collections.UserDict):
    pass


def test_items_without_a_length_are_refused():
    with pytest.raises(TypeError):
        pvq.encode_batched((it for it in ()), torch.float32, 32, 50, 16, None)
    with pytest.raises(TypeError):
        pvq.decode_batched(iter([]), 32, 50, 16, None)


def test_missing_entries_are_key_errors():
    t = torch.zeros((1, 2, 3), dtype=torch.int32)
    for kind in (dict, Lazy):
        with pytest.raises(KeyError):
            pvq.decode_batched([kind(codes=t)], 32, 50, 16, None)
        with pytest.raises(KeyError):
            pvq.decode_batched([kind(codes=t, scale_idx=t, row_norm=t)], 32, 50, 16, None)
    with pytest.raises((TypeError, AttributeError)):
        pvq.decode_batched([3], 32, 50, 16, None)


@pytest.mark.gpu
@pytest.mark.parametrize("kind", [Lazy, collections.ChainMap, collections.OrderedDict])
def test_mappings_that_are_not_dicts(kind):
    N, K, b = 32, pvq.max_pulses(32, 96), 4
    table = pvq.build_count_table(N, K)
    results = []
    for make in (dict, lambda **kw: kind(kw)):
        items = []
        for rows, G in ((3, 5), (7, 64)):
            edges, levels = pvq.build_scale_codebook(N, G, b)
            x = torch.from_numpy(np.random.default_rng(rows).standard_normal((rows, G * N)).astype(np.float32)).cuda()
            codes, sidx, rnorm = pvq.alloc_encoded(rows, G, pvq.code_words(N, K), b)
            items.append(make(x=x, codes=codes, scale_idx=sidx, row_norm=rnorm, edges=edges, levels=levels, cols=G * N,
                              out=torch.empty((rows, G * N), dtype=torch.bfloat16, device="cuda")))
        pvq.encode_batched(tuple(items), torch.float32, N, K, b, table)
        pvq.decode_batched(collections.deque(items), N, K, b, table)
        torch.cuda.synchronize()
        results.append([it[k].cpu().view(torch.uint8) for it in items for k in ("codes", "scale_idx", "row_norm", "out")])
    assert all(torch.equal(p, q) for p, q in zip(*results))
