"""The row tiles (32, 48, 64 and 80 packed query rows per KV head, two m-blocks
above 80) against the float64 oracle: every edge of the tile choice, prefixes
around the 32-key split and the 128-key tile, causal and block masks, the fused
layer and the attention; and scores far from 0 and from each other: a row's reference
is its score against new key 0, and a CTA with a row sum above 2^64 runs its range a
second time."""
import numpy as np
import pytest
import torch

import oracle
from paper_2606_31160_gb300 import sd, workloads
from tests.helpers import attn_within, ensure_lib, to64

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    ensure_lib()


def _run(q, k, v, k_new, v_new, prefix, fused, block):
    """Position-0 new rows (an identity rotation) through the layer or the attention."""
    sections = (16, 24, 24) if q.shape[-1] == 128 else (8, 12, 12)
    B, R, Hq, D = q.shape
    bf = workloads.to_bf16
    kc, vc = np.full_like(k, np.nan), np.full_like(v, np.nan)  # stale rows hold NaN
    for b, n in enumerate(prefix):
        kc[b, :, :n], vc[b, :, :n] = k[b, :, :n], v[b, :, :n]
        if not fused:
            kc[b, :, n:n + R] = k_new[b].transpose(1, 0, 2)
            vc[b, :, n:n + R] = v_new[b].transpose(1, 0, 2)
    lens = torch.tensor([n + (0 if fused else R) for n in prefix], dtype=torch.int32).cuda()
    cache = sd.KVCache(bf(kc).cuda(), bf(vc).cuda(), lens)
    qd = bf(q).cuda()
    if fused:
        pos = torch.zeros((B, R, 3), dtype=torch.int32).cuda()
        out = sd.verify_layer(qd, bf(k_new).cuda(), bf(v_new).cuda(), pos, sections, cache, 0, 1e6, block=block)
    else:
        out = sd.verify_attention(qd, cache, block=block)
    torch.cuda.synchronize()
    assert sd.get_device_error() == 0
    ref = oracle.verify_attention(to64(qd), to64(cache.k), to64(cache.v), cache.len.cpu().numpy(), block=block)
    assert np.isfinite(to64(out)).all() and attn_within(to64(out), ref), np.abs(to64(out) - ref).max()


# (G, R): 1, 4, 17, 30, 32 (17, 31 new rows: past the 32-row tile's 16) | 33, 48 | 49, 64 | 65, 68, 80 | 81, 96 | 98, 128 packed rows, up to 31 new rows
@pytest.mark.parametrize("G,R", [(1, 1), (4, 1), (17, 1), (2, 15), (4, 8), (2, 16), (1, 17), (1, 31), (11, 3), (4, 12), (7, 7), (4, 16), (5, 13), (4, 17), (16, 5), (27, 3), (6, 16), (7, 14),
                                 (4, 31), (8, 16)])
@pytest.mark.parametrize("fused,block,D", [(True, False, 128), (True, True, 128), (False, False, 128), (False, False, 64),
                                           (False, True, 64)])
def test_tile_edges(G, R, fused, block, D):
    prefix = [0, 1, 31, 127, 128, 129, 700]
    B, Hkv, cap = len(prefix), 2, 760
    rng = np.random.default_rng(100 * G + R)
    draw = lambda *s: rng.standard_normal(s).astype(np.float32)  # noqa: E731
    _run(draw(B, R, Hkv * G, D), draw(B, Hkv, cap, D), draw(B, Hkv, cap, D), draw(B, R, Hkv, D), draw(B, R, Hkv, D),
         prefix, fused, block)


# the score (log2) around which a third of the keys, or all, lie: far outside the
# range on either side, and just inside it
@pytest.mark.parametrize("G,R", [(4, 1), (4, 8), (6, 8), (8, 8), (4, 17)])
@pytest.mark.parametrize("level", [-150.0, 100.0, -70.0, 55.0])
@pytest.mark.parametrize("part", [1, 3])
@pytest.mark.parametrize("cluster,D", [(0, 128), (1, 128), (4, 128), (0, 64), (1, 64)])
def test_row_sums_out_of_range(G, R, level, part, cluster, D):
    prefix = [1500, 40]
    B, Hkv, cap = len(prefix), 1, 1540
    rng = np.random.default_rng(int(1000 + level + 10 * G + R))
    draw = lambda *s: rng.standard_normal(s).astype(np.float32)  # noqa: E731
    u = np.zeros(D, dtype=np.float32)
    u[5] = 1.0
    q = draw(B, R, Hkv * G, D)
    q[..., 5] = 8.0
    k, k_new = draw(B, Hkv, cap, D), draw(B, R, Hkv, D)
    beta = level / (8.0 * 1.4426950408889634 / np.sqrt(D))
    k[:, :, :, 5] = 0.0
    k[:, :, : cap // part, 5] += beta
    k_new[..., 5] = beta if part == 1 else 0.0
    sd.set_cluster_size(cluster)
    try:
        if D == 128:
            _run(q, k, draw(B, Hkv, cap, D), k_new, draw(B, R, Hkv, D), prefix, True, False)
        _run(q, k, draw(B, Hkv, cap, D), k_new, draw(B, R, Hkv, D), prefix, False, False)
    finally:
        sd.set_cluster_size(0)


# prefixes that leave most CTAs of a cluster without a key, or end in a partial 32-key
# split, on capacities that get large clusters (which ones: test_sizes_that_only_the_rule_chooses)
@pytest.mark.parametrize("prefix,Hkv,cap", [([0, 37, 4099], 8, 4112), ([70, 4099], 2, 4112), ([4088], 4, 4112), ([16390], 4, 16400), ([8189], 8, 8206)])
@pytest.mark.parametrize("G,R", [(4, 1), (4, 8), (8, 8), (5, 12)])
@pytest.mark.parametrize("fused,D", [(True, 128), (False, 64)])
def test_cluster_sizes(prefix, Hkv, cap, G, R, fused, D):
    B = len(prefix)
    rng = np.random.default_rng(cap + 10 * G + R)
    draw = lambda *s: rng.standard_normal(s).astype(np.float32)  # noqa: E731
    prefix = [min(n, cap - R) for n in prefix]
    _run(draw(B, R, Hkv * G, D), draw(B, Hkv, cap, D), draw(B, Hkv, cap, D), draw(B, R, Hkv, D), draw(B, R, Hkv, D),
         prefix, fused, False)


# The sizes that sd_set_cluster_size does not force, and 16, on every row tile that the
# rule gives them on 152 SMs: 32, 48, 64, 80 rows, 48 with two-term weights, two m-blocks
@pytest.mark.parametrize("cs,Hkv,cap,G,R", [(cs, Hkv, cap, G, R) for cs, Hkv, cap in ((5, 14, 600), (10, 9, 8200), (12, 8, 12300), (16, 1, 4112))
                                            for G, R in ((4, 8), (4, 12), (4, 16), (5, 16), (1, 20))]
                         + [(5, 12, 2100, 6, 16), (12, 4, 8200, 6, 16), (16, 1, 4112, 6, 16)])
@pytest.mark.parametrize("fused,D", [(True, 128), (False, 128), (False, 64)])
def test_sizes_that_only_the_rule_chooses(cs, Hkv, cap, G, R, fused, D):
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("the rule's choice is that of 152 SMs")
    assert sd.verify_cluster_size(1, R, G * Hkv, Hkv, D, cap, fused) == cs
    rng = np.random.default_rng(cap + 10 * G + R)
    draw = lambda *s: rng.standard_normal(s, dtype=np.float32)  # noqa: E731
    prefix = [min(701, cap - R)]
    _run(draw(1, R, Hkv * G, D), draw(1, Hkv, cap, D), draw(1, Hkv, cap, D), draw(1, R, Hkv, D), draw(1, R, Hkv, D),
         prefix, fused, False)


def test_forced_size_is_the_size():
    for cs in (1, 2, 4, 6, 8, 16):
        sd.set_cluster_size(cs)
        try:
            assert sd.verify_cluster_size(1, 8, 32, 8, 128, 4112) == cs
            assert sd.verify_cluster_size(1, 17, 32, 8, 128, 4112, True) == cs
            assert sd.verify_cluster_size(1, 8, 32, 8, 64, 4112) == cs
            assert sd.verify_cluster_size(1, 40, 8, 8, 128, 4112) == cs     # every key in the loop
        finally:
            sd.set_cluster_size(0)
    assert sd.verify_cluster_size(1, 40, 8, 8, 64, 4112) == 0               # mma.sync
    assert sd.verify_cluster_size(1, 8, 32, 8, 64, 4112, True) == 0         # three kernels
