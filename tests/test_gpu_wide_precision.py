"""Error of the row-tile attention against 64 bits where few keys hold the mass, and
where scores and values are far from 1.

Every bound on few keys is the rounding of an exact output to bf16 on the same inputs, with 1% for
the weights (2^-17 each, beside the output's 2^-9) and the fp32 scores."""
import numpy as np
import pytest
import torch

import oracle
from paper_2606_31160_gb300 import sd, workloads
from tests.helpers import attn_within, ensure_lib, to64

pytestmark = pytest.mark.gpu
# packed rows 1, 32 | 48 | 64 | 68, 80 | 96 (two m-blocks)
SHAPES = [(1, 1), (4, 8), (2, 16), (4, 12), (4, 16), (4, 17), (5, 16), (6, 16)]


@pytest.fixture(scope="module", autouse=True)
def _lib():
    ensure_lib()


def _bf(x):
    return to64(workloads.to_bf16(x))


def _inputs(seed, B, G, R, Hkv, cap, D, v_scale=1.0):
    rng = np.random.default_rng(seed)
    draw = lambda *s: rng.standard_normal(s).astype(np.float32)  # noqa: E731
    return [draw(B, R, Hkv * G, D), draw(B, Hkv, cap, D), draw(B, Hkv, cap, D) * np.float32(v_scale), draw(B, R, Hkv, D),
            draw(B, R, Hkv, D) * np.float32(v_scale)]


def _call(q, k, v, k_new, v_new, prefix, fused):
    """Position-0 new rows (an identity rotation); returns (out, q, keys, values, lengths) in 64 bits."""
    B, R, Hq, D = q.shape
    bf = workloads.to_bf16
    kc, vc = k.copy(), v.copy()
    for b, n in enumerate(prefix):
        if not fused:
            kc[b, :, n:n + R] = k_new[b].transpose(1, 0, 2)
            vc[b, :, n:n + R] = v_new[b].transpose(1, 0, 2)
    cache = sd.KVCache(bf(kc).cuda(), bf(vc).cuda(),
                       torch.tensor([n + (0 if fused else R) for n in prefix], dtype=torch.int32).cuda())
    qd = bf(q).cuda()
    if fused:
        sections = (16, 24, 24) if D == 128 else (8, 12, 12)
        out = sd.verify_layer(qd, bf(k_new).cuda(), bf(v_new).cuda(), torch.zeros((B, R, 3), dtype=torch.int32).cuda(),
                              sections, cache, 0, 1e6)
    else:
        out = sd.verify_attention(qd, cache)
    torch.cuda.synchronize()
    assert sd.get_device_error() == 0
    return to64(out), to64(qd), to64(cache.k), to64(cache.v), cache.len.cpu().numpy()


def _rel(x, ref):
    return float(np.sqrt(((x - ref) ** 2).sum() / (ref ** 2).sum()))


@pytest.mark.parametrize("G,R", SHAPES)
@pytest.mark.parametrize("fused", [True, False])
def test_new_keys_alone(G, R, fused):
    """Without a prefix the weights are those of the new keys, 16 bits and more: what is left
    is the rounding of the output."""
    q, k, v, k_new, v_new = _inputs(31 * G + R, 6, G, R, 2, 40, 128)
    out, *rest = _call(q, k, v, k_new, v_new, [0] * 6, fused)
    ref = oracle.verify_attention(*rest)
    assert _rel(out, ref) <= 1.01 * _rel(_bf(ref.astype(np.float32)), ref) + 1e-6


@pytest.mark.parametrize("R", [17, 24, 31, 32])
@pytest.mark.parametrize("fused", [True, False])
@pytest.mark.parametrize("csize,prefix", [(1, [1, 7, 32, 100, 128, 200]), (4, [200, 320, 500, 512, 600, 700])])
def test_many_rows_of_one_head(R, fused, csize, prefix):
    """17 to 32 new rows of one query head a KV head: the weights of the prefix to 16 bits too."""
    q, k, v, k_new, v_new = _inputs(7 + R + csize, len(prefix), 1, R, 2, 760, 128)
    sd.set_cluster_size(csize)
    try:
        out, *rest = _call(q, k, v, k_new, v_new, prefix, fused)
    finally:
        sd.set_cluster_size(0)
    ref = oracle.verify_attention(*rest)
    assert _rel(out, ref) <= 1.01 * _rel(_bf(ref.astype(np.float32)), ref)


# (log2 of every score, log2 of the values): with weights that are not relative to one of
# the row's own scores their products leave the range of fp32
@pytest.mark.parametrize("level,scale", [(-60.0, -90), (-75.0, -60), (50.0, 90), (55.0, 75), (-20.0, -110), (0.0, -100), (0.0, 100)])
@pytest.mark.parametrize("G,R", [(4, 1), (4, 8), (4, 12), (4, 17)])
@pytest.mark.parametrize("fused,cluster,D", [(True, 0, 128), (True, 1, 128), (False, 0, 128), (False, 4, 64)])
def test_values_far_from_one(level, scale, G, R, fused, cluster, D):
    prefix = [0, 5, 700, 1500]
    q, k, v, k_new, v_new = _inputs(int(1000 + level + scale) + G * R, len(prefix), G, R, 1, 1540, D, 2.0 ** scale)
    beta = level / (8.0 * 1.4426950408889634 / np.sqrt(D))
    q[..., 5], k[..., 5], k_new[..., 5] = 8.0, beta, beta
    sd.set_cluster_size(cluster)
    try:
        out, qd, kd, vd, lens = _call(q, k, v, k_new, v_new, prefix, fused)
    finally:
        sd.set_cluster_size(0)
    ref = oracle.verify_attention(qd, kd, vd * 2.0 ** -scale, lens)
    assert attn_within(out * 2.0 ** -scale, ref), np.abs(out * 2.0 ** -scale - ref).max()


@pytest.mark.parametrize("G,R", [(4, 1), (4, 8), (4, 12), (4, 17), (6, 16)])
def test_scores_of_tens_of_thousands(G, R):
    """Rotated rows whose one pair makes scores of 3e4: fp32 sums are off by some 2^-24 of
    them there, 2% of a weight, and a row's reference has to be its rotated score (rounding
    the rotated rows to bf16 moves it by 2^-8: 100 and more)."""
    prefix = [0, 5, 700, 1500]
    B, D = len(prefix), 128
    q, k, v, k_new, v_new = _inputs(G * R, B, G, R, 2, 1540, D)
    for x in (q, k, k_new):
        x[..., 6], x[..., 7] = 500.0, 300.0
    bf = workloads.to_bf16
    cache = sd.KVCache(bf(k).cuda(), bf(v).cuda(), torch.tensor(prefix, dtype=torch.int32).cuda())
    qd = bf(q).cuda()
    pos = (37 + torch.arange(R, dtype=torch.int32))[None, :, None].expand(B, R, 3).contiguous().cuda()
    out = torch.full_like(qd, float("nan"))
    sd.verify_layer(qd, bf(k_new).cuda(), bf(v_new).cuda(), pos, (16, 24, 24), cache, 0, 1e6, out=out)
    torch.cuda.synchronize()
    assert sd.get_device_error() == 0
    ref = oracle.verify_attention(to64(qd), to64(cache.k), to64(cache.v), cache.len.cpu().numpy())
    assert np.isfinite(to64(out)).all() and np.abs(to64(out) - ref).max() < 0.2
