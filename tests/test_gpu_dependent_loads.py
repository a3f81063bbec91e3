"""Kernels that are resident while the kernel before them still writes their inputs
(programmatic dependent launches): what they read goes past the read-only path, which
is for memory that nobody writes during a kernel's life, and chains whose every link
rewrites the next one's inputs give the results of the same chain run link by link."""
import os
import re

import numpy as np
import pytest
import torch

from paper_2606_31160_gb300 import build, sd
from tests.helpers import ensure_lib


def test_sources_read_no_input_by_the_read_only_path():
    """Every source with a dependent launch: no __ldg, no const __restrict__ parameter (which the
    compiler may read the same way)."""
    seen = 0
    for name in sorted(os.listdir(build.CSRC)):
        with open(os.path.join(build.CSRC, name)) as f:
            code = re.sub(r"//[^\n]*", "", f.read())
        if "sd_pdl_enter()" not in code and "griddep_wait()" not in code:
            continue
        seen += 1
        assert "__ldg(" not in code, name
        assert not re.search(r"const\s+\w+\s*\*\s*__restrict__", code), name
    assert seen >= 7


def _run(chain, graph):
    """The chain twice, back to back or as a replayed graph, without a wait between its links."""
    if not graph:
        chain()
        torch.cuda.synchronize()
        return
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        chain()  # kernel attributes
    torch.cuda.current_stream().wait_stream(side)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        chain()
    g.replay()
    torch.cuda.synchronize()


@pytest.mark.gpu
@pytest.mark.parametrize("graph", [False, True])
def test_greedy_behind_a_kernel_that_writes_its_logits_and_drafts(graph):
    """rope_apply rotates the buffer that accept_greedy reads as logits; the drafts of a
    step are the argmax that the step before wrote."""
    ensure_lib()
    R, V, steps = 8, 151936, 12
    K = R - 1
    first = torch.randn((1, R, V), generator=torch.Generator().manual_seed(5)).to(torch.bfloat16).cuda()
    # rows 0..2 do not turn: their argmax stays, and the drafts of later steps match it
    pos = torch.tensor([0, 0, 0, 1, 2, 3, 4, 5], dtype=torch.int32, device="cuda").view(1, R, 1).expand(1, R, 3).contiguous()
    k = torch.zeros((1, R, 1, 128), dtype=torch.bfloat16, device="cuda")
    ws = sd.workspace(sd.greedy_workspace_bytes(1, K, V))
    logits = first.clone()
    star = torch.zeros((steps + 1, 1, R), dtype=torch.int32, device="cuda")
    n_emit = torch.zeros((steps, 1), dtype=torch.int32, device="cuda")
    tokens = torch.zeros((steps, 1, R), dtype=torch.int32, device="cuda")

    def link(z, s):
        sd.rope_apply(z.view(1, R, V // 128, 128), k, pos, (16, 24, 24))
        sd.accept_greedy(z, star[s].view(-1)[:K].view(1, K), ws=ws, n_emit=n_emit[s], tokens=tokens[s], argmax=star[s + 1])

    def chain():
        logits.copy_(first)
        for s in range(steps):
            link(logits, s)

    _run(chain, graph)
    got = star.cpu().numpy(), n_emit.cpu().numpy(), tokens.cpu().numpy()
    z = first.clone()
    want = np.zeros(K, dtype=np.int64)
    for s in range(steps):
        sd.rope_apply(z.view(1, R, V // 128, 128), k, pos, (16, 24, 24))
        torch.cuda.synchronize()
        draft, want_star = want[:K], z[0].float().cpu().numpy().argmax(-1)
        ell = int(np.cumprod(draft == want_star[:K]).sum())
        assert got[0][s + 1, 0].tolist() == want_star.tolist()
        assert got[1][s, 0] == ell + 1
        assert got[2][s, 0].tolist() == [int(want_star[j]) if j <= ell else -1 for j in range(R)]
        want = want_star
    assert sd.get_device_error() == 0


@pytest.mark.gpu
@pytest.mark.parametrize("graph", [False, True])
@pytest.mark.parametrize("offset", [0, 1])  # rows on 16-byte boundaries, and off them
def test_sampling_behind_a_kernel_that_writes_its_logits(graph, offset):
    """kv_append copies the buffers that accept_sample reads as logits."""
    ensure_lib()
    K, V, steps, T = 3, 4096, 8, 0.8
    cap = ((K + 1) * V + 64) // 64  # rows of 128 bf16, 64 fp32 logits each
    g = torch.Generator().manual_seed(9)
    z_t = (torch.randn((steps, cap * 64), generator=g) * 3).cuda()
    z_d = (z_t.cpu() + 0.5 * torch.randn((steps, cap * 64), generator=g)).cuda()
    draft = torch.randint(0, V, (steps, 1, K), generator=g, dtype=torch.int32).cuda()
    u = torch.rand((steps, 1, K + 1), generator=g).cuda()
    cache = sd.KVCache(torch.zeros((1, 1, cap, 128), dtype=torch.bfloat16, device="cuda"),
                       torch.zeros((1, 1, cap, 128), dtype=torch.bfloat16, device="cuda"),
                       torch.zeros(1, dtype=torch.int32, device="cuda"))
    none = torch.zeros(1, dtype=torch.int32, device="cuda")
    ws = sd.workspace(sd.sample_workspace_bytes(1, K, V))
    rows = lambda flat, n: flat[offset:offset + n * V].view(1, n, V)  # noqa: E731
    n_emit = torch.zeros((steps, 1), dtype=torch.int32, device="cuda")
    tokens = torch.zeros((steps, 1, K + 1), dtype=torch.int32, device="cuda")
    as_rows = lambda z: z.view(torch.bfloat16).view(1, cap, 1, 128)  # noqa: E731

    def chain():
        for s in range(steps):
            sd.kv_append(cache, as_rows(z_t[s]), as_rows(z_d[s]))
            sd.accept_sample(rows(cache.k.view(-1).view(torch.float32), K + 1), rows(cache.v.view(-1).view(torch.float32), K),
                             draft[s], u[s], T, ws=ws, n_emit=n_emit[s], tokens=tokens[s])
            sd.kv_rollback(cache.len, none, cap)

    _run(chain, graph)
    for s in range(steps):
        n, t = sd.accept_sample(rows(z_t[s], K + 1), rows(z_d[s], K), draft[s], u[s], T)
        torch.cuda.synchronize()
        assert n.tolist() == n_emit[s].tolist() and t.tolist() == tokens[s].tolist()
    assert sd.get_device_error() == 0 and cache.len.item() == 0
