"""The tensor-core prefill path against the general kernels (fp32 products, one virtual unit per position) on the same
inputs: every group size, block size and head dim class it has code for, at the edges of its tiles and ranges.

Tolerance: probabilities and linear coefficients enter their products as two bf16 parts (2^-17 relative per term), phi as
22 bits, everything else in fp32, so single outputs agree to a few 1e-5; the residual's error is that of its operands,
2^-17 |o_bar|, times the RMSNorm's amplification 1 / |o_rla|, which the sizes below keep under about 10 (near-complete
selection, where it is larger, is the last case, with its own bound)."""
import ctypes as C

import numpy as np
import pytest
import torch

from paper_2601_22379_b200 import binding, runner, synth
from tests import parity

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
RTOL, ATOL = 3e-4, 3e-5

CASES = [
    # batch, hkv, G, d, B, top_k, n_sink, n_local, L0, T, flags
    (1, 2, 4, 128, 64, 8, 1, 2, 0, 64, 0),             # exactly one range
    (2, 2, 4, 128, 64, 6, 1, 2, 63, 130, 0),           # a chunk that starts on a block's last token
    (1, 1, 4, 128, 64, 16, 1, 4, 64 * 40, 1, 0),       # a single position
    (1, 2, 4, 128, 128, 6, 1, 2, 1000, 200, 0),        # two tiles of tokens per block
    (1, 2, 4, 128, 32, 8, 1, 4, 700, 97, 0),           # two blocks per tile
    (1, 2, 4, 128, 16, 8, 0, 0, 333, 75, 0),           # four blocks per tile; own block not always selected
    (1, 1, 1, 128, 64, 5, 1, 1, 900, 140, 0),          # groups of 1, 2, 3, 5, 8, 16
    (1, 1, 2, 64, 32, 5, 1, 1, 500, 70, 0),
    (1, 1, 3, 128, 64, 6, 1, 2, 700, 66, 0),
    (2, 2, 5, 128, 64, 8, 1, 4, 1500, 131, 0),
    (1, 2, 8, 64, 64, 8, 1, 2, 801, 65, 0),
    (1, 1, 16, 128, 64, 8, 1, 4, 64 * 21 + 1, 90, 0),
    (1, 2, 4, 64, 64, 8, 1, 2, 64 * 30 + 5, 300, binding.SPLA_STATS_BF16),
    (1, 2, 4, 128, 64, 64, 1, 4, 64 * 90, 100, 0),     # longest selection
    (1, 1, 4, 128, 64, 8, 1, 2, 700, 90, binding.SPLA_FIRST_ORDER),
    (1, 1, 4, 128, 64, 8, 0, 0, 700, 90, binding.SPLA_NO_RLA),
    (1, 1, 4, 128, 16, 8, 1, 4, 16 * 600, 40, 0),      # more than 512 blocks: 32 keys per lane of a warp
    (1, 1, 4, 64, 16, 8, 1, 4, 16 * 1100, 33, binding.SPLA_DEBUG_BOUNDS),   # more than 1024: a CTA selects
]


def _inputs(case, seed=11):
    batch, hkv, G, d, B, top_k, ns, nl, L0, T, flags = case
    w = synth.Workload("case", seed, batch=batch, n_q_heads=hkv * G, n_kv_heads=hkv, head_dim=d, block_size=B, top_k=top_k,
                       context=max(L0, 1), n_sink=ns, n_local=nl, n_outlier_channels=4, outlier_scale=3.0, n_steps=T)
    g = torch.Generator(device=DEV).manual_seed(seed)
    K0, V0, _ = runner.generate_prefill(w, DEV)
    k = torch.randn(batch, hkv, T, d, generator=g, device=DEV)
    k[..., :3] *= 3.0
    v = torch.randn(batch, hkv, T, d, generator=g, device=DEV)
    q0 = synth.query_directions(w).to(DEV).repeat_interleave(G, dim=1)[:, None]
    q = (q0 + torch.randn(batch, T, hkv * G, d, generator=g, device=DEV)) / 1.4
    return w, K0[:, :, :L0].contiguous(), V0[:, :, :L0].contiguous(), *(x.to(torch.bfloat16).contiguous() for x in (k, v, q))


def _run(w, K0, V0, k, v, q, flags, **kw):
    cache = binding.SplaCache(runner.config_for(w, flags=flags), DEV)
    for t in (cache.bufs.k_cache, cache.bufs.v_cache):
        t.fill_(float("nan"))                           # nothing past a sequence's end may reach a result
    if K0.shape[2]:
        cache.append_tokens(K0, V0)
    T = k.shape[2]
    sel = torch.full((w.batch, T, w.n_kv_heads, w.top_k), -7, dtype=torch.int32, device=DEV)
    n0 = binding.launch_count()
    out = cache.prefill(k, v, q, synth.gamma(w).to(DEV), sel_idx=sel, **kw)
    cache.launches = binding.launch_count() - n0
    torch.cuda.synchronize()
    assert cache.sync_status() == 0
    return out, sel, cache


def _launches(w, T, flags, tensor):
    """Kernels of one prefill whose scratch holds the whole chunk: the append, then own-block masses, states, scan, scores,
    selection and attention, or (general) statistics, scan, scores and attention."""
    one_pass = tensor and w.head_dim == 128 and w.batch * w.n_kv_heads * T >= 64
    rla = not flags & binding.SPLA_NO_RLA
    return (1 if T <= 32 or one_pass else 2) + (4 + 2 * rla if tensor else 3 + rla)


@pytest.mark.parametrize("case", CASES, ids=lambda c: "-".join(map(str, c)))
def test_tensor_core_prefill_equals_the_general_kernels(case):
    w, K0, V0, k, v, q = _inputs(case)
    flags = case[-1]
    a, sel_a, ca = _run(w, K0, V0, k, v, q, flags)
    b, sel_b, cb = _run(w, K0, V0, k, v, q, flags | binding.SPLA_GENERAL_KERNELS)
    assert ca.launches == _launches(w, k.shape[2], flags, True)
    batches, odd = divmod(cb.launches - _launches(w, k.shape[2], flags, False), 2)   # (batches of positions beyond the first)
    assert batches in (0, 1) and not odd
    assert torch.isfinite(a).all()
    same = (sel_a == sel_b).all(dim=-1)                 # [batch, T, hkv]; near-ties may fall the other way
    assert same.float().mean().item() >= 0.99
    rows = same.repeat_interleave(w.group, dim=2)
    np.testing.assert_allclose(a[rows].cpu().numpy(), b[rows].cpu().numpy(), rtol=RTOL, atol=ATOL)
    if not flags & binding.SPLA_NO_RLA:
        rel = (ca.bufs.rla_state - cb.bufs.rla_state).norm() / cb.bufs.rla_state.norm()
        assert rel.item() < parity.STATE_TOL_TENSOR + parity.STATE_TOL_FMA   # (the history went in on either kernel)
    least, _, _ = _run(w, K0, V0, k, v, q, flags, workspace_bytes=1)
    assert torch.equal(least, a)                        # positions per launch change nothing


def test_tensor_core_prefill_under_near_complete_selection():
    """All blocks but one or two selected: |o_bar| is 20 to 40 times |o_rla| here, and with it the tolerance."""
    case = (1, 2, 4, 128, 64, 30, 1, 4, 64 * 30 + 9, 60, 0)
    w, K0, V0, k, v, q = _inputs(case)
    a, sel_a, _ = _run(w, K0, V0, k, v, q, 0)
    b, sel_b, _ = _run(w, K0, V0, k, v, q, binding.SPLA_GENERAL_KERNELS)
    rows = (sel_a == sel_b).all(dim=-1).repeat_interleave(w.group, dim=2)
    np.testing.assert_allclose(a[rows].cpu().numpy(), b[rows].cpu().numpy(), rtol=40 * RTOL, atol=40 * ATOL)


def test_a_wait_that_runs_out_is_reported_and_leaves_the_device_usable():
    case = CASES[1]
    w, K0, V0, k, v, q = _inputs(case)
    cache = binding.SplaCache(runner.config_for(w), DEV)
    cache.append_tokens(K0, V0)
    cache.debug_wait_hook(2000, 16)
    cache.prefill(k, v, q, synth.gamma(w).to(DEV))
    torch.cuda.synchronize()
    assert cache.sync_status() == binding.SPLA_ERR_TIMEOUT
    a, _, _ = _run(w, K0, V0, k, v, q, 0)
    assert torch.isfinite(a).all()


EDGES = [(1, 2, 4, 64 if n % 2 else 128, 16, 8, 1, 2, 16 * n + 3, 20, flags)   # n complete records: edges of the score's tiles of 64
         for n in (1, 63, 64, 65, 128, 129) for flags in (0, binding.SPLA_STATS_BF16)]
EDGES += [(1, 2, 16, 64, 64, 8, 1, 2, 0, t, 0) for t in (17 * 64, 18 * 64)]    # 288 and 304 row tiles: either side of two waves


@pytest.mark.parametrize("case", EDGES, ids=lambda c: "-".join(map(str, c)))
def test_score_tiles_and_launch_sizes_at_their_edges(case):
    """Same bounds as the first test: one record tile more or less, rows for one launch rule or the other."""
    test_tensor_core_prefill_equals_the_general_kernels(case)


@pytest.mark.parametrize("k", [8, 32, 64])                # few keys reach the bound, about as many as are ranked, too many
@pytest.mark.parametrize("blocks", [257, 513, 1023])
def test_selection_from_the_keys_that_reach_a_bound(blocks, k):
    T = 20 if k < 64 else 60                              # (20 positions of the longest selection take the general kernels)
    test_tensor_core_prefill_equals_the_general_kernels((1, 2, 4, 64, 16, k, 1, 2, 16 * blocks + 3, T, 0))


def test_selection_among_equal_scores_takes_the_first_blocks():
    """All keys alike: every free block ties, the bound keeps them all, and the list is the forced blocks and the first free ones."""
    w, K0, V0, k, v, q = _inputs((1, 2, 4, 64, 16, 16, 1, 2, 16 * 300, 5, 0))
    _, sel, _ = _run(w, torch.ones_like(K0), V0, torch.ones_like(k), v, q, 0)
    want = list(range(14)) + [299, 300]
    assert (sel.cpu() == torch.tensor(want, dtype=torch.int32)).all()


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("tiles", [1, 4, 5, 8, 9, 13, 17])
def test_without_the_residual_the_merge_waits_for_the_last_products(tiles, d):
    """A chunk of 5 positions that select all `tiles` blocks of 64: the accumulator is complete when the merge reads it, however
    many groups of four tiles the walk has (the same bits every time, and those of the general kernels to the usual bound)."""
    case = (2, 2, 4, d, 64, tiles, 0, 1, 64 * (tiles - 1) + 3, 5, binding.SPLA_NO_RLA)
    w, K0, V0, k, v, q = _inputs(case)
    a, sel_a, _ = _run(w, K0, V0, k, v, q, case[-1])
    assert (sel_a >= 0).sum(dim=-1).eq(tiles).all()
    for _ in range(10):
        again, _, _ = _run(w, K0, V0, k, v, q, case[-1])
        assert torch.equal(again, a)
    b, _, _ = _run(w, K0, V0, k, v, q, case[-1] | binding.SPLA_GENERAL_KERNELS)
    np.testing.assert_allclose(a.cpu().numpy(), b.cpu().numpy(), rtol=RTOL, atol=ATOL)


@pytest.mark.parametrize("flags", [0, binding.SPLA_STATS_BF16])
@pytest.mark.parametrize("d,B", [(64, 16), (64, 128), (128, 32), (128, 64)])
def test_a_positions_own_block_has_the_record_that_a_step_stores(d, B, flags):
    """The log mass of each position's growing block (the workspace begins with it) against 64 bits on the record that a
    token-by-token append leaves in the cache.  2e-6: the fast logarithm's 4e-7 and sums of 128 terms of size 1 at most in
    fp32; a record rounded to the other 16-bit neighbour moves it by 1e-4 and more."""
    case = (1, 2, 4, d, B, 8, 1, 2, B * 9 + 7, B + 30, flags)
    w, K0, V0, k, v, q = _inputs(case)
    _, _, cache = _run(w, K0, V0, k, v, q, flags)
    T, G = k.shape[2], w.group
    got = cache._prefill_ws[:2 * T * G * 4].view(torch.float32).view(2, T, G).double()
    step = binding.SplaCache(runner.config_for(w, flags=flags), DEV)
    step.append_tokens(K0, V0)
    worst = 0.0
    for t in range(T):
        step.append_tokens(k[:, :, t:t + 1].contiguous(), v[:, :, t:t + 1].contiguous())
        pos = K0.shape[2] + t
        mean, var = step.bufs.stats[0, :, pos // B].double().unbind(1)
        x = q[0, t].double().view(2, G, d) / d ** 0.5
        want = np.log((pos % B + 1) / B) + (x * mean[:, None]).sum(-1) + torch.log1p((0.5 * x * x * var[:, None]).sum(-1))
        worst = max(worst, (got[:, t] - want).abs().max().item())
    assert worst < 2e-6, worst


def test_scratch_that_is_enough_for_the_general_kernels_only():
    """Few tokens of small groups: the general kernels need less than the tensor-core path (a state per range); a call with their
    minimum runs on them, one with less is refused."""
    case = (2, 2, 1, 128, 64, 1, 0, 0, 300, 3, 0)
    w, K0, V0, k, v, q = _inputs(case)
    gamma = synth.gamma(w).to(DEV)
    want, sel, _ = _run(w, K0, V0, k, v, q, binding.SPLA_GENERAL_KERNELS)
    sizes = []
    for flags in (0, binding.SPLA_GENERAL_KERNELS):
        lo = C.c_size_t()
        assert binding.load().spla_query_prefill_workspace(C.byref(runner.config_for(w, flags=flags)), 3, C.byref(lo), None) == 0
        sizes.append(lo.value)
    assert sizes[1] < sizes[0]
    for size, status in ((sizes[1], 0), (sizes[1] - 1, binding.SPLA_ERR_INVALID_ARG)):
        cache = binding.SplaCache(runner.config_for(w), DEV)
        cache.append_tokens(K0, V0)
        ws, out = torch.empty(size, dtype=torch.uint8, device=DEV), torch.empty_like(want)
        assert cache.lib.spla_prefill(cache.handle, k.data_ptr(), v.data_ptr(), q.data_ptr(), 3, gamma.data_ptr(), out.data_ptr(),
                                      None, ws.data_ptr(), size, torch.cuda.current_stream().cuda_stream) == status
        torch.cuda.synchronize()
        assert cache.sync_status() == 0
        if status == 0:
            np.testing.assert_allclose(out.cpu().numpy(), want.cpu().numpy(), rtol=RTOL, atol=ATOL)


@pytest.mark.parametrize("case,tensor", [
    ((1, 2, 4, 128, 128, 40, 1, 4, 128 * 60, 1, 0), False),       # 80 tiles of 64 tokens one after the other, or 80 CTAs
    ((1, 2, 4, 128, 128, 40, 1, 4, 128 * 60, 64, 0), True),
    ((2, 4, 1, 64, 64, 64, 1, 4, 64 * 150, 8, 0), False),
    ((2, 4, 1, 64, 64, 64, 1, 4, 64 * 150, 33, 0), True),         # more than 256 virtual units
    ((1, 4, 8, 128, 64, 8, 1, 4, 64 * 150, 4, 0), True),          # a short selection
], ids=str)
def test_a_short_chunk_takes_the_path_that_is_faster_for_it(case, tensor):
    w, K0, V0, k, v, q = _inputs(case)
    a, sel_a, ca = _run(w, K0, V0, k, v, q, 0)
    b, sel_b, cb = _run(w, K0, V0, k, v, q, binding.SPLA_GENERAL_KERNELS)
    T = k.shape[2]
    assert ca.launches - (_launches(w, T, 0, True) - 6) == (6 if tensor else 4)     # (the appends differ; not what follows)
    rows = (sel_a == sel_b).all(dim=-1).repeat_interleave(w.group, dim=2)
    assert rows.float().mean().item() >= 0.99
    np.testing.assert_allclose(a[rows].cpu().numpy(), b[rows].cpu().numpy(), rtol=RTOL, atol=ATOL)
    least, _, _ = _run(w, K0, V0, k, v, q, 0, workspace_bytes=1)
    assert torch.equal(least, a)


@pytest.mark.parametrize("d,B,G", [(128, 64, 4), (64, 16, 4), (128, 128, 2), (128, 32, 1)])
def test_a_value_that_is_not_finite_reaches_only_the_positions_that_attend_to_it(d, B, G):
    """Without the residual: a NaN in a late token of the chunk, an infinity in one old block.  Positions before the token, and
    those that did not select the block, are as if the values were finite; the others are not finite in those channels."""
    T = 300                                                   # (more than the short chunks that take the general kernels)
    case = (1, 2, G, d, B, 4, 0, 1, B * 12 + 5, T, binding.SPLA_NO_RLA)
    w, K0, V0, k, v, q = _inputs(case)
    clean, sel, cache = _run(w, K0, V0, k, v, q, case[-1])
    assert cache.launches == _launches(w, T, case[-1], True)
    V1, v1 = V0.clone(), v.clone()
    blk = next(x for x in range(12) if 0 < (sel[:, :, 0] == x).sum() < T)     # an old block that some positions select
    late = 41
    V1[:, 0, B * blk + 1, 7] = float("inf")
    v1[:, 1, late, d - 1] = float("nan")
    a, sel_a, _ = _run(w, K0, V1, k, v1, q, case[-1])
    b, _, _ = _run(w, K0, V1, k, v1, q, case[-1] | binding.SPLA_GENERAL_KERNELS)
    assert torch.equal(sel_a, sel)
    hit = torch.zeros_like(a, dtype=torch.bool)
    hit[:, :, :G, 7] = (sel[:, :, 0] == blk).any(-1)[..., None]
    seen = (sel[:, :, 1] == (K0.shape[2] + late) // B).any(-1) & (torch.arange(T, device=DEV) >= late)
    hit[:, :, G:, d - 1] = seen[..., None]
    assert seen.any()
    assert torch.equal(~torch.isfinite(a), hit) and torch.equal(~torch.isfinite(b), hit)
    assert torch.equal(a[~hit], clean[~hit])


@pytest.mark.parametrize("blocks", [1024, 1025, 4096, 4097, 16384])
def test_selection_by_a_warp_and_by_a_cta_up_to_the_longest_sequence(blocks):
    """Either side of each instance of the selection kernel, and of the tiles' bitmap of selected blocks at its last word."""
    for more in (0, 1):                                       # a chunk that ends with a block, and inside one
        test_tensor_core_prefill_equals_the_general_kernels((1, 1, 4, 64, 16, 8, 1, 2, 16 * blocks - 20 - 7 * more, 20, 0))


def test_above_the_longest_sequence_of_the_tensor_core_path():
    """16385 blocks: the general kernels, and their scratch."""
    w, K0, V0, k, v, q = _inputs((1, 1, 4, 64, 16, 8, 1, 2, 16 * 16384 - 19, 20, 0))
    sizes = []
    for flags in (0, binding.SPLA_GENERAL_KERNELS):
        lo = C.c_size_t()
        assert binding.load().spla_query_prefill_workspace(C.byref(runner.config_for(w, flags=flags)), 20, C.byref(lo), None) == 0
        sizes.append(lo.value)
    assert sizes[0] == sizes[1]
    a, sel_a, ca = _run(w, K0, V0, k, v, q, 0)
    b, sel_b, cb = _run(w, K0, V0, k, v, q, binding.SPLA_GENERAL_KERNELS)
    assert ca.launches == cb.launches and torch.equal(a, b) and torch.equal(sel_a, sel_b)
