"""The one-pass bulk append (bf16, d = 128, more than 32 tokens) against the three-kernel one (SPLA_GENERAL_KERNELS), at the
edges of its 64-token tiles, of blocks and of its shares: K/V, statistics and log-sum-exps bit for bit, nothing written past
the end.  S_bar: phi enters as 16 bits from 256 tokens on (2^-18 relative per term, undiminished in sums of signed terms: the
tensor-core tolerance), as 24 below, where what is left is the tensor core's accumulation (cut after two tiles) and fp32."""
import pytest
import torch

from paper_2601_22379_b200 import binding, runner, synth
from tests import parity

pytestmark = pytest.mark.gpu
DEV = "cuda:0"

CASES = [
    # batch, hkv, B, window, [tokens per append, longest sequence], ragged, flags
    (2, 2, 64, None, [64], False, 0),                        # one whole tile
    (2, 2, 64, None, [33, 40, 100], False, 0),               # shorter than a tile; across a boundary
    (1, 2, 64, None, [63, 65, 64], False, 0),                # ends on, starts before a boundary
    (1, 1, 64, None, [64 * 37 + 1], False, 0),               # 16 shares of one unit
    (3, 8, 64, None, [700, 333], True, 0),
    (20, 8, 64, None, [150, 64], True, 0),                   # 160 units: more CTAs than SMs, one share each
    (2, 2, 128, None, [70, 190, 1000], False, 0),            # blocks of two tiles; a block opened in its second half
    (2, 3, 128, None, [300, 65], True, 0),
    (2, 2, 32, None, [47, 200], False, 0),
    (2, 2, 16, None, [50, 131], True, 0),
    (2, 2, 64, (32, 16), [77, 240], False, 0),               # strided windows
    (1, 2, 128, (32, 16), [150, 500], True, 0),
    (2, 2, 64, None, [130, 77], False, binding.SPLA_STATS_BF16),
    (2, 2, 64, None, [130, 77], False, binding.SPLA_NO_RLA),
    (1, 2, 64, None, [500, 301], True, binding.SPLA_DEBUG_BOUNDS),
]


@pytest.mark.parametrize("case", CASES, ids=lambda c: "-".join(map(str, c)))
def test_one_pass_append_equals_the_three_kernel_append(case):
    batch, hkv, B, window, sizes, ragged, flags = case
    w = synth.Workload("case", 5, batch=batch, n_q_heads=hkv, n_kv_heads=hkv, head_dim=128, block_size=B, top_k=8,
                       context=sum(sizes), n_outlier_channels=4, outlier_scale=3.0)
    caches = [binding.SplaCache(runner.config_for(w, flags=f, window=window, extra_context=B), DEV)
              for f in (flags, flags | binding.SPLA_GENERAL_KERNELS)]
    for c in caches:
        c.bufs.k_cache.fill_(float("nan"))
        c.bufs.v_cache.fill_(float("nan"))
    g = torch.Generator(device=DEV).manual_seed(3)
    state = torch.zeros(batch, hkv, 128, 128, dtype=torch.float64, device=DEV)
    for n in sizes:
        k, v = (torch.randn(batch, hkv, n, 128, generator=g, device=DEV).to(torch.bfloat16) for _ in range(2))
        n_new = torch.randint(0, n + 1, (batch,), generator=torch.Generator().manual_seed(n), dtype=torch.int32).to(DEV) if ragged else None
        before = binding.launch_count()
        caches[0].append_tokens(k, v, n_new)
        assert binding.launch_count() - before <= 2
        caches[1].append_tokens(k, v, n_new)
        phi = torch.softmax(k.double(), dim=-1)
        if ragged:
            phi = phi * (torch.arange(n, device=DEV)[None, :] < n_new[:, None])[:, None, :, None]
        state += phi.transpose(-1, -2) @ v.double()
    torch.cuda.synchronize()
    a, b = caches
    assert a.sync_status() == 0 and b.sync_status() == 0
    assert torch.equal(a.bufs.seq_lens, b.bufs.seq_lens)
    for name in ("k_cache", "v_cache"):
        assert torch.equal(getattr(a.bufs, name).view(torch.int16), getattr(b.bufs, name).view(torch.int16)), name
    for name in ("stats", "tok_lse"):
        assert torch.equal(getattr(a.bufs, name), getattr(b.bufs, name)), name
    if flags & binding.SPLA_NO_RLA:
        assert not a.bufs.rla_state.any()
    else:
        err = (a.bufs.rla_state.double() - state).flatten(2).norm(dim=-1) / state.flatten(2).norm(dim=-1).clamp_min(1e-30)
        assert err.max().item() < (parity.STATE_TOL_TENSOR if max(sizes) >= 256 else parity.STATE_TOL_FMA)


def test_one_pass_append_skips_and_reports_a_sequence_that_would_overflow():
    w = synth.Workload("case", 6, batch=2, n_q_heads=2, n_kv_heads=2, head_dim=128, block_size=64, top_k=8, context=300)
    cache = binding.SplaCache(runner.config_for(w), DEV)
    k = torch.randn(2, 2, 200, 128, device=DEV).to(torch.bfloat16)
    cache.append_tokens(k, k, torch.tensor([200, 100], dtype=torch.int32, device=DEV))
    before = cache.bufs.rla_state.clone()
    cache.set_length_bound(0)                                # the host is told too little: the device has to notice
    cache.append_tokens(k, k)
    torch.cuda.synchronize()
    assert cache.sync_status() == binding.SPLA_ERR_CAPACITY
    assert cache.bufs.seq_lens.cpu().tolist() == [200, 300]
    assert torch.equal(cache.bufs.rla_state[0], before[0]) and not torch.equal(cache.bufs.rla_state[1], before[1])


@pytest.mark.parametrize("batch", [1, 80], ids=["shares", "one_share"])      # 16 shares of a unit, added by a second kernel; one share
def test_a_wait_that_runs_out_is_reported_and_adds_nothing_to_the_state(batch):
    """The copies' barriers are told to expect more than arrives: every role gives up, the state is left as it was (no partial
    sum of an earlier append reaches it), and the next append of the same cache is right."""
    hkv, n = 2, 64 * 20
    w = synth.Workload("case", 7, batch=batch, n_q_heads=hkv, n_kv_heads=hkv, head_dim=128, block_size=64, top_k=8, context=2 * n)
    cache, want = (binding.SplaCache(runner.config_for(w), DEV) for _ in range(2))
    for c in (cache, want):
        c.bufs.k_cache.zero_()
        c.bufs.v_cache.zero_()
    g = torch.Generator(device=DEV).manual_seed(4)
    parts = [torch.randn(batch, hkv, n, 128, generator=g, device=DEV).to(torch.bfloat16) for _ in range(4)]
    cache.append_tokens(parts[0], parts[1])
    lens, state = cache.bufs.seq_lens.clone(), cache.bufs.rla_state.clone()
    cache.debug_wait_hook(500, 16)
    cache.append_tokens(parts[2], parts[3])
    torch.cuda.synchronize()
    assert cache.sync_status() == binding.SPLA_ERR_TIMEOUT
    assert torch.equal(cache.bufs.rla_state, state)
    cache.debug_wait_hook(0, 0)
    cache.bufs.seq_lens.copy_(lens)
    cache.set_length_bound(n)
    cache.append_tokens(parts[2], parts[3])
    want.append_tokens(parts[0], parts[1])
    want.append_tokens(parts[2], parts[3])
    torch.cuda.synchronize()
    assert cache.sync_status() == 0
    for name in ("seq_lens", "k_cache", "v_cache", "stats", "tok_lse", "rla_state"):
        assert torch.equal(getattr(cache.bufs, name), getattr(want.bufs, name)), name


@pytest.mark.parametrize("n,ragged,launches", [(47, True, 3), (48, True, 1), (47, False, 1)])
def test_few_tokens_of_many_sequences_of_different_lengths_take_the_three_kernels(n, ragged, launches):
    """75 x 4 units, more than two waves of the one-pass kernel's CTAs; the same statistics, log-sum-exps and state either way."""
    w = synth.Workload("case", 8, batch=75, n_q_heads=4, n_kv_heads=4, head_dim=128, block_size=64, top_k=8, context=200)
    caches = [binding.SplaCache(runner.config_for(w, flags=f), DEV) for f in (0, binding.SPLA_GENERAL_KERNELS)]
    g = torch.Generator(device=DEV).manual_seed(9)
    k, v = (torch.randn(75, 4, n, 128, generator=g, device=DEV).to(torch.bfloat16) for _ in range(2))
    n_new = torch.randint(0, n + 1, (75,), generator=torch.Generator().manual_seed(n), dtype=torch.int32).to(DEV) if ragged else None
    for i, c in enumerate(caches):
        before = binding.launch_count()
        c.append_tokens(k, v, n_new)
        assert binding.launch_count() - before == (launches, 3)[i]
    torch.cuda.synchronize()
    a, b = caches
    assert a.sync_status() == 0 and torch.equal(a.bufs.seq_lens, b.bufs.seq_lens)
    assert torch.equal(a.bufs.stats, b.bufs.stats) and torch.equal(a.bufs.tok_lse, b.bufs.tok_lse)
    assert parity.rel_l2(a.bufs.rla_state.cpu().numpy(), b.bufs.rla_state.cpu().numpy()) < 2 * parity.STATE_TOL_FMA


@pytest.mark.parametrize("outlier", [1.0, 10.0])
@pytest.mark.parametrize("n,times", [(40, 1), (100, 1), (255, 1), (200, 10)])
def test_state_below_256_tokens_is_no_less_exact_than_the_fp32_kernels(n, times, outlier):
    """Against 64 bits; phi enters the products with all its bits, and no sum is longer than a tile."""
    errs = []
    for flags in (0, binding.SPLA_GENERAL_KERNELS):
        w = synth.Workload("case", 9, batch=2, n_q_heads=4, n_kv_heads=4, head_dim=128, block_size=64, top_k=8, context=n * times)
        cache = binding.SplaCache(runner.config_for(w, flags=flags), DEV)
        g = torch.Generator(device=DEV).manual_seed(6)
        state = torch.zeros(2, 4, 128, 128, dtype=torch.float64, device=DEV)
        for _ in range(times):
            k, v = (torch.randn(2, 4, n, 128, generator=g, device=DEV) for _ in range(2))
            k[..., :4] *= outlier
            k, v = k.to(torch.bfloat16), v.to(torch.bfloat16)
            cache.append_tokens(k, v)
            state += torch.softmax(k.double(), dim=-1).transpose(-1, -2) @ v.double()
        errs.append(((cache.bufs.rla_state.double() - state).norm() / state.norm()).item())
    assert errs[0] <= errs[1], errs


@pytest.mark.parametrize("dtype,d,batch,hkv,sizes,ragged", [
    ("f32", 64, 1, 1, [33, 255, 257], False),       # one share, the last token of it, two; 16 rows per CTA
    ("f32", 64, 2, 2, [256 * 74 + 31], False),      # as many shares as the workspace holds, ragged at their end
    ("bf16", 64, 2, 2, [40, 700], True),            # shares sized by the longest: some of a short sequence are empty
    ("f32", 128, 3, 20, [300, 770], True),          # two shares, 16 rows per CTA; four, all rows
    ("bf16", 64, 40, 4, [513], False),              # all rows and one share, more units than SMs
    ("f32", 128, 38, 4, [255, 40], False),          # ... d = 128, twice onto the state in place
    ("bf16", 128, 75, 4, [33, 47], True),           # a few tokens of many sequences of different lengths
])
def test_state_of_the_three_kernel_append(dtype, d, batch, hkv, sizes, ragged):
    """S_bar against 64 bits at the edges of staged tokens and of shares; the tolerance of fp32 sums."""
    w = synth.Workload("case", 10, batch=batch, n_q_heads=hkv, n_kv_heads=hkv, head_dim=d, block_size=64, top_k=8,
                       context=sum(sizes), kv_dtype=dtype)
    cache = binding.SplaCache(runner.config_for(w), DEV)
    g = torch.Generator(device=DEV).manual_seed(8)
    state = torch.zeros(batch, hkv, d, d, dtype=torch.float64, device=DEV)
    for n in sizes:
        k, v = (torch.randn(batch, hkv, n, d, generator=g, device=DEV).to(w.torch_dtype) for _ in range(2))
        n_new = torch.randint(0, n + 1, (batch,), generator=torch.Generator().manual_seed(n), dtype=torch.int32).to(DEV) if ragged else None
        cache.append_tokens(k, v, n_new)
        phi = torch.softmax(k.double(), dim=-1)
        if ragged:
            phi = phi * (torch.arange(n, device=DEV)[None, :] < n_new[:, None])[:, None, :, None]
        state += phi.transpose(-1, -2) @ v.double()
    torch.cuda.synchronize()
    assert cache.sync_status() == 0
    err = (cache.bufs.rla_state.double() - state).flatten(2).norm(dim=-1) / state.flatten(2).norm(dim=-1).clamp_min(1e-30)
    assert err.max().item() < parity.STATE_TOL_FMA
