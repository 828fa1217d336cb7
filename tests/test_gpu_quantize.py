"""GPU parity: stage-1 kernels against the oracle, bit for bit (codes, block scales, tensor
scales, means, compensation vector, V codes), through the C ABI."""
import numpy as np
import pytest
import torch

from oracle import mpfa_oracle as orc
from paper_2609_33135_b200 import workloads as wl

from layouts import codes_to_logical, pad128, sf_to_logical

pytestmark = pytest.mark.gpu


def _cases():
    return {
        "cfg1": lambda: wl.config1_tiny(),
        "cfg1b": lambda: wl.config1b_tiny_qbias(),
        "ragged_gqa": lambda: wl.prefill_workload("ragged", 41, 2, 333, 4, 2, True, N_q=300, q_bias=True),
        "gqa5_2k": lambda: wl.prefill_workload("gqa5", 42, 1, 2048 + 77, 10, 2, True, q_bias=True),
    }


def run_stage1_gpu(w, smooth=True, v_scale=1.0):
    from paper_2609_33135_b200 import binding
    return binding.stage1(w.q.cuda(), w.k.cuda(), w.v.cuda(), smooth=smooth, v_scale=v_scale)


def check_stage1(w, s1, z, smooth=True):
    B, Nq, Hq, Nkv, Hkv = w.B, w.N_q, w.H_q, w.N_kv, w.H_kv
    torch.cuda.synchronize()
    assert np.array_equal(s1.stats.q_mean.cpu().numpy(), z.q_mean)
    assert np.array_equal(s1.stats.k_mean.cpu().numpy(), z.k_mean)
    assert np.array_equal(s1.stats.q_gscale.cpu().numpy(), z.dq)
    assert np.array_equal(s1.stats.k_gscale.cpu().numpy(), z.dk)
    for t, codes, sf, H, N in ((s1.q, z.q_codes, z.q_sf, Hq, Nq), (s1.k, z.k_codes, z.k_sf, Hkv, Nkv)):
        got, padrows = codes_to_logical(t.codes.cpu().numpy(), B, H, N)
        assert np.array_equal(got, codes)
        assert not padrows.any()
        gsf = sf_to_logical(t.sf.cpu().numpy(), B, H, N)
        assert np.array_equal(gsf[:, :, :N], sf)
        assert not gsf[:, :, N:].any()
    gv = s1.v_fp8.cpu().numpy().reshape(B, Hkv, pad128(Nkv), 128)
    assert np.array_equal(gv[:, :, :Nkv], z.v_codes)
    assert not gv[:, :, Nkv:].any()
    if smooth:
        gd = s1.delta.view(torch.uint16).cpu().numpy()
        assert np.array_equal(gd[:, :, :Nkv], z.delta)
        assert not gd[:, :, Nkv:].any()
    else:
        assert s1.delta is None


@pytest.mark.parametrize("name", list(_cases()))
def test_stage1_bit_exact(name):
    w = _cases()[name]()
    z = orc.stage1(orc.bf16_bits(w.q), orc.bf16_bits(w.k), orc.bf16_bits(w.v))
    check_stage1(w, run_stage1_gpu(w), z)


@pytest.mark.parametrize("B,N,N_q,H_q,H_kv", [
    (1, 1, 1, 1, 1), (1, 129, 7, 3, 1), (2, 127, 9, 2, 2), (1, 128, 128, 8, 1),   # smallest, few query rows, one tile
    (1, 1024, 1024, 12, 2), (1, 1031, 1500, 7, 1),                                  # statistics in two slices, groups of six and seven
    (1, 4099, 4099, 40, 8), (3, 2500, 700, 32, 8),                                  # several tiles per CTA, ragged last tile
    (7, 1300, 1, 40, 8), (19, 260, 130, 8, 8),                                      # more heads than CTAs in a wave
])
def test_stage1_bit_exact_over_tile_and_slice_counts(B, N, N_q, H_q, H_kv):
    w = wl.prefill_workload("edges", 44, B, N, H_q, H_kv, True, N_q=N_q, q_bias=True)
    z = orc.stage1(orc.bf16_bits(w.q), orc.bf16_bits(w.k), orc.bf16_bits(w.v))
    check_stage1(w, run_stage1_gpu(w), z)


def test_stage1_with_more_heads_than_a_grid_dimension():
    """65538 heads of Q and K in one call (a launch's second and third dimensions end at 65535)."""
    from paper_2609_33135_b200 import binding
    H = 32769
    g = torch.Generator(device="cuda").manual_seed(9)
    q, k, v = (torch.randn(1, 2, H, 128, generator=g, device="cuda").bfloat16() for _ in range(3))
    ws = torch.empty(binding.lib().mpfa_quantize_workspace_min_bytes(1, H, H), dtype=torch.uint8, device="cuda")
    s1 = binding.stage1(q, k, v, workspace=ws)
    for x, mean in ((q, s1.stats.q_mean), (k, s1.stats.k_mean)):
        assert torch.equal(mean, x.double().mean(1).float())
    m = (k.float() - s1.stats.k_mean[:, None]).abs().max()
    assert s1.stats.k_gscale.cpu().numpy()[0] == np.float32(m.item()) / np.float32(2688.0)


def test_stage1_from_inputs_on_16_byte_boundaries():
    """The interface asks for 16-byte alignment; 32-byte aligned inputs take wider loads."""
    from paper_2609_33135_b200 import binding
    w = _cases()["ragged_gqa"]()
    z = orc.stage1(orc.bf16_bits(w.q), orc.bf16_bits(w.k), orc.bf16_bits(w.v))

    def shifted(x):
        raw = torch.empty(x.numel() + 8, dtype=x.dtype, device="cuda")
        y = raw[8:].view(x.shape).copy_(x)
        assert y.data_ptr() % 32 == 16
        return y
    check_stage1(w, binding.stage1(shifted(w.q), shifted(w.k), shifted(w.v)), z)


def test_statistics_on_any_float_boundary():
    """The interface asks for no alignment of the statistics: stage 1, a query with frozen statistics, a page write and an append
    with every array four bytes past a 16-byte boundary give what they give with aligned ones."""
    from paper_2609_33135_b200 import binding
    w = wl.prefill_workload("shifted", 46, 1, 333, 10, 2, True, q_bias=True)
    q, k, v = w.q.cuda(), w.k.cuda(), w.v.cuda()
    frozen = binding.MPFA_SMOOTH | binding.MPFA_STATS_FROZEN

    def run(shift):
        def arr(*shape):
            n = int(np.prod(shape))
            t = torch.zeros(n + 4, dtype=torch.float32, device="cuda")[shift:shift + n].view(*shape)
            assert t.data_ptr() % 16 == 4 * shift
            return t
        st = binding.Stats(arr(1, 10, 128), arr(1, 2, 128), arr(1), arr(1))
        s1 = binding.stage1(q, k, v)
        s1.stats = st
        binding.stage1(q, k, v, out=s1)
        q4 = binding.Fp4Tensor.empty(1, 10, 1)
        binding.mpfa_quantize_qk(q[:, 9:10].contiguous(), None, frozen, st, q4, None, None, None)
        kv = binding.PagedKV.empty(6, 10, 2)
        for t in (kv.k_codes, kv.k_sf, kv.v_fp8, kv.delta):
            t.zero_()
        row = torch.arange(6, dtype=torch.int32, device="cuda").view(1, 6)
        binding.mpfa_quantize_kv_paged(k[0, :300].contiguous(), v[0, :300].contiguous(), 0, 10, binding.MPFA_SMOOTH, st, 1.0, kv, row[0],
                                       binding.quantize_workspace(1, 10, 2))
        binding.mpfa_append_kv_paged(k[:, 300:301].contiguous(), v[:, 300:301].contiguous(), 10, frozen, st, 1.0, kv, row,
                                     torch.tensor([300], dtype=torch.int32, device="cuda"))
        return [s1.q.codes, s1.q.sf, s1.k.codes, s1.k.sf, s1.delta.view(torch.int16), st.q_mean, st.k_mean, st.q_gscale, st.k_gscale, q4.codes,
                q4.sf, kv.k_codes, kv.k_sf, kv.v_fp8, kv.delta.view(torch.int16)]
    want = run(0)
    for shift in (1, 2, 3):
        for a, b in zip(run(shift), want):
            assert torch.equal(a, b)


def test_means_of_columns_with_non_finite_values():
    """The statistics add bit patterns of finite values; a column that holds an infinity or a NaN still gets the mean that a
    plain sum gives, and its neighbours theirs."""
    from paper_2609_33135_b200 import binding
    w = wl.prefill_workload("inf", 45, 1, 700, 2, 1, True)
    ref = run_stage1_gpu(w).stats.q_mean.clone()
    q = w.q.clone()
    q[0, 5, 0, 3], q[0, 600, 0, 4], q[0, 9, 1, 100], q[0, 10, 1, 100] = float("inf"), float("nan"), float("inf"), float("-inf")
    m = binding.stage1(q.cuda(), w.k.cuda(), w.v.cuda()).stats.q_mean.cpu()[0]
    assert m[0, 3] == float("inf") and torch.isnan(m[0, 4]) and torch.isnan(m[1, 100])
    m[0, 3], m[0, 4], m[1, 100] = ref[0, 0, 3], ref[0, 0, 4], ref[0, 1, 100]
    assert torch.equal(m, ref.cpu()[0])


def test_stage1_direct_variant_and_v_scale():
    w = _cases()["ragged_gqa"]()
    z = orc.stage1(orc.bf16_bits(w.q), orc.bf16_bits(w.k), orc.bf16_bits(w.v), smooth=False, v_scale=0.5)
    s1 = run_stage1_gpu(w, smooth=False, v_scale=0.5)
    check_stage1(w, s1, z, smooth=False)
    assert not s1.stats.q_mean.any() and not s1.stats.k_mean.any()


def test_frozen_statistics_single_token_query():
    """Decode-time query: one token centered and scaled with the frozen prefill statistics."""
    from paper_2609_33135_b200 import binding
    w = _cases()["ragged_gqa"]()
    z = orc.stage1(orc.bf16_bits(w.q), orc.bf16_bits(w.k), orc.bf16_bits(w.v))
    s1 = run_stage1_gpu(w)
    qn = w.q[:, 17:18].contiguous()
    zq = orc.stage1(orc.bf16_bits(qn), orc.bf16_bits(w.k), orc.bf16_bits(w.v), frozen=z)
    q4 = binding.Fp4Tensor.empty(w.B, w.H_q, 1)
    binding.mpfa_quantize_qk(qn.cuda(), None, binding.MPFA_SMOOTH | binding.MPFA_STATS_FROZEN, s1.stats, q4, None,
                             None, None)
    torch.cuda.synchronize()
    got, pad = codes_to_logical(q4.codes.cpu().numpy(), w.B, w.H_q, 1)
    assert np.array_equal(got, zq.q_codes) and not pad.any()
    assert np.array_equal(sf_to_logical(q4.sf.cpu().numpy(), w.B, w.H_q, 1)[:, :, :1], zq.q_sf)


def _rows_by_both_paths(x, gscale):
    """Codes and scale bytes of eight tokens x [1, 8, H, 128] with given statistics, from the kernel of at most eight queries and, as
    the first rows of sixteen, from the tile kernel; and K codes and scale bytes of the same tokens from the page kernel and, one
    by one, from the append kernel."""
    from paper_2609_33135_b200 import binding
    H = x.shape[2]
    st = binding.Stats.empty(1, H, H)
    g = torch.Generator().manual_seed(5)
    for m in (st.q_mean, st.k_mean):
        m.copy_(torch.randn(1, H, 128, generator=g) * 0.25)
    st.q_gscale.fill_(gscale), st.k_gscale.fill_(gscale)
    x = x.cuda()
    rows = []
    for q in (x, torch.cat([x, x.flip(1)], 1).contiguous()):
        q4 = binding.Fp4Tensor.empty(1, H, q.shape[1])
        binding.mpfa_quantize_qk(q, None, binding.MPFA_STATS_FROZEN, st, q4, None, None, None)
        rows.append((codes_to_logical(q4.codes.cpu().numpy(), 1, H, q.shape[1])[0][:, :, :8],
                     sf_to_logical(q4.sf.cpu().numpy(), 1, H, q.shape[1])[:, :, :8]))
    pages = []
    table = torch.zeros(1, 1, dtype=torch.int32, device="cuda")
    for one_by_one in (False, True):
        kv = binding.PagedKV.empty(1, H, H, with_delta=False)
        if one_by_one:
            for t in range(8):
                k = x[:, t:t + 1].contiguous()
                binding.mpfa_append_kv_paged(k, k, H, 0, st, 1.0, kv, table, torch.tensor([t], dtype=torch.int32, device="cuda"))
        else:
            binding.mpfa_quantize_kv_paged(x[0].contiguous(), x[0].contiguous(), 0, H, binding.MPFA_STATS_FROZEN, st, 1.0, kv, table[0], None)
        pages.append((kv.k_codes.cpu().numpy(), kv.k_sf.cpu().numpy()))
    torch.cuda.synchronize()
    return rows, pages


@pytest.mark.parametrize("value", [float("nan"), float("inf"), float("-inf")])
def test_blocks_without_a_finite_value(value):
    """A block of 16 NaNs has scale 0 on every path, so that it does not turn its token's scores into NaNs; an infinity saturates."""
    x = torch.randn(1, 8, 2, 128, generator=torch.Generator().manual_seed(6))
    x[0, 3, 0, 32:48] = value
    x[0, 5, 1] = value
    x[0, 6, 1, 7] = value
    (few, tile), (page, one) = _rows_by_both_paths(x.bfloat16(), 0.003)
    assert (few[1][0, 0, 3, 2], few[1][0, 1, 5, 4]) == ((0, 0) if np.isnan(value) else (0x7E, 0x7E))
    for a, b in ((few, tile), (page, one)):
        assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])


@pytest.mark.parametrize("gscale", [-0.003, -0.0, 0.0, 1e-38, 3e-31, 1e30, float("inf"), float("nan")])
def test_frozen_tensor_scales_of_any_value(gscale):
    """The caller's frozen scale is taken as it is.  A negative one gives scale codes with the sign bit, beyond the 128 entries of
    the tile kernel's table of reciprocals; outside 1e-30 .. 1e30 the scale code is divided out."""
    x = torch.randn(1, 8, 2, 128, generator=torch.Generator().manual_seed(7))
    x[0, 2, 1, 16:32] = 0.0
    (few, tile), (page, one) = _rows_by_both_paths(x.bfloat16(), gscale)
    for a, b in ((few, tile), (page, one)):
        assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])


def test_deterministic_and_argument_errors():
    from paper_2609_33135_b200 import binding
    w = _cases()["cfg1b"]()
    a = run_stage1_gpu(w)
    b = run_stage1_gpu(w)
    torch.cuda.synchronize()
    assert torch.equal(a.q.codes, b.q.codes) and torch.equal(a.k.sf, b.k.sf) and torch.equal(a.delta, b.delta)
    q = w.q.cuda()
    st = binding.Stats.empty(1, 1, 1)
    q4 = binding.Fp4Tensor.empty(1, 1, 256)
    ws = binding.quantize_workspace(1, 1, 1)
    with pytest.raises(binding.MpfaError, match="workspace"):
        binding.mpfa_quantize_qk(q, None, 0, st, q4, None, None, ws[:256])
    with pytest.raises(binding.MpfaError, match="misaligned"):
        bad = binding.Fp4Tensor(q4.codes[16:], q4.sf, 1, 1, 255)
        binding.mpfa_quantize_qk(q[:, :255].contiguous(), None, 0, st, bad, None, None, ws)
    with pytest.raises(binding.MpfaError, match="invalid"):
        binding.mpfa_quantize_qk(q, None, 0, st, binding.Fp4Tensor(q4.codes, q4.sf, 1, 1, 128), None, None, ws)


def _adversarial(kind: str, seed: int):
    """Small tensors with the values that break sloppy quantizers: hand-built, not drawn from the workload recipe."""
    import dataclasses
    g = torch.Generator().manual_seed(seed)
    B, N, Hq, Hkv = 2, 300, 4, 2
    q = torch.randn(B, N, Hq, 128, generator=g)
    k = torch.randn(B, N, Hkv, 128, generator=g)
    v = torch.randn(B, N, Hkv, 128, generator=g)
    if kind == "zeros":                 # an all-zero batch element (tensor scale 1) next to an ordinary one
        q[0].zero_(); k[0].zero_(); v[0].zero_()
    elif kind == "zero_blocks":         # blocks and whole heads of zeros inside a non-zero tensor, negative zeros
        k[:, :, 0, :].zero_(); q[:, :, 1, 32:48] = 0.0; q[:, ::2, 2, :] = -0.0; v[:, 5:9] = -0.0
    elif kind == "dynamic_range":       # 2^-120 .. 2^100 in one tensor: scales underflow to 0 and saturate at 448
        e = torch.randint(-120, 100, (B, N, Hkv, 128), generator=g).float()
        k = k.sign() * torch.exp2(e)
        q = q * 1e-30
        v = v * 1e30
    elif kind == "ties":                # values on the E2M1 and E4M3 rounding boundaries after scaling
        grid = torch.tensor([0.25, 0.75, 1.25, 1.75, 2.5, 3.5, 5.0, 6.0, 0.5, 1.0, 1.5, 2.0, 3.0, 4.0, 0.0, 7.0])
        idx = torch.randint(0, 16, (B, N, Hkv, 128), generator=g)
        k = grid[idx] * k.sign()
        k[:, 0, :, 0] = 6.0 * 448.0 / 448.0
        q = (torch.randint(-8, 9, (B, N, Hq, 128), generator=g).float()) * 0.25
        v = torch.randint(-32, 33, (B, N, Hkv, 128), generator=g).float() * 0.0625 + 448.0 * (torch.rand(B, N, Hkv, 128, generator=g) < 0.01)
    elif kind == "constant":            # every token identical: centered values are exactly zero
        q = q[:, :1].expand(B, N, Hq, 128).clone(); k = k[:, :1].expand(B, N, Hkv, 128).clone()
    w = wl.prefill_workload("adv", 1, B, N, Hq, Hkv, True)
    return dataclasses.replace(w, q=q.to(torch.bfloat16), k=k.to(torch.bfloat16), v=v.to(torch.bfloat16))


@pytest.mark.parametrize("kind", ["zeros", "zero_blocks", "dynamic_range", "ties", "constant"])
def test_stage1_bit_exact_on_adversarial_values(kind):
    w = _adversarial(kind, 400 + len(kind))
    z = orc.stage1(orc.bf16_bits(w.q), orc.bf16_bits(w.k), orc.bf16_bits(w.v))
    check_stage1(w, run_stage1_gpu(w), z)


def test_means_are_deterministic_on_unflushed_inputs():
    """Eq. 7 on inputs the seeded generator never produces: magnitudes from 2^-60 up to O(1) mixed in every column,
    so the FP64 column sums are no longer exact and their value depends on the order of addition.  The kernels add
    in a fixed order (no floating-point atomics): two runs must agree bit for bit in every output, and the means
    must be within one FP32 ulp of the oracle's single ascending sum."""
    from paper_2609_33135_b200 import binding
    g = torch.Generator(device="cpu").manual_seed(77)
    B, N, Hq, Hkv = 2, 3000, 4, 2
    def draw(H):
        x = torch.randn(B, N, H, 128, generator=g)
        e = torch.randint(-60, 1, (B, N, H, 128), generator=g).float()
        return (x * torch.exp2(e)).to(torch.bfloat16)
    q, k, v = draw(Hq), draw(Hkv), draw(Hkv)
    assert float(q.float().abs()[q.float().abs() > 0].min()) < 2.0 ** -55
    runs = []
    for _ in range(2):
        s1 = binding.stage1(q.cuda(), k.cuda(), v.cuda())
        torch.cuda.synchronize()
        runs.append([t.clone() for t in (s1.stats.q_mean, s1.stats.k_mean, s1.stats.q_gscale, s1.stats.k_gscale, s1.q.codes,
                                         s1.q.sf, s1.k.codes, s1.k.sf, s1.delta.view(torch.uint16))])
    for a, b in zip(*runs):
        assert torch.equal(a, b)
    for got, x in ((runs[0][0], q), (runs[0][1], k)):
        ref = orc.means(orc.bf16_bits(x))
        got = got.cpu().numpy()
        ulp = np.spacing(np.abs(ref).astype(np.float32))
        assert np.all(np.abs(got.astype(np.float64) - ref.astype(np.float64)) <= ulp)
        assert (got == ref).mean() > 0.99


def test_stage1_with_a_one_slice_workspace_is_the_same_on_exact_inputs():
    """The statistics pass takes as many token slices as the workspace holds; on the generator's inputs (exact
    sums) the slice count cannot change a bit."""
    from paper_2609_33135_b200 import binding
    w = wl.prefill_workload("ws", 43, 1, 2500, 4, 2, True, q_bias=True)
    z = orc.stage1(orc.bf16_bits(w.q), orc.bf16_bits(w.k), orc.bf16_bits(w.v))
    n_min = binding.lib().mpfa_quantize_workspace_min_bytes(1, 4, 2)
    assert n_min < binding.lib().mpfa_quantize_workspace_bytes(1, 4, 2)
    for nbytes in (n_min, 3 * n_min):
        ws = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
        check_stage1(w, binding.stage1(w.q.cuda(), w.k.cuda(), w.v.cuda(), workspace=ws), z)
    with pytest.raises(binding.MpfaError, match="workspace"):
        binding.stage1(w.q.cuda(), w.k.cuda(), w.v.cuda(), workspace=torch.empty(n_min - 256, dtype=torch.uint8, device="cuda"))


def test_a_workspace_for_two_slices_is_used_as_two():
    """Sums of one column that depend on the slices: 2^60, then at the start of the second half -2^60 and 1 in the same lane.  In one
    slice the two large values cancel first and the mean is 1 / 1024, in two the 1 is lost beside -2^60 and the mean is 0."""
    from paper_2609_33135_b200 import binding
    L = binding.lib()
    n_min, n_full = L.mpfa_quantize_workspace_min_bytes(1, 1, 1), L.mpfa_quantize_workspace_bytes(1, 1, 1)
    per = (n_full - n_min) // 31
    x = torch.zeros(1, 1024, 1, 128)
    x[0, 0, 0, 5], x[0, 512, 0, 5], x[0, 528, 0, 5] = 2.0 ** 60, -2.0 ** 60, 1.0
    x = x.bfloat16().cuda()
    for nbytes, mean in ((n_min, 1.0 / 1024), (n_min + per - 256, 1.0 / 1024), (n_min + per, 0.0), (n_full, 0.0)):
        s1 = binding.stage1(x, x, x, workspace=torch.empty(nbytes, dtype=torch.uint8, device="cuda"))
        assert float(s1.stats.q_mean[0, 0, 5]) == mean and float(s1.stats.k_mean[0, 0, 5]) == mean, nbytes


@pytest.mark.parametrize("B,N_q,N,Hq,Hkv", [
    (1, 129, 129, 1, 1),          # two CTAs of a cluster, one row in the last tile
    (3, 1, 1025, 2, 1),           # a head with one token: seven slices of its cluster are empty
    (1, 2049, 2049, 2, 1),        # clusters of sixteen
    (1, 10240, 10240, 1, 1), (1, 10241, 10241, 1, 1),   # the longest that a cluster takes, and one more
    (2, 1281, 1281, 8, 2),        # clusters of eight
    (5, 300, 300, 12, 12),        # more heads than clusters of four fit
    (37, 257, 257, 4, 4),         # one CTA per head
])
def test_stage1_in_one_call_around_the_rule_for_clusters(B, N_q, N, Hq, Hkv):
    """Statistics by clusters, slices and single CTAs, V's tiles behind them: bit for bit the oracle's, and what the two calls give."""
    from paper_2609_33135_b200 import binding
    w = wl.prefill_workload("clusters", 57, B, N, Hq, Hkv, False, N_q=N_q, q_bias=True)
    q, k, v = w.q.cuda(), w.k.cuda(), w.v.cuda()
    s1 = binding.stage1(q, k, v, v_scale=0.5)
    check_stage1(w, binding.stage1(q, k, v), orc.stage1(orc.bf16_bits(w.q), orc.bf16_bits(w.k), orc.bf16_bits(w.v)))
    one = [t.clone() for t in (s1.q.codes, s1.q.sf, s1.k.codes, s1.k.sf, s1.v_fp8, s1.delta.view(torch.uint8))]
    for frozen in (0, binding.MPFA_STATS_FROZEN):
        for t in (s1.q.codes, s1.q.sf, s1.k.codes, s1.k.sf, s1.v_fp8, s1.delta.view(torch.uint8)):
            t.fill_(0xA5)
        ws = None if frozen else binding.quantize_workspace(B, Hq, Hkv)
        if frozen:
            binding.mpfa_quantize_qkv(q, k, v, binding.MPFA_SMOOTH | frozen, 0.5, s1.stats, s1.q, s1.k, s1.v_fp8, s1.delta, ws)
        else:
            binding.mpfa_quantize_qk(q, k, binding.MPFA_SMOOTH, s1.stats, s1.q, s1.k, s1.delta, ws)
            binding.mpfa_quantize_v(v, 0.5, s1.v_fp8)
        for t, u in zip((s1.q.codes, s1.q.sf, s1.k.codes, s1.k.sf, s1.v_fp8, s1.delta.view(torch.uint8)), one):
            assert torch.equal(t, u)


@pytest.mark.parametrize("B,N,Hq,Hkv", [(1, 129, 1, 1), (1, 2049, 2, 1), (2, 1281, 8, 2), (1, 10240, 1, 1)])   # clusters of 2, 16, 8, 16
def test_stage1_by_clusters_without_smoothing_and_from_a_graph(B, N, Hq, Hkv):
    """Statistics by clusters where no mean is subtracted, and both forms replayed from a graph on other inputs than it was captured with."""
    from paper_2609_33135_b200 import binding
    w, other = (wl.prefill_workload("clusters", seed, B, N, Hq, Hkv, False, q_bias=True) for seed in (58, 59))
    for smooth in (False, True):
        z = orc.stage1(orc.bf16_bits(w.q), orc.bf16_bits(w.k), orc.bf16_bits(w.v), smooth=smooth)
        check_stage1(w, run_stage1_gpu(w, smooth=smooth), z, smooth=smooth)
        q, k, v = other.q.cuda(), other.k.cuda(), other.v.cuda()
        ws = binding.quantize_workspace(B, Hq, Hkv)
        s1 = binding.stage1(q, k, v, smooth=smooth, workspace=ws)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            binding.stage1(q, k, v, smooth=smooth, workspace=ws, out=s1)
        for t, x in ((q, w.q), (k, w.k), (v, w.v)):
            t.copy_(x)
        graph.replay()
        check_stage1(w, s1, z, smooth=smooth)
