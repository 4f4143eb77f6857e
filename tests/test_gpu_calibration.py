"""GPU parity of the n-sigma bound (Section 3.2.2) against the oracle's sort-and-pick definition:
the radix select must return the same integer for every input, duplicates, negatives and
extremes included."""
import numpy as np
import pytest
import torch

from oracle import planner as P
from paper_2006_11735_b200 import binding as B

pytestmark = pytest.mark.gpu


def _bound(Y, frac, offset=0):
    """Runs the library on a device copy of Y placed `offset` elements into its buffer."""
    buf = torch.empty(Y.size + offset + 3, dtype=torch.int32, device="cuda")
    buf[offset:offset + Y.size] = torch.from_numpy(Y.reshape(-1)).cuda()
    got = B.iq_sigma_bound(buf.data_ptr() + 4 * offset, Y.size, frac, torch.cuda.current_stream().cuda_stream)
    B.iconv_check(torch.cuda.current_stream().cuda_stream)
    return got


@pytest.mark.parametrize("size", [1, 2, 7, 1000, 4099, 1 << 20, 20_000_003])
@pytest.mark.parametrize("frac", [0.0015, 0.00023, 0.5, 1.0])
def test_sigma_bound_matches_oracle_on_normal_feature_maps(size, frac):
    rng = np.random.default_rng(size % 9973 + int(frac * 1e6))
    Y = np.floor(rng.normal(-2000.0, 90000.0, size=size) + 0.5).astype(np.int32)
    want = P.sigma_bound(Y, frac)
    for offset in (0, 1, 3):                     # the 16-byte fast path starts at every alignment
        assert _bound(Y, frac, offset) == want


def test_sigma_bound_degenerate_inputs():
    cases = [
        np.full(100_000, 77, dtype=np.int32),                                          # every value equal
        np.full(5000, -5, dtype=np.int32),                                             # all negative: clamped to 1
        np.array([np.iinfo(np.int32).min, np.iinfo(np.int32).max, 0, -1, 1] * 2000, dtype=np.int32),
        np.repeat(np.arange(-50, 50, dtype=np.int32), 3000),                           # heavy duplicates
        (np.arange(300_000, dtype=np.int64) * 7919 % 1_000_003 - 500_000).astype(np.int32),   # all distinct
        np.random.default_rng(3).integers(-2 ** 31, 2 ** 31, size=700_001, dtype=np.int64).astype(np.int32),   # full range
    ]
    for Y in cases:
        for frac in (0.0015, 0.01, 0.999):
            assert _bound(Y, frac) == P.sigma_bound(Y, frac)
    assert B.iq_sigma_bound(None, 0) == 1
    with pytest.raises(B.IconvError):
        B.iq_sigma_bound(torch.zeros(4, dtype=torch.int32, device="cuda").data_ptr() + 1, 2)    # misaligned


@pytest.mark.parametrize("size", [8192, 8193, 3_000_001])
@pytest.mark.parametrize("kind", ["mass_at_bound", "mass_inside", "outliers", "two_values", "ascending"])
def test_sigma_bound_where_the_sampled_bracket_is_awkward(kind, size):
    """The edge of the directly selected size, a value that fills a bracket's end or its inside by itself (the
    lists overflow), a sampled range that outliers widen, ranks at both ends."""
    rng = np.random.default_rng(size)
    Y = np.floor(rng.normal(0.0, 90000.0, size=size) + 0.5).astype(np.int32)
    if kind == "mass_at_bound":
        Y = np.minimum(Y, 200000)
    elif kind == "mass_inside":
        Y[rng.random(size) < 0.2] = 150000
    elif kind == "outliers":
        Y[:4] = [2 ** 31 - 1, -2 ** 31, 2 ** 31 - 2, -2 ** 31 + 1]
    elif kind == "two_values":
        Y = np.where(Y > 0, 7, 3).astype(np.int32)
    else:
        Y = np.sort(Y)
    for frac in (0.0015, 0.02, 0.19, 0.5, 1.0, 1e-7):
        assert _bound(Y, frac, 1) == P.sigma_bound(Y, frac), (kind, frac)


@pytest.mark.parametrize("size", [8193, 1_000_003])
@pytest.mark.parametrize("sampled_high", [False, True])
def test_sigma_bound_where_the_sample_misleads(size, sampled_high):
    """All keys that the bracket is taken from lie on one side of the wanted one: the rank is outside the
    bracket, and the radix select has to answer."""
    h = (np.arange(8192, dtype=np.uint64) + 1) * 0x9E3779B9 & 0xffffffff          # the kernel's positions
    for shift, mul in ((16, 0x85EBCA6B), (13, 0xC2B2AE35), (16, 1)):
        h = (h ^ h >> np.uint64(shift)) * mul & 0xffffffff
    at = np.unique(h * np.uint64(size) >> np.uint64(32)).astype(np.int64)
    rng = np.random.default_rng(size)
    Y = rng.integers(-1000, 1000, size=size).astype(np.int32)
    Y[at] = rng.integers(-9000, -8000, size=at.size) if not sampled_high else rng.integers(8000, 9000, size=at.size)
    rest = size - at.size
    for k in (max(1, rest // 3), rest // 2) if not sampled_high else (at.size + rest // 2, at.size + 2 * rest // 3 + 1):
        frac = (k - 0.5) / size
        assert _bound(Y, frac, 1) == P.sigma_bound(Y, frac) == max(1, int(np.sort(Y)[size - k]))


@pytest.mark.parametrize("size", [3_000_000, 8_000_003])
def test_sigma_bound_where_few_warps_meet_the_largest_values(size):
    """Each of them meets more than 384 keys of the bracket, the others hardly any: the blocks' lists are of very different lengths, and
    most lanes of a few warps go through their queues."""
    rng = np.random.default_rng(size)
    Y = np.sort(np.floor(rng.normal(0.0, 90000.0, size=size) + 0.5).astype(np.int32))
    warp = (np.arange(size) // 4 % (444 * 512)) // 32                   # of a tensor at a 16-byte boundary, 444 blocks of 512
    few = np.flatnonzero(warp % 263 == 7)                               # 27 warps, whole: 0.38 % of the tensor
    few = few[:few.size - few.size % 16]
    assert 0.0036 < few.size / size < 0.0042 and np.bincount(warp[few]).max() > 400
    out = np.empty_like(Y)
    mask = np.zeros(size, dtype=bool)
    mask[few] = True
    out[mask] = rng.permutation(Y[size - few.size:])
    out[~mask] = rng.permutation(Y[:size - few.size])
    assert _bound(out, 0.0015) == P.sigma_bound(out, 0.0015)


@pytest.mark.parametrize("trips", [1, 2])
@pytest.mark.parametrize("extra", [-130, -1, 0, 1, 4 * 512 + 7])
def test_sigma_bound_at_the_edges_of_the_one_pass(trips, extra):
    """Around whole rounds of the pass's grid (444 blocks of 512 threads, four vectors of four values each): what is left
    for the last, partial round.  From few lanes with a value of the bracket (its queue drains at the end only) to every lane."""
    size = trips * 444 * 512 * 16 + extra
    rng = np.random.default_rng(size % 9973)
    Y = np.floor(rng.normal(0.0, 90000.0, size=size) + 0.5).astype(np.int32)
    srt = np.sort(Y)
    for frac in (2e-6, 0.0015, 0.06):
        k = max(1, int(np.ceil(size * frac)))
        assert _bound(Y, frac) == max(1, int(srt[size - k]))
    Y[-5:] = 2 ** 31 - 1                         # the wanted key among the last values that are read
    assert _bound(Y, 3.5 / size, 1) == 2 ** 31 - 1


def test_sigma_bound_where_a_blocks_list_overflows():
    """The largest values lie where two blocks of the one pass read: each meets more keys of the bracket than its list
    holds (6144), and the radix select has to answer."""
    size = 8_000_003
    rng = np.random.default_rng(size)
    Y = np.sort(np.floor(rng.normal(0.0, 90000.0, size=size) + 0.5).astype(np.int32))
    block = (np.arange(size) // 4 % (444 * 512)) // 512                 # of a tensor at a 16-byte boundary, 444 blocks of 512
    few = np.flatnonzero((block == 5) | (block == 300))
    few = few[:int(0.0038 * size)]
    assert np.bincount(block[few]).max() > 2 * 6144
    out = np.empty_like(Y)
    mask = np.zeros(size, dtype=bool)
    mask[few] = True
    out[mask] = rng.permutation(Y[size - few.size:])
    out[~mask] = rng.permutation(Y[:size - few.size])
    assert _bound(out, 0.0015) == P.sigma_bound(out, 0.0015)


@pytest.mark.parametrize("spread", [1, 300, 40_000, 2 ** 30])
@pytest.mark.parametrize("frac", [0.0015, 0.004, 0.012])
def test_sigma_bound_with_brackets_of_every_width(spread, frac):
    """Kept keys of one value to thirty bits (the upper nine are histogrammed by the pass, the rest takes no round to two),
    lists longer than the 480 keys that are held in registers."""
    rng = np.random.default_rng(spread % 9973)
    Y = np.minimum(np.floor(rng.exponential(spread, size=40_000_001)), 2.0 ** 31 - 1).astype(np.int32)
    k = int(np.ceil(Y.size * frac))
    assert _bound(Y, frac) == max(1, int(np.partition(Y, Y.size - k)[Y.size - k]))


def test_the_scratch_is_given_back():
    Y = np.arange(100_000, dtype=np.int32)
    _bound(Y, 0.01)
    B.iq_release_scratch()
    free = torch.cuda.mem_get_info()[0]
    for _ in range(3):
        assert _bound(Y, 0.01) == P.sigma_bound(Y, 0.01)
    assert 10 << 20 <= free - torch.cuda.mem_get_info()[0] <= 16 << 20          # one scratch, whatever the calls
    B.iq_release_scratch()
    assert torch.cuda.mem_get_info()[0] == free
    assert _bound(Y, 0.01) == P.sigma_bound(Y, 0.01)


def test_sigma_bound_where_memory_is_scarce():
    """Too little for the scratch of the one-pass selection: the radix select needs 2 KB."""
    rng = np.random.default_rng(8)
    Y = np.floor(rng.normal(0.0, 90000.0, size=1_000_001) + 0.5).astype(np.int32)
    y = torch.from_numpy(Y).cuda()
    stream = torch.cuda.current_stream().cuda_stream
    for frac in (0.0015, 0.5):                   # (every kernel has been loaded once)
        assert B.iq_sigma_bound(y.data_ptr(), Y.size, frac, stream) == P.sigma_bound(Y, frac)
    torch.cuda.empty_cache()
    B.iq_release_scratch()
    try:
        rest = torch.empty((torch.cuda.mem_get_info()[0] - (8 << 20),), dtype=torch.uint8, device="cuda")
    except torch.cuda.OutOfMemoryError:
        pytest.skip("the device's memory cannot be filled to within 8 MB")
    assert torch.cuda.mem_get_info()[0] < 10 << 20
    for frac in (0.0015, 0.5):
        assert B.iq_sigma_bound(y.data_ptr(), Y.size, frac, stream) == P.sigma_bound(Y, frac)
    del rest
    torch.cuda.empty_cache()
    B.iconv_check(stream)


def test_sigma_bound_in_a_capture_is_refused_and_leaves_everything_as_it_was():
    Y = np.arange(100_000, dtype=np.int32)
    y, other = torch.from_numpy(Y).cuda(), torch.zeros(4, device="cuda")
    stream, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    want = _bound(Y, 0.01)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    with torch.cuda.graph(graph, stream=stream):
        with pytest.raises(B.IconvError) as e:
            B.iq_sigma_bound(y.data_ptr(), Y.size, 0.01, stream.cuda_stream)
        other.add_(1.0)
    assert e.value.status == B.ERR_CUDA
    graph.replay()
    torch.cuda.synchronize()
    assert other.tolist() == [1.0] * 4 and _bound(Y, 0.01) == want == P.sigma_bound(Y, 0.01)
    assert free - torch.cuda.mem_get_info()[0] < 8 << 20         # (the graph's own memory; a lost scratch would be 12 MB)


def test_sigma_bound_calibrates_a_layer_like_the_oracle():
    """The bound of a raw convolution output computed on the GPU feeds Eq. 9-13 to the same
    mul, shift and h_i as the oracle's calibration of that layer."""
    from gpu_util import gpu_conv, oracle_conv
    rng = np.random.default_rng(17)
    X = rng.integers(0, 256, size=(2, 40, 44, 64), dtype=np.uint8)
    W = np.clip(np.floor(rng.normal(0, 40, size=(64, 3, 3, 64)) + 0.5), -127, 127).astype(np.int8)
    b = rng.integers(-4096, 4097, size=(64,), dtype=np.int32)
    Yo = oracle_conv(X, W, b, [1], [0], [0], pad=1, out_dtype=B.I32, brelu=False)
    Yg, _ = gpu_conv(X, W, b, [1], [0], [0], pad=1, out_dtype=B.I32, brelu=False)
    assert np.array_equal(Yg, Yo)
    h_ri = _bound(Yg.astype(np.int32), 0.0015)
    assert h_ri == P.sigma_bound(Yo)
    assert B.iq_brelu_params(float(h_ri), 1.0, 255) == {k: v for k, v in P.brelu_params(float(h_ri), 1.0, 255).items()}


def test_batch_norm_folded_per_channel_layer_end_to_end():
    """A float convolution + batch normalisation + ReLU-like clamp becomes an integer layer with
    one quantisation step per output channel (Section 3.4.3) and per-channel mul / shift / h_i
    from Algorithm 2 with every channel a branch; the GPU equals the oracle bit for bit and the
    dequantised result tracks the float layer."""
    from gpu_util import gpu_conv, oracle_conv
    rng = np.random.default_rng(33)
    n, h, w, c_in, c_out, k, max_int, h_rf = 2, 20, 24, 32, 48, 3, 255, 4.0
    x_f = rng.uniform(0.0, 1.0, size=(n, h, w, c_in))
    ratio_X = 255.0
    X = np.floor(x_f * ratio_X + 0.5).astype(np.uint8)
    W_f = rng.normal(0, 0.08, size=(c_out, k, k, c_in)).astype(np.float32)
    gamma = rng.uniform(0.05, 3.0, size=c_out).astype(np.float32)          # steps differing 60-fold between channels
    beta = rng.normal(0, 0.2, size=c_out).astype(np.float32)
    mean = rng.normal(0, 0.3, size=c_out).astype(np.float32)
    var = rng.uniform(0.2, 2.0, size=c_out).astype(np.float32)
    Wp, bp, delta = B.iq_bn_fold(W_f, None, gamma, beta, mean, var, 1e-5)
    assert delta.max() / delta.min() > 10
    ratio_Y = [ratio_X / d for d in delta]
    ratio_V = [P.brelu_params(h_rf, ry, max_int)["ratio_V"] for ry in ratio_Y]
    sync = P.concat_sync(ratio_Y, ratio_V)                                   # Algorithm 2, one branch per channel
    got_plan = B.iconcat_plan(ratio_Y, ratio_V)
    assert list(got_plan["mul"]) == list(sync["mul"]) and list(got_plan["shift"]) == list(sync["shift"])
    Wq = np.stack([P.quantize_weights(Wp[c], delta[c] * sync["delta_scale"][c]) for c in range(c_out)])
    b_i = np.array([P.round_half_up(bp[c] * sync["ratio_Y_new"][c]) for c in range(c_out)], dtype=np.int32)
    mul = np.array(sync["mul"], dtype=np.int32)
    shift = np.array(sync["shift"], dtype=np.int32)
    h_i = np.array([P.round_half_up(P.Fraction(max_int * (1 << int(s)), int(m))) for m, s in zip(mul, shift)], dtype=np.int32)
    want = oracle_conv(X, Wq, b_i, mul, shift, h_i, pad=1)
    for kernel in (B.KERNEL_AUTO, B.KERNEL_UMMA_IM2COL, B.KERNEL_DIRECT):
        got, _ = gpu_conv(X, Wq, b_i, mul, shift, h_i, pad=1, kernel=kernel)
        assert np.array_equal(got, want)
    # the float layer: convolution, batch normalisation, clamp to [0, h_f]
    xp = np.pad(x_f, ((0, 0), (1, 1), (1, 1), (0, 0)))
    y = np.zeros((n, h, w, c_out))
    for r in range(k):
        for s in range(k):
            y += xp[:, r:r + h, s:s + w, :] @ W_f[:, r, s, :].astype(np.float64).T
    y = (y - mean) / np.sqrt(var.astype(np.float64) + 1e-5) * gamma + beta
    h_f = max_int / sync["ratio_V_min"]
    y = np.clip(y, 0.0, h_f)
    err = np.abs(want.astype(np.float64) / sync["ratio_V_min"] - y)
    assert err.mean() < 0.02 * h_f and (want > 0).mean() > 0.2 and (want == max_int).mean() < 0.5
