"""Merge kernels (the evaluation side, Eq. merged-state): WA, TA, DARE + TA and
TIES over K experts, bit-identical to the CPU oracle on ragged lists (vector
and element paths), including the TIES trim thresholds, in place, with DARE
ties and element offsets, and on inputs with many equal magnitudes."""

import numpy as np
import pytest
import torch

import oracle as O
from paper_2609_33437_gb300 import smat as S

from _parity import f32_of, to_host

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")


METHODS = {S.SMAT_MERGE_WA: O.MERGE_WA, S.SMAT_MERGE_TA: O.MERGE_TA, S.SMAT_MERGE_DARE_TA: O.MERGE_DARE_TA,
           S.SMAT_MERGE_TIES: O.MERGE_TIES}


def _experts(sizes, K, dtype, seed, quantum=None):
    g = torch.Generator(device="cuda").manual_seed(seed)
    tdt = torch.bfloat16 if dtype == O.BF16 else torch.float32
    t0s, exs = [], []
    for n in sizes:
        t0 = torch.randn(n, device="cuda", generator=g) * 0.02
        ex = []
        for _ in range(K):
            d = torch.randn(n, device="cuda", generator=g) * 1e-3
            if quantum:
                d = torch.round(d / quantum) * quantum
            ex.append((t0 + d).to(tdt))
        t0s.append(t0.to(tdt))
        exs.append(ex)
    return t0s, exs


def _check(t0s, exs, outs, dtype, method, kw, elem_offsets=None, thr=None):
    K = len(exs[0])
    for k, (t0, ex, out) in enumerate(zip(t0s, exs, outs)):
        ref, rthr = O.merge(METHODS[method], to_host(t0), [to_host(x) for x in ex], dtype=dtype,
                            gamma=kw.get("gamma", 1.0), p_drop=kw.get("p_drop", 0.0),
                            retention=kw.get("retention", 1.0), seed=kw.get("seed", 0), tensor_id=k,
                            elem_offset=0 if elem_offsets is None else elem_offsets[k])
        got = to_host(out)
        view = np.uint16 if dtype == O.BF16 else np.uint32
        assert np.array_equal(got.view(view), ref.view(view)), f"tensor {k}"
        if thr is not None:
            nan = np.uint32(0x7F800001)  # the first of the NaN keys, which all stand for one threshold
            got_thr = np.minimum(thr[k].cpu().numpy().view(np.uint32), nan)
            assert np.array_equal(got_thr, np.minimum(rthr, nan)), f"tensor {k} thresholds"


SIZES = [1, 15, 16, 17, 4096, 65_536 + 33, 131_073]


@pytest.mark.parametrize("method", list(METHODS))
@pytest.mark.parametrize("dtype", [O.F32, O.BF16])
def test_merge_matches_oracle(method, dtype):
    K = 5
    t0s, exs = _experts(SIZES, K, dtype, seed=100 + method)
    outs = [torch.empty_like(t) for t in t0s]
    kw = dict(gamma=0.7, p_drop=0.3, retention=0.3, seed=99)  # p_drop 0.3: threshold with low bits (ties)
    thr = S.merge(t0s, exs, outs, method, return_thresholds=method == S.SMAT_MERGE_TIES, **kw)
    torch.cuda.synchronize()
    _check(t0s, exs, outs, dtype, method, kw, thr=thr)


@pytest.mark.parametrize("method", list(METHODS))
def test_merge_in_place_equals_out_of_place(method):
    t0s, exs = _experts([70_001, 4096 + 5], 3, O.BF16, seed=7)
    kw = dict(gamma=0.5, p_drop=0.5, retention=0.5, seed=3)
    outs = [torch.empty_like(t) for t in t0s]
    S.merge(t0s, exs, outs, method, **kw)
    inplace = [t.clone() for t in t0s]
    S.merge(inplace, exs, inplace, method, **kw)
    torch.cuda.synchronize()
    for a, b in zip(outs, inplace):
        assert torch.equal(a.view(torch.int16), b.view(torch.int16))


@pytest.mark.parametrize("method", [S.SMAT_MERGE_DARE_TA, S.SMAT_MERGE_TIES])
def test_merge_element_path_and_offsets(method):
    """Unaligned pointers take the element path; elem_offset keys the DARE
    masks like a shard of a larger tensor."""
    n, K = 33_333, 4
    t0s, exs = _experts([n + 3], K, O.F32, seed=11)
    base, ex_base = t0s[0], exs[0]
    t0 = base[3:]
    ex = [x[3:] for x in ex_base]  # 12-byte offset: not 32-byte aligned
    out = torch.empty(n + 8, device="cuda")[5:5 + n]
    kw = dict(gamma=1.0, p_drop=0.3, retention=0.5, seed=5)
    S.merge([t0], [ex], [out], method, elem_offsets=[1000], **kw)
    torch.cuda.synchronize()
    _check([t0], [ex], [out], O.F32, method, kw, elem_offsets=[1000])


def test_merge_ties_many_equal_magnitudes():
    """Deltas on a coarse grid: thousands of equal |Delta| at the threshold,
    all kept, thresholds equal to the oracle's."""
    t0s, exs = _experts([100_003, 5000], 6, O.F32, seed=13, quantum=5e-4)
    outs = [torch.empty_like(t) for t in t0s]
    kw = dict(gamma=1.0, retention=0.2)
    thr = S.merge(t0s, exs, outs, S.SMAT_MERGE_TIES, return_thresholds=True, **kw)
    torch.cuda.synchronize()
    _check(t0s, exs, outs, O.F32, S.SMAT_MERGE_TIES, kw, thr=thr)


def test_merge_argument_errors():
    t0s, exs = _experts([1000], 2, O.F32, seed=1)
    out = [torch.empty_like(t0s[0])]
    for bad in (dict(p_drop=1.0), dict(retention=0.0), dict(gamma=float("inf")), dict(philox_rounds=8)):
        with pytest.raises(S.SmatError):
            S.merge(t0s, exs, out, S.SMAT_MERGE_DARE_TA, **bad)
    with pytest.raises(S.SmatError):
        S.merge(t0s, [exs[0] * 9], out, S.SMAT_MERGE_TA)  # 18 experts > 16
    with pytest.raises(S.SmatError):
        S.merge(t0s, exs, [exs[0][0]], S.SMAT_MERGE_TA)  # out is an expert
    with pytest.raises(S.SmatError):
        S.merge(t0s + [t0s[0].to(torch.bfloat16)], exs + [[x.to(torch.bfloat16) for x in exs[0]]],
                out + [torch.empty(1000, device="cuda", dtype=torch.bfloat16)], S.SMAT_MERGE_TA)  # two dtypes


def test_merge_dare_seven_rounds():
    """DARE masks with the 7-round stream option equal the oracle's."""
    t0s, exs = _experts([70_001, 4096], 3, O.BF16, seed=17)
    outs = [torch.empty_like(t) for t in t0s]
    S.merge(t0s, exs, outs, S.SMAT_MERGE_DARE_TA, gamma=0.5, p_drop=0.3, seed=8, philox_rounds=7)
    torch.cuda.synchronize()
    for k, (t0, ex, out) in enumerate(zip(t0s, exs, outs)):
        ref, _ = O.merge(O.MERGE_DARE_TA, to_host(t0), [to_host(x) for x in ex], dtype=O.BF16, gamma=0.5,
                         p_drop=0.3, seed=8, tensor_id=k, rounds=7)
        assert np.array_equal(to_host(out).view(np.uint16), ref.view(np.uint16)), k


@pytest.mark.parametrize("K", [1, 2, 8, 9, 15, 16])
def test_merge_dare_expert_counts(K):
    """DARE with one to sixteen experts (the kernel loads experts in batches
    of four, so every remainder occurs) equals the oracle."""
    t0s, exs = _experts([17, 4096, 65_536 + 33], K, O.BF16, seed=40 + K)
    outs = [torch.empty_like(t) for t in t0s]
    kw = dict(gamma=0.6, p_drop=0.3, seed=5)
    S.merge(t0s, exs, outs, S.SMAT_MERGE_DARE_TA, **kw)
    torch.cuda.synchronize()
    _check(t0s, exs, outs, O.BF16, S.SMAT_MERGE_DARE_TA, kw)


@pytest.mark.parametrize("method", list(METHODS))
@pytest.mark.parametrize("dtype", [O.F32, O.BF16])
def test_merge_special_values(method, dtype):
    """Signed zeros, infinities, NaN, subnormals and experts equal to theta0
    sprinkled into theta0 and the experts: every result equals the oracle's
    bit for bit, NaN matching any NaN (payloads differ between host and GPU).
    Retention keeps the TIES thresholds among the finite keys."""
    n, K = 20_000 + 7, 5
    g = torch.Generator().manual_seed(23)
    t0 = torch.randn(n, generator=g) * 0.02
    ex = [t0 + torch.randn(n, generator=g) * 1e-3 for _ in range(K)]
    specials = torch.tensor([0.0, -0.0, float("inf"), float("-inf"), float("nan"), 1e-40, -1e-40, 3e-39])
    for arr in [t0] + ex:
        pos = torch.randint(0, n, (n // 50,), generator=g)
        arr[pos] = specials[torch.randint(0, len(specials), (len(pos),), generator=g)]
    for e in range(K):  # Delta exactly 0 on a few coordinates
        pos = torch.randint(0, n, (n // 100,), generator=g)
        ex[e][pos] = t0[pos]
    tdt = torch.bfloat16 if dtype == O.BF16 else torch.float32
    t0d = t0.to(tdt).cuda()
    exd = [x.to(tdt).cuda() for x in ex]
    out = torch.empty_like(t0d)
    kw = dict(gamma=0.7, p_drop=0.3, retention=0.3, seed=4)
    S.merge([t0d], [exd], [out], method, **kw)
    torch.cuda.synchronize()
    ref, _ = O.merge(METHODS[method], to_host(t0d), [to_host(x) for x in exd], dtype=dtype, tensor_id=0, **kw)
    got = to_host(out)
    gf, rf = f32_of(got), f32_of(ref)
    view = np.uint16 if dtype == O.BF16 else np.uint32
    nan_g, nan_r = np.isnan(gf), np.isnan(rf)
    assert np.array_equal(nan_g, nan_r)
    assert np.array_equal(got.view(view)[~nan_g], ref.view(view)[~nan_r])


@pytest.mark.parametrize("dtype", [O.F32, O.BF16])
@pytest.mark.parametrize("shape", ["normal", "mostly_zero", "sample_low", "sample_high", "infinities", "two_values",
                                   "sample_nan", "sample_half_nan", "half_nan", "all_nan_but_sample"])
@pytest.mark.parametrize("retention", [1e-4, 0.25, 0.5, 1.0])
def test_merge_ties_threshold_selection(dtype, shape, retention):
    """Thresholds of tensors larger than the selection's sample (32,768
    elements, in 16-element groups at 16 floor(g (n / 16) / 2048)) equal the
    oracle's, also where the sample shows other magnitudes than the rest (its
    interval misses, and the next passes start from the whole range), where
    most keys are equal, with infinities, and with NaN in all or half of the
    sample, all over the tensor, or everywhere else (a NaN threshold is any NaN)."""
    n, K = 200_000 + 37, 2
    g = torch.Generator().manual_seed(31)
    t0 = torch.randn(n, generator=g) * 0.02
    d = torch.randn(K, n, generator=g) * 1e-3
    seen = torch.zeros(n, dtype=torch.bool)
    first = 16 * (torch.arange(2048) * (n // 16) // 2048)
    seen[(first[:, None] + torch.arange(16)).reshape(-1)] = True
    if shape == "mostly_zero":
        d[torch.rand(K, n, generator=g) < 0.8] = 0.0
    elif shape == "sample_low":
        d[:, seen] *= 1e-3
    elif shape == "sample_high":
        d[:, seen] *= 1e3
    elif shape == "infinities":
        d[torch.rand(K, n, generator=g) < 0.7] = float("inf")
    elif shape == "two_values":
        d = torch.where(d > 0, 0.25, 0.5)
        t0 = torch.zeros(n)
    elif shape == "sample_nan":
        d[:, seen] = float("nan")
    elif shape == "sample_half_nan":
        d[(torch.rand(K, n, generator=g) < 0.5) & seen] = float("nan")
    elif shape == "half_nan":
        d[torch.rand(K, n, generator=g) < 0.5] = float("nan")
    elif shape == "all_nan_but_sample":
        d[:, ~seen] = float("nan")
    tdt = torch.bfloat16 if dtype == O.BF16 else torch.float32
    t0d = t0.to(tdt).cuda()
    exd = [(t0 + d[e]).to(tdt).cuda() for e in range(K)]
    out = torch.empty_like(t0d)
    kw = dict(gamma=0.7, retention=retention)
    thr = S.merge([t0d], [exd], [out], S.SMAT_MERGE_TIES, return_thresholds=True, **kw)
    torch.cuda.synchronize()
    _check([t0d], [exd], [out], dtype, S.SMAT_MERGE_TIES, kw, thr=thr)


@pytest.mark.parametrize("K", [1, 3, 4, 8, 12, 16])
@pytest.mark.parametrize("dtype", [O.F32, O.BF16])
def test_merge_ties_expert_counts(K, dtype):
    """TIES over one to sixteen experts (the merge pass has builds for batches
    of eight and four and for a remainder; the threshold passes take four at a
    time) equals the oracle, with groups of eight that hold a NaN, infinities of
    one sign and of both."""
    t0s, exs = _experts([17, 4096, 65_536 + 41, 140_000], K, dtype, seed=60 + K)
    for k in (1, 3):
        n = t0s[k].numel()
        exs[k][0][n // 3] = float("nan")
        exs[k][K - 1][n // 5] = float("inf")
        exs[k][0][n // 7] = float("-inf")
        exs[k][K - 1][n // 7] = float("inf")
    outs = [torch.empty_like(t) for t in t0s]
    kw = dict(gamma=0.6, retention=0.4)
    S.merge(t0s, exs, outs, S.SMAT_MERGE_TIES, **kw)
    torch.cuda.synchronize()
    for k, (t0, ex, out) in enumerate(zip(t0s, exs, outs)):
        ref, _ = O.merge(O.MERGE_TIES, to_host(t0), [to_host(x) for x in ex], dtype=dtype, tensor_id=k, **kw)
        got = to_host(out)
        view = np.uint16 if dtype == O.BF16 else np.uint32
        nan_g, nan_r = np.isnan(f32_of(got)), np.isnan(f32_of(ref))
        assert np.array_equal(nan_g, nan_r)
        assert np.array_equal(got.view(view)[~nan_g], ref.view(view)[~nan_r]), k


def test_merge_refuses_mismatched_tensors():
    """The binding's list checks refuse what a tensor-by-tensor check would,
    naming the tensor, and take views, in-place outputs and empty tensors."""
    t0s, exs = _experts([1000, 64, 0, 4096], 3, O.F32, seed=2)
    outs = [torch.empty_like(t) for t in t0s]

    def refused(k, t0=None, ex=None, out=None, error=ValueError):
        a, b, c = list(t0s), [list(e) for e in exs], list(outs)
        a[k] = t0 if t0 is not None else a[k]
        c[k] = out if out is not None else c[k]
        if ex is not None:
            b[k][1] = ex
        with pytest.raises(error) as e:
            S.merge(a, b, c, S.SMAT_MERGE_TA)
        return str(e.value)

    for k in (0, 3):
        n = t0s[k].numel()
        wrong = torch.empty(n + 1, device="cuda")
        other = torch.empty(n, device="cuda", dtype=torch.bfloat16)
        strided = torch.empty(2 * n, device="cuda")[::2]
        for kind in ("t0", "ex", "out"):
            for bad in (wrong, other, strided):
                assert f"tensor {k}" in refused(k, **{kind: bad})
    with pytest.raises(ValueError):
        S.merge(t0s, [exs[0], exs[1][:2], exs[2], exs[3]], outs, S.SMAT_MERGE_TA)
    with pytest.raises(ValueError):
        S.merge(t0s[:3], exs, outs, S.SMAT_MERGE_TA)
    half = [t.half() for t in t0s]
    with pytest.raises(TypeError):
        S.merge(half, [[x.half() for x in e] for e in exs], [t.half() for t in outs], S.SMAT_MERGE_TA)
    with pytest.raises(S.SmatError):
        S.merge(t0s, [[] for _ in exs], outs, S.SMAT_MERGE_TA)
    with pytest.raises(S.SmatError):
        S.merge([], [], [], S.SMAT_MERGE_TA)  # no tensor, so no expert either
    S.merge(t0s, exs, outs, S.SMAT_MERGE_TA, gamma=0.5, tensor_ids=[7, 5, 3, 1], elem_offsets=[0, 16, 0, 1 << 40])
    flat = torch.cat([t.reshape(-1) for t in t0s])
    at, views = 0, []
    for t in t0s:
        views.append(flat[at:at + t.numel()])
        at += t.numel()
    S.merge(views, exs, views, S.SMAT_MERGE_TA, gamma=0.5)
    for a, b in zip(outs, views):
        assert torch.equal(a, b)


@pytest.mark.parametrize("dtype", [O.F32, O.BF16])
@pytest.mark.parametrize("K", [2, 5])
def test_merge_ties_long_threshold_items(dtype, K):
    """The threshold passes' items are as long as fill whole rounds of the CTAs
    (here no power of two), the merge pass's chunks are not: the thresholds and
    the merge equal the oracle's on several tensors, one of them unaligned."""
    t0s, exs = _experts([3_000_017, 40_000, 2_500_003 + 1], K, dtype, seed=90 + K)
    t0s[2], exs[2] = t0s[2][1:], [x[1:] for x in exs[2]]
    outs = [torch.empty_like(t) for t in t0s]
    kw = dict(gamma=0.4, retention=0.2)
    thr = S.merge(t0s, exs, outs, S.SMAT_MERGE_TIES, return_thresholds=True, **kw)
    torch.cuda.synchronize()
    _check(t0s, exs, outs, dtype, S.SMAT_MERGE_TIES, kw, thr=thr)


@pytest.mark.parametrize("method", list(METHODS))
@pytest.mark.parametrize("sizes", [[35_000_011], [200_003] * 170])
def test_merge_returns_before_the_work_ahead_of_it(method, sizes):
    """smat_merge is asynchronous: it returns while earlier work of the stream
    still runs (no table of the call is long enough for its upload to wait), and
    its tables are its own by then: the merge is the same."""
    t0s, exs = _experts(sizes, 2, O.F32, seed=3)
    outs = [torch.empty_like(t) for t in t0s]
    kw = dict(gamma=0.4, retention=0.3, p_drop=0.3 if method == S.SMAT_MERGE_DARE_TA else 0.0)
    S.merge(t0s, exs, outs, method, **kw)  # the workspace's first allocation
    first = [x.clone() for x in outs]
    for x in outs:
        x.zero_()
    torch.cuda.synchronize()
    ahead = torch.cuda.Event()
    torch.cuda._sleep(200_000_000)  # about 0.1 s
    ahead.record()
    S.merge(t0s, exs, outs, method, **kw)
    assert not ahead.query()
    torch.cuda.synchronize()
    assert all(torch.equal(a, b) for a, b in zip(first, outs))
