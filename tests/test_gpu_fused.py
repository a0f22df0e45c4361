"""Fused statistics + forward launch: identical results with and without the
fusion, no device errors in normal runs, and the bounded wait: forward items
whose statistics are never published give up after about a second, set the
error flag (read back on the host) and leave the context usable."""

import time

import numpy as np
import pytest
import torch

import oracle as O
from paper_2609_33437_gb300 import smat as S
from paper_2609_33437_gb300 import workloads as W

from _parity import run_and_check_full, session_for, to_host

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")


def _rel_list():
    specs = [W.TensorSpec(f"t{i}", (n,), "linear" if i % 2 else "other", 0.7 if i % 2 else 1.0, 0.0, 0.1)
             for i, n in enumerate([70_001, 262_144 * 3 + 5, 17, 600_000, 4096])]
    specs.append(W.TensorSpec("fixed", (300_003,), "linear", 0.5, 1e-3, 0.0))
    return W.Workload("rel_mix", specs, O.BF16, O.BF16, 0.3, 1.0, 1, O.NOISE_GAUSSIAN, 0.02, 3e-4, seed=11)


@pytest.mark.parametrize("chunk_log2", [0, 18])
def test_fused_and_unfused_give_identical_outputs(chunk_log2):
    w = _rel_list()
    dev = torch.device("cuda")
    th, t0, sim_a, gs, go = W.generate(w, device=dev)
    sim_b = [torch.empty_like(x) for x in sim_a]
    chunk = S.SMAT_FLAG_CHUNK_LOG2(chunk_log2) if chunk_log2 else 0
    a = session_for(w, th, t0, sim_a, flags=chunk)
    b = S.SmatSession(th, t0, sim_b, [t.keep_prob for t in w.tensors], [t.sigma for t in w.tensors],
                      [t.sigma_rel for t in w.tensors], seed=w.seed, alpha_min=w.alpha_min, alpha_max=w.alpha_max,
                      alpha_mode=w.alpha_mode, noise=w.noise, flags=S.SMAT_FLAG_UNFUSED_STATS | chunk)
    for step in (0, 3):
        a.simulate_multi(step)
        b.simulate_multi(step)
        torch.cuda.synchronize()
        for x, y in zip(sim_a, sim_b):
            assert torch.equal(x.view(torch.int16), y.view(torch.int16))
    assert a.poll_errors() == 0 and b.poll_errors() == 0


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("noise,alpha_mode", [(S.SMAT_NOISE_GAUSSIAN, S.SMAT_ALPHA_PER_TENSOR),
                                              (S.SMAT_NOISE_UNIFORM, S.SMAT_ALPHA_PER_ELEMENT),
                                              (S.SMAT_NOISE_LAPLACE, S.SMAT_ALPHA_GLOBAL)])
def test_work_list_walked_and_one_cta_per_item_equal(dtype, noise, alpha_mode):
    """The work list is walked by CTAs that take several items, or has a CTA per
    item, by its length against the resident CTAs (a round at two, three or four
    per SM): lists of 0.1 to 2.4 rounds, on both sides of each line, some with
    a tensor of fixed sigma and in place, equal the separate passes bit for bit."""
    bits = torch.int16 if dtype == torch.bfloat16 else torch.int32
    for sizes, inplace in (([100_003], False), ([500_009], False), ([2_000_003, 33], False), ([2_000_003], True),
                           ([3_000_017], False), ([5_000_011], False), ([9_000_011, 17, 70_001], False)):
        th = [(torch.randn(n, device="cuda") * 0.02).to(dtype) for n in sizes]
        t0 = [(t.float() + torch.randn(t.numel(), device="cuda") * 1e-3).to(dtype) for t in th]
        rel = [0.1 if n != 70_001 else 0.0 for n in sizes]
        got = []
        for flags in (0, S.SMAT_FLAG_UNFUSED_STATS):
            base = [t.clone() for t in t0]
            sim = base if inplace else [torch.empty_like(t) for t in th]
            sess = S.SmatSession(th, base, sim, [0.7] * len(sizes), [1e-3] * len(sizes), rel, seed=9, alpha_min=0.2,
                                 alpha_mode=alpha_mode, noise=noise, flags=flags)
            sess.simulate_multi(2)
            torch.cuda.synchronize()
            assert sess.poll_errors() == 0
            got.append(sim)
            sess.close()
        for a, b in zip(*got):
            assert torch.equal(a.view(bits), b.view(bits)), sizes


@pytest.mark.parametrize("chunk_log2", [0, 18])
def test_fused_list_matches_oracle_and_reports_no_errors(chunk_log2):
    run_and_check_full(_rel_list(), steps=(0, 1, 5), flags=S.SMAT_FLAG_CHUNK_LOG2(chunk_log2) if chunk_log2 else 0)


def test_bounded_wait_runs_out_and_reports():
    w = _rel_list()
    dev = torch.device("cuda")
    th, t0, sim, gs, go = W.generate(w, device=dev)
    sess = session_for(w, th, t0, sim)
    sess.simulate_multi(0)
    assert sess.poll_errors() == 0
    # one forward item of tensor 0 (a sigma_rel tensor), its chunk 0; no statistics item publishes it
    items = torch.tensor([np.int32(np.uint32(0x80000000).view(np.int32))], dtype=torch.int32, device=dev)
    t = time.perf_counter()
    sess.debug_fused(1, items, epoch_skew=1000)
    err = sess.poll_errors()
    dt = time.perf_counter() - t
    assert err == 1, err
    assert dt < 30.0
    assert sess.poll_errors() == 0  # cleared
    # the context still works afterwards
    sess.simulate_multi(2)
    assert sess.poll_errors() == 0
    sess2 = session_for(w, th, t0, [torch.empty_like(x) for x in sim])
    sess2.simulate_multi(2)
    torch.cuda.synchronize()
    assert all(torch.equal(x.view(torch.int16), y.view(torch.int16)) for x, y in zip(sim, sess2._keep[2]))


@pytest.mark.parametrize("noise", [S.SMAT_NOISE_UNIFORM, S.SMAT_NOISE_GAUSSIAN, S.SMAT_NOISE_LAPLACE])
@pytest.mark.parametrize("alpha_mode", [S.SMAT_ALPHA_GLOBAL, S.SMAT_ALPHA_PER_TENSOR, S.SMAT_ALPHA_PER_ELEMENT])
@pytest.mark.parametrize("draw_bits", [32, 16])
def test_list_without_statistics_equals_the_grid_stride_forward(noise, alpha_mode, draw_bits):
    """A list without sigma_rel tensors runs one launch per dtype that draws the
    scalars itself; theta~ and the mapped gradients equal, bit for bit, those of
    the separate scalars launch and grid-stride forward, over both dtypes in one
    list, empty tensors, sizes around a group and a chunk, an offset, sigma 0, and
    in place."""
    sizes = [0, 1, 15, 16, 4097, 70_001, 16, 0, 131_072 + 5]
    dts = [torch.bfloat16, torch.float32]
    th = [(torch.randn(n, device="cuda") * 0.02).to(dts[k % 2]) for k, n in enumerate(sizes)]
    t0 = [(t.float() + torch.randn(t.numel(), device="cuda") * 1e-3).to(t.dtype) for t in th]
    gs = [torch.randn(n, device="cuda") for n in sizes]
    keep = [0.5, 0.7, 1.0, 0.3, 0.9, 0.7, 0.0, 0.5, 0.3]
    sigma = [1e-3, 1e-3, 0.0, 2e-3, 1e-3, 1e-4, 1e-3, 0.0, 1e-3]
    got = []
    for flags, inplace in ((0, False), (S.SMAT_FLAG_UNFUSED_STATS, False), (0, True), (S.SMAT_FLAG_CHUNK_LOG2(16), False)):
        base = [t.clone() for t in t0]
        sim = base if inplace else [torch.empty_like(t) for t in th]
        sess = S.SmatSession(th, base, sim, keep, sigma, seed=21, alpha_min=0.2, alpha_mode=alpha_mode, noise=noise,
                             flags=flags, draw_bits=draw_bits, elem_offsets=[16 * k for k in range(len(sizes))])
        for step in (1, 4):
            if inplace and step > 1:
                for s, t in zip(sim, t0):
                    s.copy_(t)
                sess.mark_theta0_resident()
            sess.simulate_multi(step)
        out = [torch.empty_like(g) for g in gs]
        sess.grad_map_multi(4, gs, out)
        torch.cuda.synchronize()
        got.append([x.view(torch.int16 if x.dtype == torch.bfloat16 else torch.int32) for x in sim + out])
        sess.close()
    for other in got[1:]:
        for k, (a, b) in enumerate(zip(got[0], other)):
            assert torch.equal(a, b), k
