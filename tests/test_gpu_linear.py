"""sbd_linear (y = x W^T on the LM-head kernel, used to time full forwards
around the block step) against the oracle's fp64 product: every element
within bf16 output rounding plus the fp32 accumulation bound."""
import numpy as np
import pytest

import gen
import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sbd():
    import paper_2509_04185_gb300 as m
    return m


def _bf16(rng, shape, scale):
    return gen.f32_to_bf16_bits((rng.standard_normal(shape) * scale).astype(np.float32))


@pytest.mark.parametrize("T,K,N", [(1, 4096, 6144), (5, 64, 1), (16, 256, 129), (17, 256, 1000),
                                   (64, 4096, 128), (100, 512, 777), (128, 1024, 2048),
                                   (200, 256, 300), (256, 4096, 4096), (300, 128, 129),
                                   (512, 256, 1000),
                                   # few rows, narrow layers: K split over CTAs
                                   (16, 4096, 4096), (2, 14336, 512), (64, 1024, 300),
                                   # above 160 rows: CTA pairs (one or two row
                                   # groups; narrow layers with K ranges)
                                   (161, 64, 1), (193, 64, 1), (257, 128, 513), (384, 1024, 257),
                                   (512, 4096, 6144), (512, 14336, 4096), (256, 14336, 512),
                                   (320, 4096, 4096)])
def test_matches_fp64_product(sbd, T, K, N):
    import torch
    rng = np.random.default_rng(T * 7 + N)
    xb, wb = _bf16(rng, (T, K), 1.0), _bf16(rng, (N, K), 0.02)
    x = torch.from_numpy(xb.view(np.int16)).view(torch.bfloat16).cuda()
    w = torch.from_numpy(wb.view(np.int16)).view(torch.bfloat16).cuda()
    y = sbd.sbd_linear(x, w).float().cpu().numpy()
    xf, wf = gen.bf16_bits_to_f32(xb), gen.bf16_bits_to_f32(wb)
    ref = oracle.linear(xf, wf)
    bound = np.abs(xf).astype(np.float64) @ np.abs(wf).astype(np.float64).T
    tol = 2.0 ** -8 * np.abs(ref) + K * 2.0 ** -23 * bound + 1e-6
    assert y.shape == (T, N)
    assert np.all(np.abs(y - ref) <= tol), float(np.max(np.abs(y - ref) - tol))
    assert sbd.sbd_device_error() == 0


@pytest.mark.parametrize("T,K,N", [
    # up to 160 rows: K ranges of a tile in one cluster, 2 to 8 of them, of unequal length, outputs that
    # end inside a group of four; one range where the tiles fill the SMs
    (1, 64 * 37, 700), (16, 64 * 33, 1030), (33, 64 * 8, 5), (160, 64 * 9, 130), (160, 64 * 67, 4099),
    (128, 64 * 21, 6145), (7, 64 * 16, 9730), (16, 64 * 5, 20000),
    # CTA pairs: unit widths from 2 x 128 down, with and without K ranges; a second row group of one row
    (161, 64 * 40, 6144), (200, 64 * 12, 4096), (256, 64 * 64, 2050), (257, 64 * 16, 9001),
    (385, 64 * 8, 4096), (512, 64 * 32, 6144), (512, 64 * 3, 28672)])
def test_split_and_unit_edges(sbd, T, K, N):
    import torch
    g = torch.Generator(device="cuda").manual_seed(T + N)
    x = torch.randn(T, K, generator=g, device="cuda").to(torch.bfloat16)
    w = (torch.randn(N, K, generator=g, device="cuda") * 0.02).to(torch.bfloat16)
    y = torch.full((T + 1, N), 7.0, dtype=torch.bfloat16, device="cuda")
    sbd.sbd_linear(x, w, out=y[:T])
    ref = x.double() @ w.double().T
    # half a unit in the last place of the output, plus K fp32 additions of the products
    bound = x.double().abs() @ w.double().abs().T
    tol = 2.0 ** -8 * ref.abs() + K * 2.0 ** -23 * bound + 1e-6
    assert bool(((y[:T].double() - ref).abs() <= tol).all())
    assert bool((y[T] == 7.0).all())
    assert sbd.sbd_device_error() == 0


@pytest.mark.parametrize("T,K,N", [
    # rows of outputs, or of fp32 partials, that start on 16 bytes but not on 32, on 8 and on 2
    (161, 512, 1000), (300, 512, 1000), (512, 512, 1000), (161, 1024, 100), (257, 1024, 100), (200, 2048, 1004),
    (512, 64, 24), (161, 2048, 1002), (384, 2048, 1001),
    # up to 160 rows: 16, 8, 4 and 2 K ranges through the workspace, fewer and more outputs than are summed
    # four at a time, and a count that four does not divide
    (1, 4096, 1024), (160, 4096, 1024), (128, 8192, 2048), (64, 2048, 2048), (33, 2048, 2049), (100, 8192, 2050),
    (160, 4096, 28672), (96, 4096, 2048), (5, 64 * 12, 20001)])
def test_store_widths_and_range_sums(sbd, T, K, N):
    test_split_and_unit_edges(sbd, T, K, N)


def test_out_of_range_rows_are_not_written(sbd):
    import torch
    rng = np.random.default_rng(1)
    x = torch.from_numpy(_bf16(rng, (3, 128), 1.0).view(np.int16)).view(torch.bfloat16).cuda()
    w = torch.from_numpy(_bf16(rng, (200, 128), 0.1).view(np.int16)).view(torch.bfloat16).cuda()
    big = torch.full((5, 200), 7.0, dtype=torch.bfloat16, device="cuda")
    sbd.sbd_linear(x, w, out=big[:3])
    assert torch.all(big[3:] == 7.0)


@pytest.mark.parametrize("case", range(16))
def test_random_shapes(sbd, case):
    """Seeded random shapes on both sides of the CTA-pair threshold (160
    rows): out_features that leave partial tiles, in_features of any number
    of 64-column boxes (K split where the model picks one)."""
    import torch
    rng = np.random.default_rng(500 + case)
    T = int(rng.integers(1, 513))
    K = 64 * int(rng.integers(1, 65))
    N = int(rng.integers(1, 3000))
    xb, wb = _bf16(rng, (T, K), 1.0), _bf16(rng, (N, K), 0.02)
    x = torch.from_numpy(xb.view(np.int16)).view(torch.bfloat16).cuda()
    w = torch.from_numpy(wb.view(np.int16)).view(torch.bfloat16).cuda()
    y = sbd.sbd_linear(x, w).float().cpu().numpy()
    xf, wf = gen.bf16_bits_to_f32(xb), gen.bf16_bits_to_f32(wb)
    ref = oracle.linear(xf, wf)
    bound = np.abs(xf).astype(np.float64) @ np.abs(wf).astype(np.float64).T
    tol = 2.0 ** -8 * np.abs(ref) + K * 2.0 ** -23 * bound + 1e-6
    assert np.all(np.abs(y - ref) <= tol), (T, K, N, float(np.max(np.abs(y - ref) - tol)))
    assert sbd.sbd_device_error() == 0


def test_threads_with_different_row_counts(sbd):
    """One kernel serves up to 160 rows, with shared memory by the row count:
    host threads that launch it at the same time, each on its own stream, must
    not take each other's away."""
    import threading
    import torch
    K, N = 64, 256
    w = torch.randn(N, K, device="cuda").to(torch.bfloat16)
    rows = [1, 160, 33, 96]
    streams = [torch.cuda.Stream() for _ in rows]
    xs = [torch.randn(r, K, device="cuda").to(torch.bfloat16) for r in rows]
    ys = [torch.empty(r, N, dtype=torch.bfloat16, device="cuda") for r in rows]
    calls = [sbd.prepare_linear(x, w, y, stream=s) for x, y, s in zip(xs, ys, streams)]
    torch.cuda.synchronize()
    errors = []

    def go(call):
        try:
            for _ in range(3000):
                call()
        except Exception as e:            # the launch's status
            errors.append(e)

    ts = [threading.Thread(target=go, args=(c,)) for c in calls]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    torch.cuda.synchronize()
    assert not errors, errors[0]
    for x, y in zip(xs, ys):
        ref, bound = x.double() @ w.double().T, x.double().abs() @ w.double().abs().T
        # half a unit in the last place of the output, plus K fp32 additions of the products
        assert bool(((y.double() - ref).abs() <= 2.0 ** -8 * ref.abs() + K * 2.0 ** -23 * bound + 1e-6).all())
    assert sbd.sbd_device_error() == 0
