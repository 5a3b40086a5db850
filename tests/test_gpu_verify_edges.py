"""Verification where rows start and end inside 16-byte vectors, at the borders between the warps that share a row, and
on both sides of the size up to which one kernel does the whole job.  Integer results: compared exactly."""
import numpy as np
import pytest
import torch

import oracle
from paper_2404_19124_b200 import synth
from helpers import kernels_launched, ws_view

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    from paper_2404_19124_b200 import build
    build.build()
    from paper_2404_19124_b200 import binding
    return binding


def _check(B, cand, logits):
    Bn, K, n = cand.shape
    bf16 = logits.dtype == torch.bfloat16
    host = logits.cpu().contiguous()
    acc, best, nxt, ws = B.spec_verify(cand.cuda(), logits)
    o = oracle.verify(cand.numpy(), synth.bf16_bits(host) if bf16 else host.numpy(), oracle.BF16 if bf16 else oracle.F32,
                      want_g=True)
    assert B.spec_poll_error(ws) == 0
    g = ws_view(ws, 256, Bn * K * (n + 1), torch.int32).cpu().numpy().reshape(Bn, K, n + 1)
    assert np.array_equal(g, o[3])
    for got, want in zip((acc, best, nxt), o):
        assert np.array_equal(got.cpu().numpy(), want)


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("shape", [(5, 11, 3, 32003), (2, 4, 2, 8191), (1, 3, 1, 65537), (3, 7, 2, 9), (4, 5, 3, 17),
                                   (2, 30, 1, 1093), (70, 2, 1, 4001), (1, 2, 3, 8192), (1, 2, 3, 8193), (1, 1000, 2, 21),
                                   (1, 1334, 2, 5)])
def test_rows_that_are_not_whole_vectors(B, shape, dtype):
    """Random rows, one planted maximum each at the places where a partial vector, a warp's range or the row begins or
    ends, and for every third row a second equal maximum further right (the first must win)."""
    Bn, K, n, V = shape
    g = torch.Generator().manual_seed(V)
    x = torch.randn(Bn, K, n + 1, V, generator=g).to(dtype)
    rows = x.view(-1, V)
    epv = 8 if dtype == torch.bfloat16 else 4
    for r in range(rows.shape[0]):
        start = r * V
        places = [0, V - 1, min(V - 1, -start % epv), max(0, V - 1 - (start + V) % epv), r * 37 % V, V // 2]
        p = places[r % len(places)]
        rows[r, p] = 9.0
        if r % 3 == 0:
            rows[r, p + (V - 1 - p) // 2:][-1] = 9.0
    cand = torch.randint(0, V, (Bn, K, n), generator=g, dtype=torch.int64).to(torch.int32)
    am = x.float().argmax(-1)
    for k in range(K):
        cand[:, k, :k % (n + 1)] = am[:, k, :k % (n + 1)].to(torch.int32)
    _check(B, cand, x.cuda())


@pytest.mark.parametrize("shape,dtype,kernels", [((148, 2, 1, 8192), torch.bfloat16, 1), ((149, 2, 1, 8192), torch.bfloat16, 2),
                                                 ((149, 3, 2, 512), torch.bfloat16, 1), ((149, 3, 2, 513), torch.bfloat16, 2),
                                                 ((296, 2, 1, 256), torch.float32, 1), ((296, 2, 1, 257), torch.float32, 2),
                                                 ((1332, 2, 1, 64), torch.bfloat16, 1), ((1333, 2, 1, 64), torch.bfloat16, 2)])
def test_many_short_sequences(B, shape, dtype, kernels):
    """More sequences than SMs: one kernel only while the turns they take are few for the length of a row."""
    Bn, K, n, V = shape
    g = torch.Generator().manual_seed(V)
    x = torch.randn(Bn, K, n + 1, V, generator=g).to(dtype)
    cand = torch.randint(0, V, (Bn, K, n), generator=g, dtype=torch.int64).to(torch.int32)
    am = x.float().argmax(-1).to(torch.int32)
    cand[::2, -1] = am[::2, -1, :n]
    _check(B, cand, x.cuda())
    cand, x = cand.cuda(), x.cuda()
    out = [torch.empty(Bn, dtype=torch.int32, device="cuda") for _ in range(3)]
    ws = torch.empty(B.spec_verify_workspace_bytes(*shape, B.SPEC_BF16 if dtype == torch.bfloat16 else B.SPEC_F32),
                     dtype=torch.uint8, device="cuda")
    assert kernels_launched(lambda: B.spec_verify(cand, x, *out, workspace=ws)) == kernels


@pytest.mark.parametrize("V", [1000, 30001])
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
def test_every_alignment_of_the_base(B, V, dtype):
    Bn, K, n = 2, 3, 2
    g = torch.Generator().manual_seed(V)
    size = Bn * K * (n + 1) * V
    buf = torch.randn(size + 8, generator=g).to(dtype).cuda()
    cand = torch.randint(0, V, (Bn, K, n), generator=g, dtype=torch.int64).to(torch.int32)
    for off in range(8 if dtype == torch.bfloat16 else 4):
        buf[:off] = 50.0                                  # what lies before and behind the tensor must not be seen
        buf[off + size:] = 50.0
        _check(B, cand, buf[off:off + size].view(Bn, K, n + 1, V))


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("rows,vectors,extra,off", [(130, 3072, 0, 0), (130, 3072, -1, 0), (130, 3072, -1, 3), (131, 3072, 1, 1),
                                                    (131, 3079, 2, 2), (26, 16032, 0, 0), (26, 16032, 3, 3), (26, 16032, -3, 1),
                                                    (148, 4096, 0, 0), (149, 4096, 1, 2), (401, 3100, -2, 0), (2, 210001, 1, 1),
                                                    (96, 3125, 0, 0), (96, 3125, -1, 0), (8, 16032, 0, 0), (8, 16032, 1, 3), (6, 16032, 1, 3),
                                                    (10, 12000, 0, 0), (10, 12000, -1, 0), (78, 3847, 0, 0), (78, 3846, -1, 2),
                                                    (512, 3072, 0, 0), (512, 3072, -1, 0), (512, 3080, 1, 1)])
@pytest.mark.parametrize("per_sm", [1, 2])
def test_long_rows_shared_by_the_warps_of_an_sm(B, rows, vectors, extra, off, dtype, per_sm):
    """Rows of `vectors` 16-byte vectors plus `extra` elements, the tensor `off` elements past a vector's start: below, at and above
    the sizes from which an SM's warps share one range, and rows that begin and end inside a vector.  Maxima at the ends of the
    row, of a trip, of a block and of an SM's range; a second, equal one further right in every third row; rows of -inf, of
    NaN, and with one NaN before the maximum."""
    epv = 8 if dtype == torch.bfloat16 else 4
    V = vectors * epv + extra
    g = torch.Generator(device="cuda").manual_seed(V + rows + off)
    buf = torch.randn(rows * V + 2 * epv, generator=g, device="cuda", dtype=torch.float32).clamp_(max=7.0).to(dtype)
    buf[:off] = 50.0
    buf[off + rows * V:] = 50.0                           # what lies before and behind the tensor must not be seen
    flat = buf[off:off + rows * V].view(rows, V)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    span = -(-(rows * V // epv) // (per_sm * sms)) * epv  # elements of a range, one or two to an SM
    for r in range(rows):
        start = r * V
        edge = (-start) % span                            # the first element of a range inside this row, if it has one
        p = [0, V - 1, 256 * epv - 1, 2048 * epv, min(edge, V - 1), max(0, min(edge, V) - 1), V // 3][r % 7]
        flat[r, p] = 9.0
        if r % 3 == 0:
            flat[r, p + (V - 1 - p) // 2] = 9.0
        if r % 11 == 5:
            flat[r] = float("-inf")
        if r % 11 == 6:
            flat[r] = float("nan")
        if r % 11 == 7:
            flat[r, 0] = float("nan")
    # two positions per candidate
    K = 1
    Bn, n = rows // 2, 1
    logits = flat[:2 * Bn].view(Bn, K, n + 1, V)
    cand = torch.randint(0, V, (Bn, K, n), dtype=torch.int64).to(torch.int32)
    am = logits.float().nan_to_num(nan=float("-inf"), posinf=float("inf"), neginf=float("-inf")).argmax(-1).cpu()
    cand[::2, 0, 0] = am[::2, 0, 0].to(torch.int32)
    _check(B, cand, logits)


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("trips", [0.4, 1, 1.1, 2.6, 4, 5, 5.1, 9.9, 10.1, 20, 20.1])
def test_blocks_of_a_shared_range(B, trips, dtype):
    """Long rows whose warps get `trips` trips of 256 vectors each, on both sides of the sizes where the blocks they take change:
    every row's maximum is found, wherever in a block, a trip or a warp's lanes it lies."""
    epv = 8 if dtype == torch.bfloat16 else 4
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    V = 128256 if trips < 1 else 32003
    rows = int(trips * 256 * 14 * 2 * sms * epv / V) // 4 * 4
    g = torch.Generator(device="cuda").manual_seed(rows)
    x = torch.randint(-100, 100, (rows * V,), generator=g, device="cuda", dtype=torch.int8).to(dtype).view(rows, V)
    r = torch.arange(rows, device="cuda")
    at = torch.randint(0, V, (rows,), generator=g, device="cuda")
    x[r, at] = 101.0
    second = torch.minimum(at + 1 + 37 * (r % 11), torch.full_like(at, V - 1))     # an equal one behind it in every third row
    x[r[::3], second[::3]] = 101.0
    Bn, K, n = rows // 4, 2, 1
    _, _, _, ws = B.spec_verify(torch.zeros(Bn, K, n, dtype=torch.int32, device="cuda"), x.view(Bn, K, n + 1, V))
    assert B.spec_poll_error(ws) == 0
    assert torch.equal(ws_view(ws, 256, rows, torch.int32), at.to(torch.int32))


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("V", [24577, 128256])
def test_rows_whose_maximum_rises_trip_by_trip(B, V, dtype):
    """Rows that rise from end to end, fall, or rise in every 256 vectors: the warps that share such a row raise its key again and
    again while others compare with it, and some trips of a warp reach it and some do not."""
    epv = 8 if dtype == torch.bfloat16 else 4
    Bn, K, n = 6_000_000 // V // 4, 2, 1
    i = torch.arange(V, device="cuda", dtype=torch.float32)
    rising, trip = i / V * 64.0, (i % (256 * epv)) / (256 * epv) * 32.0
    kinds = torch.stack([rising, 64.0 - rising, trip, trip + rising, (i % 2) * rising, -rising])
    rows = kinds[torch.arange(Bn * K * (n + 1), device="cuda") % len(kinds)]
    logits = rows.to(dtype).view(Bn, K, n + 1, V).contiguous()
    g = torch.Generator().manual_seed(V)
    cand = torch.randint(0, V, (Bn, K, n), generator=g, dtype=torch.int64).to(torch.int32)
    for _ in range(5):
        _check(B, cand, logits)


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("Bn,K,n,vectors", [(1, 2, 3, 6143), (1, 2, 3, 6144), (1, 3, 1, 6145), (2, 37, 2, 6150),
                                            (3, 25, 2, 6151), (4, 37, 1, 3073), (149, 1, 1, 3073), (16, 37, 1, 1535),
                                            (16, 37, 1, 1536), (593, 1, 1, 1536), (1, 1, 9, 1537), (7, 3, 3, 1)])
def test_early_exit_rows_shared_by_the_ctas_of_a_cluster(B, Bn, K, n, vectors, dtype):
    """Row lengths and candidate counts at which 1, 2, 4 and 8 CTAs share a candidate, the maxima at the ends of the parts
    and, for every third row, an equal one in a later part (the first must win)."""
    V = vectors * (8 if dtype == torch.bfloat16 else 4)
    g = torch.Generator().manual_seed(V + Bn)
    x = torch.randn(Bn, K, n + 1, V, generator=g, dtype=torch.float32).to(dtype)
    rows = x.view(-1, V)
    for r in range(rows.shape[0]):
        parts = 1 << r % 4
        end = min(V, -(-vectors // parts) * (V // vectors) * (1 + r // 4 % parts))
        p = (end - 1, end % V)[r % 2]
        rows[r, p] = 9.0
        if r % 3 == 0:
            rows[r, p + (V - 1 - p) // 2] = 9.0
    cand = torch.randint(0, V, (Bn, K, n), generator=g, dtype=torch.int64).to(torch.int32)
    am = x.float().argmax(-1)
    for k in range(Bn * K):
        m = k % (n + 1)
        cand.view(-1, n)[k, :m] = am.view(-1, n + 1)[k, :m].to(torch.int32)
    host = synth.bf16_bits(x) if dtype == torch.bfloat16 else x.numpy()
    o = oracle.verify(cand.numpy(), host, oracle.BF16 if dtype == torch.bfloat16 else oracle.F32, want_g=True)
    acc, best, nxt, ws = B.spec_verify(cand.cuda(), x.cuda(), early_exit=True)
    assert B.spec_poll_error(ws) == 0
    for got, want in zip((acc, best, nxt), o):
        assert np.array_equal(got.cpu().numpy(), want)
    got = ws_view(ws, 256, Bn * K * (n + 1), torch.int32).cpu().numpy().reshape(Bn, K, n + 1)
    read = np.cumprod(np.concatenate([np.ones((Bn, K, 1), bool), cand.numpy() == o[3][:, :, :n]], 2), 2) > 0
    assert np.array_equal(got, np.where(read, o[3], -1))
