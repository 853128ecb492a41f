"""MemoryBridge output on the GPU against the fp64 oracle: LayerNorm,
nu tanh and the 2 nu norm cap, row by row (fp32 on the GPU: within 2e-5 of
nu relative), with and without the cap active, in place, and over more rows
than the grid (grid-stride)."""

import numpy as np
import pytest
import torch

import oracle
import paper_2609_25537_gb300 as cmc

pytestmark = pytest.mark.gpu


def _case(rows, D, nu, scale, affine, dev, seed=0, in_place=False):
    rng = np.random.default_rng(seed)
    x = (rng.standard_normal((rows, D)) * scale + 0.3).astype(np.float32)
    g = (1 + 0.2 * rng.standard_normal(D)).astype(np.float32) if affine else None
    b = (0.2 * rng.standard_normal(D)).astype(np.float32) if affine else None
    xd = torch.from_numpy(x).to(dev)
    gd = None if g is None else torch.from_numpy(g).to(dev)
    bd = None if b is None else torch.from_numpy(b).to(dev)
    out = cmc.bridge_epilogue(xd, nu, gamma=gd, beta=bd, out=xd if in_place else None)
    got = out.cpu().numpy().astype(np.float64)
    ref = oracle.bridge_epilogue(x, np.ones(D) if g is None else g, np.zeros(D) if b is None else b, nu)
    np.testing.assert_allclose(got, ref, rtol=2e-5, atol=2e-5 * nu)
    assert np.all(np.linalg.norm(got, axis=1) <= 2 * nu * (1 + 1e-5))
    return ref


# rows in registers.  Plain: 128 threads a CTA, D = 64 and 36 one float4 per
# thread, 1028 three (the last one partial), 2048 four, 2600 six, 3072 six, 3588
# eight (partial), 4096 eight; 16384 512 threads, eight.  With gamma and beta
# over 2,048 features 256 threads, three or four
@pytest.mark.parametrize("rows,D", [(1024, 4096), (300, 64), (7, 16384), (50, 36), (33, 2048),
                                    (17, 3072), (29, 1028), (21, 2600), (13, 3588)])
@pytest.mark.parametrize("affine", [False, True])
def test_bridge_epilogue_shapes(cuda_device, rows, D, affine):
    ref = _case(rows, D, 0.8, 2.0, affine, cuda_device)
    # at D >= 16 these rows are capped: the norm is exactly 2 nu
    if D >= 64:
        np.testing.assert_allclose(np.linalg.norm(ref, axis=1), 1.6, rtol=1e-12)


def test_bridge_epilogue_below_the_cap_and_in_place(cuda_device):
    # a tiny gamma keeps nu tanh(m_hat) well inside the 2 nu ball: no rescale
    rng = np.random.default_rng(3)
    D = 512
    x = rng.standard_normal((64, D)).astype(np.float32)
    g = np.full(D, 0.01, dtype=np.float32)
    xd = torch.from_numpy(x).to(cuda_device)
    out = cmc.bridge_epilogue(xd, 1.5, gamma=torch.from_numpy(g).to(cuda_device), out=xd)
    assert out.data_ptr() == xd.data_ptr()
    ref = oracle.bridge_epilogue(x, g, np.zeros(D), 1.5)
    np.testing.assert_allclose(out.cpu().numpy(), ref, rtol=2e-5, atol=3e-5)
    assert np.all(np.linalg.norm(ref, axis=1) < 3.0)


def test_bridge_epilogue_many_rows(cuda_device):
    _case(20000, 64, 0.5, 1.0, True, cuda_device, seed=9)


@pytest.mark.parametrize("D,per_sm", [(4, 8), (2048, 8), (2052, 4), (4096, 4), (4100, 2), (8192, 2),
                                      (8196, 2), (10244, 2), (12288, 2), (14336, 2), (16384, 2)])
@pytest.mark.parametrize("affine", [False, True])
def test_bridge_epilogue_thread_counts(cuda_device, D, per_sm, affine):
    """The row lengths where a CTA's threads change, over three more rows than the most CTAs
    that are resident, so that some walk two (gamma and beta kept from the first)."""
    sms = torch.cuda.get_device_properties(cuda_device).multi_processor_count
    _case(per_sm * sms + 3, D, 0.8, 2.0, affine, cuda_device, in_place=True)


@pytest.mark.parametrize("D,per_sm", [(1540, 101), (1664, 101), (2052, 21), (2304, 31), (3328, 38),
                                      (3072, 61), (4076, 60), (1924, 81), (2048, 81), (2820, 51),
                                      (4096, 51)])
@pytest.mark.parametrize("gain,shift", [(False, False), (True, True), (True, False), (False, True)])
def test_bridge_epilogue_many_rows_as_few(cuda_device, D, per_sm, gain, shift):
    """So many rows that the variant for many rows takes them (with or without gamma and beta, as
    the width has it): the same bits as from calls of a few rows each where those take 128 threads
    too.  With gamma or beta and over 2,048 features they take 256, and add in another order: the
    three sums are off by some ten roundings of 2^-24 each, 2e-6 in all."""
    sms = torch.cuda.get_device_properties(cuda_device).multi_processor_count
    rows = per_sm * sms + 5
    g = torch.Generator(device=cuda_device).manual_seed(D)
    x = torch.randn(rows, D, device=cuda_device, generator=g) * 2.0 + 0.3
    kw = {}
    if gain:
        kw["gamma"] = torch.randn(D, device=cuda_device, generator=g) * 0.02
    if shift:
        kw["beta"] = torch.randn(D, device=cuda_device, generator=g) * 0.005
    few = torch.cat([cmc.bridge_epilogue(part, 0.8, **kw) for part in x.split(10 * sms)])
    many = cmc.bridge_epilogue(x, 0.8, **kw)
    if kw and D > 2048:
        assert ((many - few).norm(dim=1) <= 2e-6 * few.norm(dim=1)).all()
    else:
        assert torch.equal(many, few)
    assert torch.equal(cmc.bridge_epilogue(x, 0.8, out=x, **kw), many)
