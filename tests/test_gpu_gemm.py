"""The tensor-core projection GEMM alone, through the C ABI, against a float64 matrix product of the
same bf16 inputs (the plain definition of the contraction)."""
import numpy as np
import pytest
import torch

from paper_2407_12021_b200 import inputs as gen

pytestmark = pytest.mark.gpu

SMALL16 = gen.ModelShape("gemm-small", 1, 512, 4, 128, 1408, 1024, "bf16")


def _model(shape, dev, seed, max_rows=128):
    from paper_2407_12021_b200 import binding as B
    w = gen.model_weights(shape, seed, device=dev)
    return B, w, B.aded_model_create(shape, w, max_rows=max_rows, max_batch=1)


def _check(B, model, w, which, rows, seed):
    mats = {0: w["layers"][0]["wqkv"], 1: w["layers"][0]["wo"], 2: w["layers"][0]["wgu"], 3: w["layers"][0]["wd"],
            4: w["lm_head"]}
    W = mats[which]
    k = W.shape[1]
    x = gen.normal((rows, k), 1.0, seed, 500 + which, device=W.device, dtype=torch.bfloat16)
    y = B.aded_debug_gemm(model, 0, which, x)
    y2 = B.aded_debug_gemm(model, 0, which, x)
    torch.cuda.synchronize()
    assert B.aded_model_poll_status(model) == 0
    assert torch.equal(y, y2), "the split-tile reduction must not depend on timing"
    want = x.double().cpu().numpy() @ W.double().cpu().numpy().T
    got = y.double().cpu().numpy()
    err = np.max(np.abs(got - want)) / np.max(np.abs(want))
    assert err < 2e-5, (which, rows, err)
    # element-wise: every output within fp32 accumulation error of its own magnitude scale
    bound = 4e-6 * (np.abs(x.double().cpu().numpy()) @ np.abs(W.double().cpu().numpy()).T) + 1e-12
    assert np.all(np.abs(got - want) <= bound), (which, rows)


@pytest.mark.parametrize("rows", [1, 16, 17, 64, 100, 128])
def test_small_shapes_all_projections(cuda_device, rows):
    B, w, model = _model(SMALL16, cuda_device, 41)
    for which in range(5):
        _check(B, model, w, which, rows, 41 + rows)


@pytest.mark.parametrize("rows", [64, 128, 3])
def test_7b_shapes(cuda_device, rows):
    B, w, model = _model(gen.LLAMA7B_1L, cuda_device, 42)
    for which in range(5):
        _check(B, model, w, which, rows, 42 + rows)


def test_more_rows_than_one_pass(cuda_device):
    """Calls with more than 128 rows run as passes of up to 256 rows over the weights (one accumulator of 256
    tensor-memory columns): a single wide pass with a ragged tail (129, 256), two passes (300), five (1228)."""
    B, w, model = _model(SMALL16, cuda_device, 43, max_rows=1228)
    for which in (0, 3):
        _check(B, model, w, which, 300, 43)
        _check(B, model, w, which, 129, 44)
        _check(B, model, w, which, 256, 45)
    _check(B, model, w, 4, 1228, 46)


def test_7b_shape_wide_pass(cuda_device):
    B, w, model = _model(gen.LLAMA7B_1L, cuda_device, 47, max_rows=416)
    for which in (0, 1, 2, 3):
        _check(B, model, w, which, 416, 47)


@pytest.mark.parametrize("rows", [33, 48, 65, 80, 97, 112, 113])
def test_row_counts_between_the_powers_of_two(cuda_device, rows):
    """The rows of a pass arrive as one box of their padded number; few units per CTA (small shapes)."""
    B, w, model = _model(SMALL16, cuda_device, 45)
    for which in range(5):
        _check(B, model, w, which, rows, 45 + rows)


@pytest.mark.parametrize("rows", [177, 192, 193, 208, 256 + 177, 256 + 192])
def test_wide_passes_of_every_padded_size(cuda_device, rows):
    """Passes of 129 to 256 rows, those of 177 to 192 among them (five stages of 40 KB: the launch with the most shared memory)."""
    B, w, model = _model(SMALL16, cuda_device, 46, max_rows=rows)
    for which in (0, 1, 3):
        _check(B, model, w, which, rows, 46)


@pytest.mark.parametrize("dtype,rows", [("f32", 1), ("f32", 16), ("f32", 17), ("f32", 128), ("f32", 300), ("bf16", 33), ("bf16", 128), ("bf16", 300)])
@pytest.mark.parametrize("offset", [0, 1])
def test_plain_gemm(cuda_device, dtype, rows, offset):
    """Models the tensor-core GEMM does not take: blocks of 16, 32 and 64 rows, k in one chunk and in several (pieces of 64, 128 and 256), a ragged number of
    columns, matrices that do not start on a 16-byte boundary.  Bound: fp32 sums of k products in a fixed order are off by at
    most k 2^-24 of the sum of their magnitudes, and by far less in the mean; 4e-6 of it is the bound of the tests above."""
    shape = gen.ModelShape("plain", 1, 1088, 17, 64, 1360, 1000, dtype)
    from paper_2407_12021_b200 import binding as B
    w = gen.model_weights(shape, 47, device=cuda_device)

    def moved(m):
        flat = torch.empty(m.numel() + offset, dtype=m.dtype, device=m.device)
        flat[offset:].view(m.shape).copy_(m)
        return flat[offset:].view(m.shape)

    w["lm_head"] = moved(w["lm_head"])
    w["layers"] = [{k: moved(v) for k, v in p.items()} for p in w["layers"]]
    model = B.aded_model_create(shape, w, max_rows=rows, max_batch=1)
    mats = {0: w["layers"][0]["wqkv"], 1: w["layers"][0]["wo"], 2: w["layers"][0]["wgu"], 3: w["layers"][0]["wd"], 4: w["lm_head"]}
    for which, W in mats.items():
        x = gen.normal((rows, W.shape[1]), 1.0, 48, 500 + which, device=W.device, dtype=W.dtype)
        y = B.aded_debug_gemm(model, 0, which, x)
        torch.cuda.synchronize()
        assert B.aded_model_poll_status(model) == 0
        want = x.double() @ W.double().T
        bound = 4e-6 * (x.double().abs() @ W.double().abs().T) + 1e-12
        assert bool(((y.double() - want).abs() <= bound).all()), (which, rows)
