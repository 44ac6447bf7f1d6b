"""The LM head's lists (tf_lmhead_partials, tf_lmhead_merge) against a full fp64 log-softmax, on rows
that take each way through the merge: a few halves in the k-th's bucket, a bucket too crowded to keep
(one logit far above all others), equal logits throughout (ids in order), fewer half blocks than k,
more halves than fit in registers, and k from 1 to 512."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

CASES = [
    # V, d, k, dtype, rows
    (20000, 128, 64, "bf16", "plain"),
    (20000, 128, 1, "bf16", "plain"),
    (20000, 64, 512, "bf16", "plain"),
    (20000, 576, 32, "bf16", "plain"),       # copies of the rows with d > 512 (79 blocks)
    (20000, 4096, 32, "bf16", "plain"),      # and none from d = 4096 on
    (20000, 128, 64, "f32", "plain"),
    (60000, 128, 200, "bf16", "plain"),      # candidates around 256, up to which they are ranked by counting
    (60000, 128, 240, "bf16", "plain"),
    (60000, 128, 320, "bf16", "plain"),
    (9001, 64, 32, "bf16", "outlier"),       # every other half in the lowest bucket
    (9001, 64, 32, "f32", "outlier"),
    (5000, 64, 40, "bf16", "equal"),
    (1500, 64, 64, "bf16", "plain"),         # 12 half blocks
    (270001, 64, 48, "bf16", "plain"),       # 2110 half blocks
    (2687777, 64, 64, "bf16", "plain"),      # shared memory for k halves, but not for more
    (2895800, 64, 64, "bf16", "plain"),      # the largest vocabulary of these dims
    (20000, 320, 40, "bf16", "twins"),       # 120 equal rows of W above all others, three per chunk
    (20000, 320, 40, "f32", "twins"),
]
# numbers of rows at which the tensor-core kernel changes: four copies of the rows, two, one; then
# with d > 512 no copies (of 36 vocabulary blocks), CTA pairs, single CTAs over three (and five) M-tiles, pairs again
ROWS = [(1, 64), (32, 64), (33, 64), (64, 64), (65, 64), (128, 64), (129, 64), (1, 576), (40, 576), (129, 576),
        (256, 576), (257, 576), (385, 576), (513, 576), (641, 576)]


@pytest.mark.parametrize("n,d", ROWS)
def test_lists_at_every_row_split(n, d):
    test_lists_equal_a_full_sort(9001, d, 32, "bf16", "plain", n)


@pytest.mark.parametrize("n", [8, 16, 17, 32, 33, 65])
def test_fp32_lists_of_rows_that_are_no_multiple_of_16_bytes(n):
    test_lists_equal_a_full_sort(3001, 130, 32, "f32", "plain", n)


@pytest.mark.parametrize("V,d,k,dtype,rows", CASES)
def test_lists_equal_a_full_sort(V, d, k, dtype, rows, n=21):
    from paper_2606_03819_gb300 import Dims
    from paper_2606_03819_gb300 import binding as B
    dt = torch.bfloat16 if dtype == "bf16" else torch.float32
    g = torch.Generator().manual_seed(V + k)
    W = torch.randn(V, d, generator=g)
    x = torch.randn(n, d, generator=g) * 3.0 / d ** 0.5
    if rows == "outlier":
        W[V // 2] = 200.0 * torch.sign(x.sum(0))
        x = x.abs() * torch.sign(W[V // 2])
    elif rows == "twins":
        # their chunks are all recomputed, with the sum in another order: all of them may come out lower than
        # the k-th candidate was
        W = -(0.5 + torch.rand(V, d, generator=g))
        x = x.abs()
        W[(32 * torch.arange(50, 90)[:, None] + torch.arange(3)).flatten()] = -0.2 * torch.rand(d, generator=g)
    elif rows == "equal":
        x.zero_()
    W, x = W.to(dt).cuda(), x.to(dt).cuda()
    dims = Dims(n, d, V, 64, 1, 1, k, 8, dtype=dtype, mode="marginal")
    ws = B.alloc_workspace(dims)
    ids = torch.empty(n, k, dtype=torch.int32, device="cuda")
    logp = torch.empty(n, k, device="cuda")
    B.tf_status_reset(ws)
    B.tf_lmhead_partials(dims, W, x, n, ws)
    B.tf_lmhead_merge(dims, W, x, n, k, ids, logp, ws)
    assert B.tf_status_read(ws) & ~B.TF_DEV_RECOMPUTED == 0
    z = x.double() @ W.double().t()
    lp = torch.log_softmax(z, 1)
    ids, logp = ids.cpu().numpy(), logp.double().cpu().numpy()
    if rows == "equal":
        np.testing.assert_array_equal(ids, np.arange(k)[None].repeat(n, 0))
        np.testing.assert_allclose(logp, -np.log(V), atol=1e-5)
        return
    # fp32 sums of d products of size up to |z|: far below 1e-3 (relative 1e-5 for the outlier's 1e3)
    tol = 1e-3 * max(1.0, float(z.abs().max()) / 100)
    want = lp.topk(k, dim=1).values.cpu().numpy()
    np.testing.assert_allclose(logp, want, atol=tol)
    np.testing.assert_allclose(lp.cpu().numpy()[np.arange(n)[:, None], ids], logp, atol=tol)
    for r in range(n):
        assert len(set(ids[r].tolist())) == k
