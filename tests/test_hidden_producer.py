"""The hidden states may be written by the kernel just ahead of the call on the same stream, also by one
that lets its dependents start early (as every kernel of this library does, at its entry): Eq. 1 of one
call's h' as the next call's hidden states, without a synchronisation between them, must give the bits of
the same two calls with one."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,d,batch", [("bf16", 4096, 1), ("bf16", 1024, 9), ("f32", 512, 1)])
def test_hidden_states_of_the_kernel_just_ahead(dtype, d, batch):
    from paper_2606_03819_gb300 import binding as B
    dims = B.Dims(batch, d, 2000, 4096, 8, 4, 8, 8, dtype=dtype)
    dt = dims.torch_dtype
    g = torch.Generator(device="cuda").manual_seed(d)
    r = lambda *n: (torch.randn(*n, generator=g, device="cuda") * 0.02).to(dt)  # noqa: E731
    w = dict(lm_head=r(dims.V, d), embed=r(dims.V, d), norm_h=1 + r(d), norm_e=1 + r(d), w_gate=r(dims.I, 2 * d),
             w_up=r(dims.I, 2 * d), w_down=r(d, dims.I))
    root = torch.zeros(batch, dtype=torch.int32, device="cuda")
    top = torch.randint(0, dims.V, (batch, dims.gamma, dims.K1), generator=g, device="cuda", dtype=torch.int32)
    first, second = B.alloc_workspace(dims), B.alloc_workspace(dims)
    # the first call's h' [batch, R, d], of which the second takes the first batch * gamma rows
    middle = B.tf_workspace_h_prime(dims, first).view(-1, d)[:batch * dims.gamma].view(batch, dims.gamma, d)
    inputs = [r(batch, dims.gamma, d) * 50 for _ in range(8)]

    def chain(hidden, wait):
        B.tf_ar_approx(dims, w, hidden, root, top, None, first)
        if wait:
            torch.cuda.synchronize()
        B.tf_ar_approx(dims, w, middle, root, top, None, second)
        return B.tf_workspace_h_prime(dims, second).clone()

    want = [chain(h, True) for h in inputs]
    for _ in range(4):
        for h, x in zip(inputs, want):
            assert torch.equal(chain(h, False), x)
