"""Failure detection without a GPU fault: every wait of the tensor-core kernels is bounded.

With the progress-wait limit set far below a copy's latency (tf_set_wait_limit_ns), the
LM-head kernel must give up, set TF_DEV_TIMEOUT (tf_status_read -> TF_ERR_TIMEOUT), drain its
own copies and MMAs and return, leaving the context usable: a following call with the default
limit on the same stream must give the results of a call made before, bit for bit. Covered for
one CTA per tile (16 and 40 rows: four and two copies of the rows, whose warps wait for one another;
100 rows: one) and for CTA pairs (200 rows, two M-tiles), and for the approximator's GEMMs (clusters that
split K, and the tail split, whose warps wait for one another too). The timed-out call's results are
never used."""
import pathlib
import re

import pytest
import torch

from paper_2606_03819_gb300 import binding as Bn


def test_wait_limit_setter_checks_its_range():
    Bn.load_library()
    with pytest.raises(Bn.TreeFlashError):
        Bn.tf_set_wait_limit_ns(61 * 10 ** 9)
    Bn.tf_set_wait_limit_ns(0)


def test_warps_that_may_have_given_up_are_not_waited_for_without_limit():
    # An epilogue warp decides by itself whether its accumulator came in time. A hardware barrier of part
    # of a block's warps (bar.sync with an id, barrier.cta) would keep the others for ever once one has
    # given up; what warps of a tensor-core kernel wait for is a shared-memory barrier polled with a limit.
    import paper_2606_03819_gb300
    csrc = pathlib.Path(paper_2606_03819_gb300.__file__).parent / "csrc"
    files = [csrc / "tc_gemm.cu", csrc / "tc_ptx.cuh"]
    for f in files:
        code = re.sub(r"//[^\n]*", "", f.read_text())
        assert not re.search(r"\bbar(rier)?\.(sync|cta|red|arrive)\b|named_barrier", code), f
        # and every such poll has a limit: mbar_try_wait appears in the bounded waits alone
        for fn in re.findall(r"mbar_try_wait(?:_cluster)?\(", code) if f.name == "tc_gemm.cu" else ():
            pytest.fail(f"{f}: {fn}")


def _lmhead(dims, lm, x, rows, ws):
    ids = torch.empty(rows, dims.K1, dtype=torch.int32, device="cuda")
    lp = torch.empty(rows, dims.K1, dtype=torch.float32, device="cuda")
    Bn.tf_status_reset(ws)
    Bn.tf_lmhead_partials(dims, lm, x, rows, ws)
    Bn.tf_lmhead_merge(dims, lm, x, rows, dims.K1, ids, lp, ws)
    return ids.cpu(), lp.cpu(), Bn.tf_status_read(ws)


@pytest.mark.gpu
@pytest.mark.parametrize("batch,gamma,d,V", [(1, 16, 2048, 40960), (1, 40, 2048, 40960), (2, 50, 4096, 4096),
                                             (4, 50, 4096, 4096)],
                         ids=["four_copies", "two_copies", "one_cta_per_tile", "cta_pairs"])
def test_bounded_wait_times_out_and_the_context_stays_usable(batch, gamma, d, V):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    Bn.load_library()
    dims = Bn.Dims(batch=batch, d=d, V=V, I=64, gamma=gamma, M=4, K2=8, B=8, dtype="bf16",
                   mode="marginal")
    rows = batch * gamma
    gen = torch.Generator(device="cuda").manual_seed(7)
    lm = (torch.randn(dims.V, dims.d, generator=gen, device="cuda") * 0.02).to(torch.bfloat16)
    x = (torch.randn(rows, dims.d, generator=gen, device="cuda") * 2.0).to(torch.bfloat16)
    ws = Bn.alloc_workspace(dims)
    try:
        Bn.tf_set_wait_limit_ns(0)
        ref_ids, ref_lp, flags = _lmhead(dims, lm, x, rows, ws)
        assert not (flags & ~Bn.TF_DEV_RECOMPUTED), f"reference call flags {flags}"
        # 1 ns: any wait that is not satisfied within its first polls gives up (32 or 64 K-steps per
        # vocabulary block stream through a ring of a few stages, so many waits are real)
        Bn.tf_set_wait_limit_ns(1)
        Bn.tf_status_reset(ws)
        Bn.tf_lmhead_partials(dims, lm, x, rows, ws)
        flags = Bn.tf_status_read(ws)
        assert flags & Bn.TF_DEV_TIMEOUT, f"no timeout reported (flags {flags})"
        torch.cuda.synchronize()     # no sticky error: the kernel returned normally
        # back to the default limit, same stream and workspace: the call must be exact again
        Bn.tf_set_wait_limit_ns(0)
        ids, lp, flags = _lmhead(dims, lm, x, rows, ws)
        assert not (flags & ~Bn.TF_DEV_RECOMPUTED), f"call after the timeout: flags {flags}"
        assert torch.equal(ids, ref_ids)
        assert torch.equal(lp.view(torch.int32), ref_lp.view(torch.int32))
    finally:
        Bn.tf_set_wait_limit_ns(0)


@pytest.mark.gpu
@pytest.mark.parametrize("batch", [1, 115], ids=["k_split", "tail_split"])
def test_approximator_times_out_and_the_context_stays_usable(batch):
    # 17 rows: both GEMMs on K-splitting clusters; 1955 rows: 160 gate/up units, more than the SMs by a few
    # that run as K-chunks each (152 SMs), and clusters for the down projection
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    Bn.load_library()
    dims = Bn.Dims(batch=batch, d=512, V=1000, I=2560, gamma=5, M=4, K2=8, B=8, dtype="bf16")
    gen = torch.Generator(device="cuda").manual_seed(11)
    r = lambda *n: (torch.randn(*n, generator=gen, device="cuda") * 0.05).to(torch.bfloat16)  # noqa: E731
    d, I = dims.d, dims.I
    w = dict(lm_head=r(dims.V, d), embed=r(dims.V, d), norm_h=1 + r(d), norm_e=1 + r(d), w_gate=r(I, 2 * d),
             w_up=r(I, 2 * d), w_down=r(d, I))
    hidden = r(batch, dims.gamma, d)
    root = torch.arange(batch, dtype=torch.int32, device="cuda")
    top = torch.randint(0, dims.V, (batch, dims.gamma, dims.K1), generator=gen, device="cuda", dtype=torch.int32)
    ws = Bn.alloc_workspace(dims)

    def run():
        hp = torch.empty(batch, dims.R, d, dtype=torch.bfloat16, device="cuda")
        Bn.tf_status_reset(ws)
        Bn.tf_ar_approx(dims, w, hidden, root, top, hp, ws)
        return hp, Bn.tf_status_read(ws)

    try:
        Bn.tf_set_wait_limit_ns(0)
        want, flags = run()
        assert flags == 0
        Bn.tf_set_wait_limit_ns(1)
        assert run()[1] & Bn.TF_DEV_TIMEOUT
        torch.cuda.synchronize()
        Bn.tf_set_wait_limit_ns(0)
        got, flags = run()
        assert flags == 0
        assert torch.equal(got.view(torch.int16), want.view(torch.int16))
    finally:
        Bn.tf_set_wait_limit_ns(0)
