"""The waits between the blocks of the float-float factor give up instead of hanging: with
their limit at a nanosecond msp_nystrom returns MSP_ETIMEOUT, and with it restored the same
context forms the same factor bit for bit."""

import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("s", [100, 512])
def test_factor_wait_gives_up_and_recovers(s):
    from paper_2405_05865_gb300 import Context, MspError
    ctx = Context(0)
    g = torch.Generator(device="cuda").manual_seed(4)
    A = ctx.rbf_kernel(torch.rand((2048, 3), generator=g, device="cuda", dtype=torch.float64), 0.1)
    sk = ctx.sketch(A, s, 8)
    f = ctx.nystrom(sk, 1e-2, 0.0, phi=0)
    want = f.parts()
    f.close()
    ctx.set_grid_wait_limit(1e-9)
    try:
        with pytest.raises(MspError) as e:
            ctx.nystrom(sk, 1e-2, 0.0, phi=0)
        assert e.value.status == 7          # MSP_ETIMEOUT
    finally:
        ctx.set_grid_wait_limit(0.0)
    f = ctx.nystrom(sk, 1e-2, 0.0, phi=0)
    got = f.parts()
    assert got["retries"] == want["retries"] and got["shift"] == want["shift"]
    assert torch.equal(got["Linv"], want["Linv"]) and torch.equal(got["M2"], want["M2"])
    f.close()
    sk.close()
    ctx.close()
