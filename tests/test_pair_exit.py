"""The end of a CTA pair's work (xeng_tc.cu): the odd CTA must not exit before the commits of the even CTA's
MMA thread, which also arrive in its shared memory, have landed there.  The wait for them is bounded by
time, so it may only begin when nothing else is left to wait for; begun with the kernel, it would lapse in
any launch longer than its limit."""
import pathlib

import pytest

SRC = pathlib.Path(__file__).resolve().parents[1] / "paper_0906_1887_gb300" / "csrc" / "xeng_tc.cu"


def test_odd_cta_waits_for_the_last_commits_at_the_end_of_its_work():
    src = SRC.read_text()
    kernel = src[src.index("__global__ void __launch_bounds__(Cfg<MODE>::kThreads, 1) xeng_tc_kernel"):]
    kernel = kernel[:kernel.index("// ---- host side")]
    wait = "ptx::mbar_wait_drain(bar_drain"
    mma, epilogue = kernel.index("// ---------------- MMA issuer"), kernel.index("// ---------------- epilogue")
    conv, end = kernel.index("// ---------------- converters"), kernel.rindex("ptx::cluster_sync()")
    at = [i for i in range(len(kernel)) if kernel.startswith(wait, i)]
    assert len(at) == 2                                     # the issuer's own, and its peer's
    assert mma < kernel.index("commit(bar_drain)") < at[0] < epilogue
    assert epilogue < kernel.index("mbar_arrive_cluster(ptx::map_shared(bar_acc_empty") < at[1] < conv < end
    assert "rank != 0" in kernel[at[1] - 100:at[1]] and "wait_limit_ns" in kernel[at[1]:at[1] + 80]
    # an issuer with nothing to commit says so
    assert mma < kernel.index("mbar_arrive_cluster(ptx::map_shared(bar_drain, 1))") < epilogue


@pytest.mark.gpu
def test_launch_longer_than_the_drain_limit():
    # more than 0.2 s in one launch of CTA pairs on packed samples; some inputs' rows against float64
    # products (exact: the sums stay below 2^53)
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0906_1887_gb300 import corr
    n, c, t = 8192, 8, 196608
    plan = corr.Plan(n, c, t, 4)
    plan.set_operands(corr.OPERANDS_PACKED_F8)
    g = torch.Generator(device="cuda")
    g.manual_seed(1)
    x = torch.randint(0, 256, (t, c, n), generator=g, device="cuda", dtype=torch.uint8)
    vis = plan.empty_vis(1, "cuda")
    e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
    e[0].record()
    plan.run(x, vis)
    e[1].record()
    torch.cuda.synchronize()
    assert plan.check_device() == 0
    assert e[0].elapsed_time(e[1]) > 200.0
    rows = list(range(0, n, 1369)) + [n - 1]
    for ch in (0, c - 1):
        want = torch.zeros((len(rows), n, 2), dtype=torch.float64, device="cuda")
        for t0 in range(0, t, 16384):
            b = x[t0:t0 + 16384, ch].view(torch.int8)
            re, im = (b >> 4).double(), ((b << 4) >> 4).double()
            want[..., 0] += re[:, rows].T @ re + im[:, rows].T @ im
            want[..., 1] += im[:, rows].T @ re - re[:, rows].T @ im
        for k, i in enumerate(rows):
            b0 = i * n - i * (i - 1) // 2
            assert torch.equal(vis[0, ch, b0:b0 + n - i], want[k, i:].to(torch.int64))
    plan.close()
