"""Launches of the tensor-core X stage that overlap their start with the kernel before them (packed samples, back to
back on one stream) neither read nor overwrite what it still writes or reads."""
import numpy as np
import pytest

import oracle
from _gpu_helpers import int_case

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.mark.parametrize("n,c,t,bits", [(64, 300, 200, 8), (16, 700, 128, 4), (128, 160, 300, 8), (256, 40, 200, 4)])
def test_back_to_back_calls_on_one_stream(n, c, t, bits):
    # accumulating calls whose samples the call before has just been given to, outputs that the next call reads
    from paper_0906_1887_gb300 import corr
    p = int_case(n + t, n, c, t, bits)
    ref = torch.from_numpy(oracle.xcorr_int(p, n, c, t, bits)).cuda()
    plan = corr.Plan(n, c, t, bits)
    x = torch.from_numpy(np.ascontiguousarray(p).view(np.uint8).reshape(-1).copy()).cuda()
    y, junk = torch.empty_like(x), torch.randint(0, 256, x.shape, device="cuda", dtype=torch.uint8)
    vis, other = plan.empty_vis(1, "cuda"), plan.empty_vis(1, "cuda")
    ws = plan.empty_workspace(corr.ENGINE_TC, 1, "cuda")
    for rep in range(20):
        y.copy_(x)                                  # a kernel that the X stage must wait for
        plan.run(y, vis, ws)
        plan.run(y, vis, ws, accumulate=True)       # adds into what the call before writes
        y.copy_(junk)                               # must wait for its reads
        plan.run(y, other, ws)
        y.copy_(x)
        plan.run(y, vis, ws, accumulate=True)
    torch.cuda.synchronize()
    assert plan.check_device() == 0
    assert torch.equal(vis[0], 3 * ref)
    plan.close()


def test_fused_dump_waits_for_its_phasors():
    # alternating delays: the phasors of a call overwrite those of the one before, in one workspace
    from oracle import dump as odump
    from paper_0906_1887_gb300 import corr
    n, c, t = 64, 40, 200
    p = int_case(5, n, c, t, 8)
    plan = corr.Plan(n, c, t, 8)
    x = torch.from_numpy(np.ascontiguousarray(p).view(np.uint8).reshape(-1).copy()).cuda()
    ws = torch.empty(plan.dump_workspace_size(), dtype=torch.uint8, device="cuda")
    nu = 1.5e8 + 1e4 * np.arange(c)
    taus = [np.random.default_rng(k).normal(0, 2e-6, n) for k in range(2)]
    dev = [torch.from_numpy(tau).cuda() for tau in taus]
    nu_d = torch.from_numpy(nu).cuda()
    outs = [torch.empty((c, plan.n_baselines, 2), device="cuda") for _ in range(20)]
    for k, o in enumerate(outs):
        plan.run_dump(x, o, 3, dev[k % 2], nu_d, ws)
    torch.cuda.synchronize()
    acc = oracle.xcorr_int(p, n, c, t, 8)
    for k, o in enumerate(outs):
        if k > 1:
            assert torch.equal(o, outs[k % 2])
            continue
        ref = odump.dump_corrected(acc, 3, taus[k], nu)
        err = np.hypot(*(o.cpu().numpy().astype(np.float64) - ref).transpose(2, 0, 1))
        assert np.all(err <= 8 * 2.0 ** -24 * np.hypot(ref[..., 0], ref[..., 1]) + 1e-30)
    plan.close()
