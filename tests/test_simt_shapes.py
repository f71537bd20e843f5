"""The fp32 and layout kernels at the sizes where their variants change over: GEMM tiles of four or six
columns and four or eight rows a thread with and without a K split, gathers whose row counts leave a
remainder of the four loads in flight, rows of whole 16-byte chunks and others."""
import numpy as np
import pytest

from paper_1906_11786_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,P,F,S,n,lam", [
    (96, 3, 3, 32, 95, 2.0),       # six columns; ragged rows, no K split in the forward
    (96, 5, 5, 64, 6100, 1.0),     # six columns and eight rows
    (64, 4, 4, 64, 513, 3.0),      # four and four, K split in the backward
    (160, 2, 2, 32, 200, 0.0),     # a width that is a multiple of neither 64 nor 96
    (32, 6, 6, 128, 4000, 1.0),    # eight rows over half-empty tiles
    (256, 1, 1, 256, 300, 0.0)])   # one type; K = 256, the shortest that is split
def test_fp32_propagation_matches_the_oracle(H, P, F, S, n, lam):
    import oracle
    import torch
    from gpu_common import Case, L, TOL, assert_close, ensure_built, f32_dev
    ensure_built()
    c = Case([synth.gen_graph(n, F, False, S // 3, S // 3, lam, 9 * n + H)], P, S, H, "f32", seed=H)
    Y = torch.empty((c.N, H), device="cuda")
    L.band_propagate_fwd(c.plan, "f32", H, c.E_band_dev, c.dprm["W"], c.dprm["b"], Y,
                         c.ws(L.BG_OP_PROPAGATE_FWD))
    dY = np.zeros((c.N, H))
    dY[: c.n_real] = np.random.default_rng(3).standard_normal((c.n_real, H)).astype(np.float32)
    dE, dW = torch.empty((c.N, H), device="cuda"), torch.empty((P, H, H), device="cuda")
    db = torch.empty((P, H), device="cuda")
    L.band_propagate_bwd(c.plan, "f32", H, c.E_band_dev, c.dprm["W"], f32_dev(dY), dE, dW, db,
                         c.ws(L.BG_OP_PROPAGATE_BWD))
    torch.cuda.synchronize()
    args = (c.N, P, H, *c.edges, c.E_band, c.prm["W"])
    assert_close(Y.cpu().numpy(), oracle.propagate_fwd(*args, c.prm["b"]), TOL["f32"], "Y")
    for got, ref, what in zip((dE, dW, db), oracle.propagate_bwd(*args, dY), ("dE", "dW", "db")):
        assert_close(got.cpu().numpy(), ref, TOL["f32"], what)


@pytest.mark.parametrize("H", [1, 3, 8, 20, 64, 100, 256])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_pack_and_unpack_are_exact_at_any_row_size(H, dtype):
    import torch
    from gpu_common import L, ensure_built
    ensure_built()
    plan = L.band_plan([synth.gen_graph(n, 4, False, 9, 9, 1.0, n) for n in (130, 1, 77)], 4, 64)
    plan.upload()
    info, idx = plan.info(), torch.from_numpy(plan.export(L.BG_EXPORT_GATHER).astype(np.int64)).cuda()
    tdt = torch.float32 if dtype == "f32" else torch.bfloat16
    E = torch.randn((208, H), device="cuda").to(tdt)
    Eb = torch.full((info["n_pad"], H), 7.0, device="cuda", dtype=tdt)
    L.pack_states(plan, dtype, H, E, Eb)
    assert torch.equal(Eb[: info["n_real"]], E[idx]) and not Eb[info["n_real"]:].any()
    back = torch.zeros_like(E)
    L.unpack_states(plan, dtype, H, Eb, back)
    assert torch.equal(back, E)
