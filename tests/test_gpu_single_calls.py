"""Single-tile calls on the merging engine, whose two status areas take turns: a
violation is reported by its own call only, whatever came before and follows, with
and without a wait after each call. Results against the oracle."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1311_0378_gb300 as rc  # noqa: E402


@pytest.mark.parametrize("shape", [(64, 64), (70, 65), (300, 200)])
@pytest.mark.parametrize("pattern", ["gggg", "bg", "gbg", "bbg", "gbbgg", "bgbgb", "ggb"])
@pytest.mark.parametrize("flags", [rc.RECON_FLAG_SYNC, 0])
def test_status_belongs_to_its_call(shape, pattern, flags):
    import paper_1311_0378_gb300.build as b
    b.build()
    H, W = shape
    rng = np.random.default_rng(H + len(pattern))
    c = rc.recon_init(0, 0, flags)
    try:
        tiles = []
        for kind in pattern:
            I = rng.integers(20, 61, size=shape).astype(np.uint8)
            J = I - 10
            if kind == "b":
                J[H - 1, W - 2] = I[H - 1, W - 2] + 1
            dI, dJ = torch.from_numpy(I).cuda(), torch.from_numpy(J).cuda()
            tiles.append((kind, I, J, dI, dJ))
        torch.cuda.synchronize()
        for kind, I, J, dI, dJ in tiles:
            st = rc.recon_run(c, dI.data_ptr(), dJ.data_ptr(), H, W, 8)
            want = rc.RECON_EMARKER if kind == "b" else rc.RECON_OK
            if flags:
                assert st == want and rc.recon_last_error_tile(c) == (0 if kind == "b" else -1)
                assert rc.recon_get_work(c, 1)[0]["visits"] >= (0 if kind == "b" else 1)
        assert rc.recon_sync(c) == want and rc.recon_last_error_tile(c) == (0 if kind == "b" else -1)
        for kind, I, J, dI, dJ in tiles:
            if kind == "g":
                np.testing.assert_array_equal(dJ.cpu().numpy(), oracle.recon(I, J, 8))
        if pattern[-1] == "g":
            assert rc.recon_get_work(c, 1)[0]["visits"] == -(-H // 64) * -(-W // 64)
    finally:
        rc.recon_free(c)
