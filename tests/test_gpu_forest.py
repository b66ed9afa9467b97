"""The region-merging engine (what a context runs with its default settings)
against the CPU oracle, bit for bit: sizes around its 64 x 64 blocks, images
that stress its parts (plateaus, ramps, the most basins a block can hold, so
that its pass table overflows), every operation, odd row lengths and
unaligned buffers, and agreement with the wavefront engine. R is unique, so
the tolerance is zero."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1311_0378_gb300 as rc  # noqa: E402


@pytest.fixture(scope="module")
def ctx():
    import paper_1311_0378_gb300.build as b
    b.build()
    c = rc.recon_init(0, 0, rc.RECON_FLAG_SYNC)
    yield c
    rc.recon_free(c)


def image(kind, H, W, rng):
    y, x = np.mgrid[0:H, 0:W]
    if kind == "noise":
        return rng.integers(20, 61, size=(H, W)).astype(np.uint8)
    if kind == "walls":
        return np.where(rng.random((H, W)) < 0.3, 0, rng.integers(0, 256, size=(H, W))).astype(np.uint8)
    if kind == "binary":
        return np.where(rng.random((H, W)) < 0.6, 255, 0).astype(np.uint8)
    if kind == "flat":
        return np.full((H, W), 77, np.uint8)
    if kind == "ramp":
        return ((3 * x + 5 * y) % 256).astype(np.uint8)
    if kind == "steps":
        return (16 * ((x // 7 + y // 5) % 16)).astype(np.uint8)
    # "board": every second pixel a top of its own height, low pixels between
    # them: the most basins (and passes) a block can have
    hi = rng.integers(128, 256, size=(H, W))
    lo = rng.integers(1, 128, size=(H, W))
    return np.where((x + y) % 2 == 0, hi, lo).astype(np.uint8)


def markers(I, rng):
    H, W = I.shape
    border = np.zeros_like(I)
    border[0, :], border[-1, :], border[:, 0], border[:, -1] = I[0, :], I[-1, :], I[:, 0], I[:, -1]
    one = np.zeros_like(I)
    one[H // 2, W // 3] = I[H // 2, W // 3]
    return [np.maximum(I.astype(int) - 10, 0).astype(np.uint8), border, one,
            np.where(rng.random((H, W)) < 0.02, I, 0).astype(np.uint8),
            np.minimum(I, rng.integers(0, 256, size=(H, W))).astype(np.uint8)]


def put(a, lead=0, pitch=None):
    """A device copy with `lead` bytes before it and rows `pitch` bytes apart;
    returns (buffer, address, host copy of the buffer)."""
    H, W = a.shape
    pitch = pitch or W
    host = np.full(lead + H * pitch + 16, 0x5A, np.uint8)
    v = host[lead:lead + H * pitch].reshape(H, pitch)
    v[:, :W] = a
    t = torch.from_numpy(host).cuda()
    torch.cuda.synchronize()
    return t, t.data_ptr() + lead, host


KINDS = ["noise", "walls", "binary", "flat", "ramp", "steps", "board"]
SHAPES = [(1, 1), (1, 65), (130, 1), (5, 63), (63, 64), (64, 64), (65, 66), (128, 129), (200, 321)]


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("shape", SHAPES)
def test_matches_oracle(ctx, kind, shape):
    H, W = shape
    rng = np.random.default_rng(H * 1000 + W + KINDS.index(kind))
    I = image(kind, H, W, rng)
    tiles, keep, wants = [], [], []
    for J in markers(I, rng):
        for conn in (4, 8):
            for op in (rc.RECON_OP_DILATE, rc.RECON_OP_ERODE):
                a, b = (I, J) if op == rc.RECON_OP_DILATE else (255 - I, 255 - J)
                wants.append(oracle.recon(a, b, conn) if op == rc.RECON_OP_DILATE else oracle.recon_erode(a, b, conn))
                dI, dJ = put(a), put(b)
                keep.append((dI, dJ))
                tiles.append((dI[1], dJ[1], H, W, W, conn, op))
    for conn in (4, 8):
        wants.append(oracle.fill_holes(I, conn))
        dI, dJ = put(I), put(np.full_like(I, 0xA5))
        keep.append((dI, dJ))
        tiles.append((dI[1], dJ[1], H, W, W, conn, rc.RECON_OP_FILL_HOLES))
    rc.check(rc.recon_batch(ctx, tiles), "recon_batch")
    for k, ((dI, dJ), want) in enumerate(zip(keep, wants)):
        np.testing.assert_array_equal(dJ[0].cpu().numpy()[:H * W].reshape(H, W), want, err_msg="tile %d" % k)
    assert all(w["visits"] == -(-H // 64) * -(-W // 64) for w in rc.recon_get_work(ctx, len(tiles)))


@pytest.mark.parametrize("lead,pad", [(0, 0), (1, 0), (2, 3), (3, 64), (0, 7), (8, 16)])
def test_any_alignment_and_pitch(ctx, lead, pad):
    """Rows and bases on any byte: nothing outside the image is written."""
    H, W = 141, 197
    rng = np.random.default_rng(lead * 10 + pad)
    I = image("noise", H, W, rng)
    J = markers(I, rng)[1]
    dI, dJ = put(I, (lead + 1) % 4, W + pad), put(J, lead, W + pad)
    rc.check(rc.recon_batch(ctx, [(dI[1], dJ[1], H, W, W + pad, 8)]), "recon_batch")
    got = dJ[0].cpu().numpy()
    want = dJ[2].copy()
    want[lead:lead + H * (W + pad)].reshape(H, W + pad)[:, :W] = oracle.recon(I, J, 8)
    np.testing.assert_array_equal(got, want)


def test_violation_in_one_tile_leaves_the_others(ctx):
    rng = np.random.default_rng(3)
    pairs = [(image("noise", 150, 170, rng),) for _ in range(3)]
    pairs = [(I, markers(I, rng)[0]) for (I,) in pairs]
    pairs[1][1][100, 160] = 61
    dev = [(put(I), put(J)) for I, J in pairs]
    assert rc.recon_batch(ctx, [(a[1], b[1], 150, 170, 170, 8) for a, b in dev]) == rc.RECON_EMARKER
    assert rc.recon_last_error_tile(ctx) == 1
    for k in (0, 2):
        np.testing.assert_array_equal(dev[k][1][0].cpu().numpy()[:150 * 170].reshape(150, 170),
                                      oracle.recon(*pairs[k], 8))


@pytest.mark.parametrize("conn", [4, 8])
def test_agrees_with_the_wavefront_engine(conn):
    """A large border-seeded tile through both engines (an explicit schedule
    asks for the wavefront engine)."""
    rng = np.random.default_rng(conn)
    H, W = 1500, 2111
    I = image("noise", H, W, rng)
    J = markers(I, rng)[1]
    c = rc.recon_init(0, 0, rc.RECON_FLAG_SYNC)
    try:
        dI, d1, d2 = put(I), put(J), put(J)
        rc.check(rc.recon_batch(c, [(dI[1], d1[1], H, W, W, conn)]), "merging")
        rc.check(rc.recon_batch_ex(c, [(dI[1], d2[1], H, W, W, conn)], [1], [0]), "wavefront")
        assert torch.equal(d1[0], d2[0])
    finally:
        rc.recon_free(c)
