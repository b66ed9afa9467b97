"""Distance transforms of rows of different widths at the same time, from
several threads with a context each: the row kernels' shared memory follows the
width, and no call may take another's away."""
import threading

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1311_0378_gb300 as rc  # noqa: E402


@pytest.mark.parametrize("with_site", [False, True])
def test_widths_in_parallel(with_site):
    import paper_1311_0378_gb300.build as b
    b.build()
    bad = []

    def work(W):
        B = torch.ones((2, W), dtype=torch.uint8, device="cuda")
        B[:, W // 2] = 0
        d2 = torch.empty((2, W), dtype=torch.int32, device="cuda")
        site = torch.empty_like(d2)
        torch.cuda.synchronize()
        c = rc.recon_init(0, 0, rc.RECON_FLAG_SYNC)
        for _ in range(600):
            st = rc.recon_dt(c, B.data_ptr(), d2.data_ptr(), site.data_ptr() if with_site else 0, 2, W)
            if st != rc.RECON_OK:
                bad.append((W, st))
                break
        x = torch.arange(W, device="cuda", dtype=torch.int32)
        if not (d2 == (x - W // 2) ** 2).all():
            bad.append((W, "distances"))
        rc.recon_free(c)

    threads = [threading.Thread(target=work, args=(W,)) for W in (13000, 32768, 17000, 25000)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad
