"""Several threads at once, each on its own stream: builds and operators of models of
different sizes succeed and give the single-threaded results."""
import threading

import pytest

SHAPES = [(32, 32, 48, 192, 11), (20, 12, 17, 256, 71), (64, 66, 47, 188, 9), (150, 90, 51, 192, 7)]


def run_threads(n, work):
    errors = []

    def guard(i):
        try:
            work(i)
        except Exception as e:  # reported by the main thread
            errors.append((i, repr(e)))

    threads = [threading.Thread(target=guard, args=(i,)) for i in range(n)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors[:3]


@pytest.mark.gpu
@pytest.mark.parametrize("form", ["OAM_PREC_FP32", "OAM_PREC_BF16X3", "OAM_PREC_FFT"])
def test_operators_from_threads(form):
    import torch

    from paper_2009_10173_gb300 import binding as B
    from paper_2009_10173_gb300 import configs
    from paper_2009_10173_gb300.model import Model
    jobs = []
    for px, py, nz, nt, win in SHAPES:
        m = Model(configs.scaled(configs.TINY_32, px=px, py=py, nz=nz, nt=nt, win=win, dx_m=4e-6, dy_m=4e-6,
                                 n_patches=200), precision=getattr(B, form))
        H = torch.randn(m.vol_shape, device="cuda")
        f = m.forward(H).clone()
        jobs.append((m, H, f, m.adjoint(f).clone()))
    torch.cuda.synchronize()

    def work(i):
        m, H, f, a = jobs[i]
        st = torch.cuda.Stream()
        with torch.cuda.stream(st):
            for _ in range(30):
                g = m.forward(H)
                b = m.adjoint(g)
                st.synchronize()
                assert torch.equal(g, f) and torch.equal(b, a)

    run_threads(len(jobs), work)
    for job in jobs:
        job[0].close()


@pytest.mark.gpu
def test_builds_from_threads():
    """Windows of 187 taps and more: the spectrum build's shared memory is above the 48 KB default."""
    import torch

    from paper_2009_10173_gb300 import binding as B
    from paper_2009_10173_gb300 import configs
    from paper_2009_10173_gb300.model import Model

    def work(i):
        cfg = configs.scaled(configs.TINY_32, px=4, py=4, nz=2, nt=512, win=(187, 255, 203, 239)[i], dx_m=2e-6,
                             dy_m=2e-6, n_patches=40)
        st = torch.cuda.Stream()
        with torch.cuda.stream(st):
            for _ in range(25):
                Model(cfg, precision=B.OAM_PREC_FFT, stream=st.cuda_stream).close()

    run_threads(4, work)
