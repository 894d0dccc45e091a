"""The split-BF16 form's line transforms (``csrc/mix_lines.cu``, ``csrc/op_tc.cu``).

On the CPU: segments of a line cover every output row once, no circular wrap
reaches an output row, and the mark words' arithmetic finds exactly the rows
whose window holds a marked row.  On the GPU, against the FP64 oracle at the
split-BF16 operators' tolerance (1e-4): grids of one row, fewer rows than the
half window, a line in two and three segments, and exact zeros and NaN where
the window of a position holds no input or a non-finite one.
"""
import numpy as np
import pytest

LINE_MAX = 512


def plan(py, R, sizes):
    halo = min(R, py - 1)
    if py + halo <= LINE_MAX:
        return min(p for p in sizes if p >= py + halo), halo, 1, py
    valid = LINE_MAX - 2 * halo
    return LINE_MAX, halo, -(-py // valid), valid


def mix_sizes():
    from test_mixed_radix import sizes
    return [p for p, _, _ in sizes()]


@pytest.mark.parametrize("py,R", [(1, 5), (2, 30), (20, 30), (200, 30), (482, 30), (483, 30), (513, 0), (900, 64),
                                  (2000, 1)])
def test_segments_give_the_correlation(py, R):
    P, halo, segs, valid = plan(py, R, mix_sizes())
    rng = np.random.Generator(np.random.PCG64(py + R))
    x = rng.standard_normal(py)
    w = rng.standard_normal(R + 1)  # even weights w[|b|]
    want = sum(w[abs(b)] * np.array([x[y + b] if 0 <= y + b < py else 0.0 for y in range(py)])
               for b in range(-R, R + 1))
    f = np.arange(P)
    spec = sum(((1 if b == 0 else 2) * w[b] * np.cos(2 * np.pi * f * b / P) for b in range(halo + 1)), np.zeros(P))
    got, written = np.zeros(py), np.zeros(py, int)
    for g in range(segs):
        first = g * valid - halo if segs > 1 else 0
        seg = np.array([x[first + i] if 0 <= first + i < py else 0.0 for i in range(P)])
        out = np.fft.ifft(np.fft.fft(seg) * spec).real
        for y in range(g * valid, min(py, (g + 1) * valid)):
            assert 0 <= y - first < P
            got[y] = out[y - first]
            written[y] += 1
    assert (written == 1).all()
    assert np.allclose(got, want, atol=1e-11 * max(1, np.abs(want).max()))


def grow(words, R):  # as grow_marks in op_tc.cu, of one column
    out = []
    for j in range(len(words)):
        win = [words[j + i - 2] if 0 <= j + i - 2 < len(words) else 0 for i in range(5)]
        bits = 0
        for lane in range(32):
            for i in range(5):
                lo, hi = max(lane - R - 32 * (i - 2), 0), min(lane + R - 32 * (i - 2), 31)
                if lo <= hi and win[i] & (0xffffffff << lo) & (0xffffffff >> (31 - hi)):
                    bits |= 1 << lane
        out.append(bits)
    return out


@pytest.mark.parametrize("py,R", [(1, 5), (31, 0), (32, 1), (200, 30), (513, 3), (900, 64)])
def test_mark_words(py, R):
    P, halo, segs, valid = plan(py, R, mix_sizes())
    rng = np.random.Generator(np.random.PCG64(py))
    for density in (0.0, 0.005, 0.1):
        marked = rng.random(py) < density
        words = [0] * ((py + 31) // 32)
        for g in range(segs):  # mark_rows: 32 points of a segment as one shifted word
            y0 = g * valid - halo if segs > 1 else 0
            for w in range((P + 31) // 32):
                bits = sum(1 << t for t in range(32) if 32 * w + t < P and 0 <= y0 + 32 * w + t < py
                           and marked[y0 + 32 * w + t])
                yw, s = (y0 + 32 * w) >> 5, (y0 + 32 * w) & 31
                lo, hi = (bits << s) & 0xffffffff, bits >> (32 - s) if s else 0
                if lo:
                    assert 0 <= yw
                    words[yw] |= lo
                if hi:
                    words[yw + 1] |= hi
        assert [bool(words[y >> 5] >> (y & 31) & 1) for y in range(py)] == list(marked)
        grown = grow(words, R)
        for y in range(py):
            assert bool(grown[y >> 5] >> (y & 31) & 1) == marked[max(0, y - R):y + R + 1].any()
        for g in range(segs):  # the words an inverse block holds
            ya, yb = g * valid, min(py, (g + 1) * valid)
            assert ((yb - 1) >> 5) - (ya >> 5) + 1 <= P // 32 + 2


# ------------------------------------------------------------------ GPU
def build(**over):
    from paper_2009_10173_gb300 import binding as B
    from paper_2009_10173_gb300 import configs
    from paper_2009_10173_gb300.model import Model
    cfg = configs.scaled(configs.TINY_32, n_patches=200, **over)
    return cfg, Model(cfg, precision=B.OAM_PREC_BF16X3)


@pytest.mark.gpu
@pytest.mark.parametrize("px,py,win,nz,nt", [(33, 1, 11, 9, 128), (5, 3, 11, 20, 128), (64, 96, 9, 48, 192),
                                             (2, 511, 3, 9, 128), (3, 520, 5, 9, 128), (130, 1100, 3, 5, 128),
                                             (257, 17, 7, 33, 160), (7, 600, 1, 9, 128)])
def test_grids_match_oracle(px, py, win, nz, nt):
    import oracle
    import torch

    from paper_2009_10173_gb300 import inputs
    cfg, m = build(px=px, py=py, win=win, nz=nz, nt=nt)
    S = oracle.slab(cfg)
    H = inputs.gaussian(m.vol_shape, 5).astype(np.float32)
    s = inputs.gaussian(m.sig_shape, 6).astype(np.float32)
    f = m.forward(torch.from_numpy(H).cuda()).double().cpu().numpy()
    a = m.adjoint(torch.from_numpy(s).cuda()).double().cpu().numpy()
    m.close()
    for got, want in ((f, oracle.forward(S, H.astype(np.float64))), (a, oracle.adjoint(S, s.astype(np.float64)))):
        assert np.linalg.norm(got - want) <= 1e-4 * np.linalg.norm(want)


@pytest.mark.gpu
@pytest.mark.parametrize("py", [40, 560])
def test_zeros_and_non_finite_values_stay_in_their_window(py):
    import torch
    cfg, m = build(px=24, py=py, win=7, nz=16, nt=128)
    R, H = 3, torch.zeros(m.vol_shape, device="cuda")
    for y, x, k, v in ((2, 3, 4, 1.0), (py - 2, 20, 9, float("nan")), (py // 2, 12, 0, float("inf"))):
        H[y, x, k] = v
    first = m.forward(H)
    bad, some = ~torch.isfinite(H).all(-1), (H != 0).any(-1)
    grow = lambda t: torch.nn.functional.max_pool2d(t.float()[None, None], 2 * R + 1, 1, R)[0, 0] > 0
    assert torch.equal(torch.isnan(first).any(-1), grow(bad))
    live = grow(some) & ~grow(bad)
    assert (first[~grow(some)] == 0).all() and (first[live] != 0).any(-1).all()
    # the marks of one application do not reach the next
    H.nan_to_num_(0.0, 0.0, 0.0)
    again = m.forward(H)
    assert torch.isfinite(again).all() and (again[~grow((H != 0).any(-1))] == 0).all()
    assert torch.equal(again[live], first[live])
    m.close()


@pytest.mark.gpu
@pytest.mark.parametrize("scale", [1e-30, 1e-10, 1e10, 1e30])
def test_operand_scaling(scale):
    """The iterate is brought into the 16-bit terms' range by a power of two per
    frequency: inputs of any magnitude give the scaled result, also next to each other."""
    import torch

    from paper_2009_10173_gb300 import inputs
    cfg, m = build(px=40, py=36, win=11, nz=40, nt=192)
    for shape, op in ((m.vol_shape, m.forward), (m.sig_shape, m.adjoint)):
        x = torch.from_numpy(inputs.gaussian(shape, 9).astype(np.float32)).cuda()
        want = op(x).double()
        got = op(x * scale).double() / scale
        assert float((got - want).norm() / want.norm()) <= 2e-5  # two runs within the form's error
        torch.testing.assert_close(op(torch.zeros_like(x)).abs().max().item(), 0.0)
    m.close()
