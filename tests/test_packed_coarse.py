"""CPU model of the detect kernels' coarse test on words of eight rows: it may
keep a pixel too many but never drops one that the rule keeps, and the rule
never drops a corner."""
import numpy as np
import pytest

U = np.uint32
M7, H = U(0x7F7F7F7F), U(0x80808080)


def gt_flags(a, b, t):
    """Bit 7 of each byte: |a - b| > t (t >= 128 exact, else also some == t)."""
    ab, bb = a.view(np.uint8).astype(np.int16), b.view(np.uint8).astype(np.int16)
    d = np.abs(ab - bb).astype(np.uint8).view(np.uint32)
    if t >= 128:
        return ((d & M7) + U((255 - t) * 0x01010101)) & d & H
    return ((d + U((127 - t) * 0x01010101)) | d) & H


def test_flags_miss_nothing():
    v = np.arange(256, dtype=np.uint8)
    d = np.stack(np.meshgrid(v, v, indexing="ij"), -1).reshape(-1, 2)  # two neighbouring bytes
    a = np.ascontiguousarray(np.concatenate([d, d[:, ::-1]], 1)).view(np.uint32).ravel()
    for t in range(256):
        f = gt_flags(a, np.zeros_like(a), t).view(np.uint8).reshape(-1, 4) >> 7
        x = a.view(np.uint8).reshape(-1, 4)
        assert not ((x > t) & (f == 0)).any(), t
        assert not ((x < t) & (f == 1)).any(), t
        if t >= 128:
            assert np.array_equal(f == 1, x > t)


def runs(f, n):
    return np.any([np.all([f[(s + j) % len(f)] for j in range(n)], axis=0) for s in range(len(f))], axis=0)


def test_even_runs_hold_every_arc():
    m = np.arange(1 << 16)
    bits = [((m >> i) & 1).astype(bool) for i in range(16)]
    for n in range(9, 17):
        need = 4 if n == 9 else 5 if n < 12 else 6
        assert not (runs(bits, n) & ~runs(bits[0::2], need)).any()


def perm(a, b, sel):
    s = np.stack([a, b], -1).view(np.uint8)
    return np.stack([s[:, (sel >> (4 * i)) & 7] for i in range(4)], -1).copy().view(np.uint32).ravel()


def model(img, t, n, rows, two):
    """Kept flags (rows x 128) of one warp's band: img is (rows + 6) x 132, score column 0 at column 0."""
    words = lambda r, k: np.ascontiguousarray(img[r, 4 * k:4 * k + 128]).view(np.uint32)
    push = lambda acc, f: ((acc >> U(1)) & M7) | f
    z = np.zeros(32, np.uint32)
    wv = w1 = w2 = we = z
    nw = (rows + 7) // 8
    fn, fs, fe, fne, fse, fsw, fnw = ([None] * nw for _ in range(7))
    done = lambda r: 0 <= r < rows and (r % 8 == 7 or r == rows - 1)
    C = [words(r, 0) for r in range(rows + 6)]
    R = [words(r, 1) for r in range(rows + 6)]
    R2 = [perm(c, r, 0x5432) for c, r in zip(C, R)]
    for jj in range(3, rows + 6):
        i = jj - 3
        wv = push(wv, gt_flags(C[i], C[jj], t))
        if done(i):
            fn[i // 8] = wv
        if done(i - 3):
            fs[(i - 3) // 8] = wv
        if i < rows:
            we = push(we, gt_flags(C[jj], perm(C[jj], R[jj], 0x6543), t))
            if done(i):
                fe[i // 8] = we
        if i < rows + 2:
            w1 = push(w1, gt_flags(C[jj - 2], R2[jj], t))
            w2 = push(w2, gt_flags(C[jj], R2[jj - 2], t))
            if done(i):
                fnw[i // 8], fne[i // 8] = w1, w2
            if done(i - 2):
                fse[(i - 2) // 8], fsw[(i - 2) // 8] = w1, w2
    left = lambda f: np.concatenate([[U(0xFFFFFFFF)], f[:-1]])
    out = np.zeros((rows, 128), bool)
    for w in range(nw):
        fw = perm(left(fe[w]), fe[w], 0x4321)
        f = [fn[w], fne[w], fe[w], fse[w], fs[w], perm(left(fsw[w]), fsw[w], 0x5432), fw,
             perm(left(fnw[w]), fnw[w], 0x5432)]
        if two:
            m = (f[0] | f[4]) & (f[2] | f[6])
        elif n == 9:
            x = [f[0] & f[1] & f[2], f[2] & f[3] & f[4], f[4] & f[5] & f[6], f[6] & f[7] & f[0]]
            m = ((x[0] | x[2]) & (f[3] | f[7])) | ((x[1] | x[3]) & (f[1] | f[5]))
        else:
            k = 5 if n < 12 else 6
            r3 = [f[i] & f[(i + 1) % 8] & f[(i + 2) % 8] for i in range(8)]
            m = z
            for i in range(8):
                m = m | (r3[i] & r3[(i + k - 3) % 8])
        if rows < 8:
            m = m >> U(8 - rows)
        for i in range(8 * w, min(rows, 8 * w + 8)):
            for j in range(4):
                out[i, j::4] = (m >> U(8 * j + i % 8)) & U(1)
    return out


@pytest.mark.parametrize("rows", [4, 8, 16])
@pytest.mark.parametrize("n", [9, 10, 11, 12, 16])
@pytest.mark.parametrize("t", [0, 7, 60, 127, 128, 200])
def test_band_keeps_the_rule_and_little_more(rows, n, t):
    rng = np.random.default_rng(rows * 1000 + n * 10 + t)
    for kind in range(3):
        # flat patches with steps, noise around the threshold, full-range noise
        full = rng.integers(0, 256, (rows + 6, 140))
        if kind == 0:
            full = np.repeat(np.repeat(rng.integers(0, 2, (6, 30)), 5, 0)[:rows + 6], 5, 1)[:, :140] * 255
        if kind == 1:
            full = 100 + rng.integers(0, 2, (rows + 6, 140)) * rng.integers(max(0, t - 1), t + 2, (rows + 6, 140)) % 156
        full = full.astype(np.uint8)
        img = np.ascontiguousarray(full[:, 4:136])  # score column 0 is column 4
        a = full.astype(np.int16)
        at = lambda dx, dy: np.abs(a[3 + dy:3 + dy + rows, 4 + dx:132 + dx] - a[3:3 + rows, 4:132])
        even = [(0, -3), (2, -2), (3, 0), (2, 2), (0, 3), (-2, 2), (-3, 0), (-2, -2)]
        need = 4 if n == 9 else 5 if n < 12 else 6
        got = model(img, t, n, rows, False)
        want = runs([at(*d) > t for d in even], need)
        loose = runs([at(*d) >= t for d in even], need)
        assert not (want & ~got).any()
        assert not (got & ~loose)[:, 4:].any()  # lane 0 keeps more at its left edge
        if n < 12:
            f = [at(*d) > t for d in ((0, -3), (3, 0), (0, 3), (-3, 0))]
            assert not ((f[0] | f[2]) & (f[1] | f[3]) & ~model(img, t, n, rows, True)).any()
