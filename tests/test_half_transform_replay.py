"""CPU replay of engine 50's half-length sine transforms (csrc/solve_stream.cu):
the kernels' shared-memory, table, position and scratch index expressions,
restated in Python and run on the numbers they move, so that each pass writes
every element it later reads, stays inside its buffers, and the three passes
together are the sine sums of Eqs. ifft-1/ffft-1.  Both engines' arithmetic is
FP64 here, so the comparison is to 1e-12 (a few roundings times log N)."""
import numpy as np
import pytest

NAN = complex(np.nan, np.nan)


def geo(lg):
    L = 1 << lg
    G = L // 16
    H = G // 16
    HC = 1 if H <= 16 else 4
    HB = H // HC
    P2 = H + 1
    RP = 17 if H == 1 else 16 * P2 + (H if H <= 8 else 0)
    PT = G // 2 + 2
    T2 = 8 * PT
    T3 = T2 + 15 * H
    return dict(L=L, N=L // 2, G=G, H=H, HC=HC, HB=HB, P2=P2, RP=RP, BUF=9 * RP, PT=PT, T2=T2,
                T3=T3, TABLE=T3 + (H if HC > 1 else 0), TP=9 * H)


def table(lg):
    g = geo(lg)
    tab = np.full(g["TABLE"], NAN)
    w = lambda num, den: np.exp(-2j * np.pi * (num % den) / den)  # noqa: E731
    for s in range(1, 9):
        for t in range(g["PT"]):
            tab[(s - 1) * g["PT"] + t] = w(t * s, g["L"])
    for q in range(1, 16):
        for j in range(g["H"]):
            tab[g["T2"] + (q - 1) * g["H"] + j] = w(q * j, g["G"])
    if g["HC"] > 1:
        for p in range(g["HB"]):
            for c in range(4):
                tab[g["T3"] + 4 * p + c] = w(p * c, g["H"])
    assert not np.isnan(tab).any()
    return tab


def dft(v):
    """R-point DFT over the first axis."""
    R = v.shape[0]
    k = np.arange(R)
    return np.exp(-2j * np.pi * (np.outer(k, k) % R) / R) @ v


def put(buf, idx, val):
    """Every index in bounds, none written twice by one pass."""
    idx = np.asarray(idx)
    assert idx.min() >= 0 and idx.max() < len(buf)
    assert len(np.unique(idx)) == idx.size
    buf[idx.ravel()] = np.asarray(val).ravel()


def get(buf, idx):
    idx = np.asarray(idx)
    assert idx.min() >= 0 and idx.max() < len(buf)
    v = buf[idx]
    assert not np.isnan(v).any()      # written before
    return v


def row_k(g):
    """[i, j]: the index k of register i of thread j of a row."""
    j = np.arange(g["H"])[None, :]
    i = np.arange(16)[:, None]
    if g["HC"] == 1:
        return j + (i // g["H"]) * g["H"] + 16 * (i % g["H"])
    p1 = (j >> 4) + (g["H"] // 16) * (i >> 2)
    return (j & 15) + 16 * (p1 + g["HB"] * (i & 3))


def pass_fwd(x, buf, tab, g):
    """x[r, t], t = 0..G/2"""
    t = np.arange(g["G"] // 2 + 1)
    Y = dft(x)
    both = (t > 0) & (t < g["G"] // 2)
    idx, val = [], []
    for s in range(9):
        w = np.ones(len(t)) if s == 0 else get(tab, (s - 1) * g["PT"] + t)
        idx += [s * g["RP"] + t, (s * g["RP"] + g["G"] - t)[both]]
        val += [Y[s] * w, (-Y[(16 - s) & 15] * np.conj(w))[both]]
    put(buf, np.concatenate(idx), np.concatenate(val))


def pass_bwd(buf, tab, g):
    t = np.arange(g["G"] // 2 + 1)
    tm = np.where(t == 0, 0, g["G"] - t)
    v = np.zeros((16, len(t)), complex)
    v[0] = get(buf, t)
    for s in range(1, 9):
        w = get(tab, (s - 1) * g["PT"] + t)
        v[s] = get(buf, s * g["RP"] + t) * w
        if s < 8:
            v[16 - s] = -get(buf, s * g["RP"] + tm) * np.conj(w)
    return dft(v)


def row_fwd(v, row, tab, g):
    """v[r, j] natural -> v[i, j] in row_k order; row: scratch of RP elements"""
    H, P2, HB = g["H"], g["P2"], g["HB"]
    j = np.arange(H)[None, :]
    v = dft(v)
    if H == 1:
        return v
    q = np.arange(1, 16)[:, None]
    v[1:] *= get(tab, g["T2"] + (q - 1) * H + j)
    q = np.arange(16)[:, None]
    row[:] = NAN
    put(row, q * P2 + j, v)
    out = np.zeros_like(v)
    if g["HC"] == 1:
        for b in range(16 // H):
            e = np.arange(H)[:, None]
            out[b * H:(b + 1) * H] = dft(get(row, (j + H * b) * P2 + e))
        return out
    j = j[0]
    q = j & 15
    e = np.arange(HB)[:, None]
    for b in range(16 // HB):
        c = (j >> 4) + (H // 16) * b
        u = dft(get(row, q * P2 + c + 4 * e))
        u[1:] *= get(tab, g["T3"] + e[1:] * 4 + c)
        put(row, q * P2 + c + 4 * e, u)
    e = np.arange(4)[:, None]
    for b in range(4):
        p = (j >> 4) + (H // 16) * b
        out[4 * b:4 * b + 4] = dft(get(row, q * P2 + 4 * p + e))
    return out


def row_bwd(v, row, tab, g):
    H, P2, HB = g["H"], g["P2"], g["HB"]
    j = np.arange(H)[None, :]
    if H == 1:
        return dft(v)
    v = v.copy()
    row[:] = NAN
    if g["HC"] == 1:
        for b in range(16 // H):
            e = np.arange(H)[:, None]
            put(row, (j + H * b) * P2 + e, dft(v[b * H:(b + 1) * H]))
    else:
        j1 = j[0]
        q = j1 & 15
        e = np.arange(4)[:, None]
        for b in range(4):
            p = (j1 >> 4) + (H // 16) * b
            put(row, q * P2 + 4 * p + e, dft(v[4 * b:4 * b + 4]))
        e = np.arange(HB)[:, None]
        for b in range(16 // HB):
            c = (j1 >> 4) + (H // 16) * b
            u = get(row, q * P2 + c + 4 * e)
            u[1:] *= get(tab, g["T3"] + e[1:] * 4 + c)
            put(row, q * P2 + c + 4 * e, dft(u))
    q = np.arange(16)[:, None]
    v = get(row, q * P2 + j)
    v[1:] *= get(tab, g["T2"] + (q[1:] - 1) * H + j)
    return dft(v)


def columns(g):
    """[r, t]: the element of register r of thread t in the radix-16 pass."""
    t = np.arange(g["G"] // 2 + 1)
    return np.array([t + g["G"] * r if r < 8 else (16 - r) * g["G"] - t for r in range(16)])


def load_natural(z, g):
    c = columns(g)
    assert c.min() >= 0 and c.max() <= g["N"]
    zz = np.concatenate([z, [0]])
    return np.where(np.arange(16)[:, None] < 8, zz[c], -zz[c])


def store_natural(v, g):
    out = np.full(g["N"], NAN)
    c = columns(g)
    half = g["G"] // 2
    idx, val = [], []
    for r in range(16):
        for t in range(half + 1):
            if (t == 0 and r % 8 == 0) or (r >= 8 and t in (0, half)):
                continue
            idx.append(c[r, t])
            val.append(v[r, t] if r < 8 else -v[r, t])
    put(out, idx, val)
    out[0] = 0
    assert not np.isnan(out).any()
    return out


def rows_of(buf, g):
    j = np.arange(g["H"])[None, :]
    r = np.arange(16)[:, None]
    return [get(buf, s * g["RP"] + j + g["H"] * r) for s in range(9)]


def dst(z):
    n = len(z)
    ext = np.concatenate([z, [0], -z[:0:-1]])
    return np.fft.fft(ext)[:n]


def position(g):
    """position of mode m, m = 0..N-1"""
    m = np.arange(g["N"])
    return (m % 16) * (g["G"] // 2) + m // 16


@pytest.mark.parametrize("lg", range(8, 15))
def test_half_transforms(lg):
    g, tab = geo(lg), table(lg)
    assert g["G"] // 2 + 1 <= g["TP"]            # the pass's butterflies fit the pair's threads
    rng = np.random.default_rng(lg)
    z = rng.normal(size=g["N"]) + 1j * rng.normal(size=g["N"])
    z[0] = 0
    Z = dst(z)
    scale = np.abs(Z).max()
    k = row_k(g)
    assert np.array_equal(np.sort(k.ravel()), np.arange(g["G"]))
    # forward: pass, rows, modes by position
    buf = np.full(g["BUF"], NAN)
    pass_fwd(load_natural(z, g), buf, tab, g)
    by_pos = np.full(g["N"], NAN)
    modes = []
    for s, u in enumerate(rows_of(buf, g)):
        v = row_fwd(u, buf[s * g["RP"]:(s + 1) * g["RP"]], tab, g)
        modes.append(v)
        low = k < g["G"] // 2
        pos = np.where(low, s * (g["G"] // 2) + k, (16 - s) * (g["G"] // 2) + g["G"] - 1 - k)
        keep = low if s in (0, 8) else np.ones_like(low)
        put(by_pos, pos[keep], np.where(low, v, -v)[keep])
        m = s + 16 * k
        assert np.abs(v - np.where(m < g["N"], Z[np.minimum(m, g["N"] - 1)], 0))[m < g["N"]].max() < 1e-12 * scale
    assert np.abs(by_pos[position(g)] - Z).max() < 1e-12 * scale
    # y pass: the rows backward, then the pass (no scaling between)
    buf[:] = NAN
    for s, v in enumerate(modes):
        row = buf[s * g["RP"]:(s + 1) * g["RP"]]
        u = row_bwd(v, row, tab, g)
        row[:] = NAN
        put(row, np.arange(g["H"])[None, :] + g["H"] * np.arange(16)[:, None], u)
    got = store_natural(pass_bwd(buf, tab, g), g)
    want = dst(Z)
    assert np.abs(got - want).max() < 1e-12 * np.abs(want).max()
    # x inverse: rows from positions, then the pass
    buf[:] = NAN
    by_pos[0] = 0
    for s in range(9):
        kk = np.arange(g["H"])[None, :] + g["H"] * np.arange(16)[:, None]
        r = np.arange(16)[:, None]
        half = g["G"] // 2
        pos = np.where(r < 8, s * half + kk, (g["G"] - kk) if s == 0 else (16 - s) * half + g["G"] - 1 - kk)
        zero = (s == 0) & ((kk == 0) | (kk == half))
        pos = np.where(zero, 0, pos)
        u = np.where(zero, 0, np.where(r < 8, 1, -1) * get(by_pos, pos))
        row = buf[s * g["RP"]:(s + 1) * g["RP"]]
        v = row_fwd(u, row, tab, g)
        row[:] = NAN
        put(row, k, v)
    got = store_natural(pass_bwd(buf, tab, g), g)
    assert np.abs(got - want).max() < 1e-12 * np.abs(want).max()


@pytest.mark.parametrize("layers", [1, 2])
@pytest.mark.parametrize("mx,my", [(128, 128), (128, 256), (256, 128), (512, 1024), (8192, 128), (128, 8192)])
def test_scratch_layouts(mx, my, layers):
    """tr and work fit their planes, the 4-value runs start on 16 bytes, and
    the inverse x pass writes only grid rows whose scratch it has read."""
    ld, ld_tr = (mx // 32 + 1) * 32, (my // 32 + 1) * 32
    assert ld % 4 == 0 and ld_tr % 4 == 0
    if layers == 1:
        assert 2 * ((mx // 2 - 1) * ld_tr + my - 1) + 1 < (mx + 1) * ld_tr
        last = ld + 2 * ((my // 2 - 1) * ld + mx - 1) + 1
        assert last < (my + 1) * ld
        # pair p's scratch lies in rows 1 + 2 p and 2 + 2 p of the array, the rows it writes
        for p in (0, my // 2 - 1):
            lo, hi = ld + 2 * p * ld, ld + 2 * (p * ld + mx - 1) + 1
            assert lo // ld == 1 + 2 * p and hi // ld <= 2 + 2 * p
    else:
        assert 2 * ((mx - 1) * ld_tr + my - 2) + 1 < 2 * (mx + 1) * ld_tr
        assert ld + 2 * ((my - 2) * ld + mx - 1) + 1 < 2 * (my + 1) * ld
