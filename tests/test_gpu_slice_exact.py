"""One FP64 digit transform against exact integer sums.

Lines and matrix rows are integers below 2^62 in units of the row's scale, so
their base-256 digits are exact and the level sums S_L (sums of digit products u + v =
L) can be formed exactly here.  The kernel adds S_0 .. S_7 and rounds once; it
leaves out S_8 .. S_14.

  cancel   random entries whose products cancel to 2^-12 of the scale: the FP64
           rounding of a result is then far below a digit, and a lost digit plane
           shows (2^-52.6 of the scale, root mean square).  The sums left out are
           2^-58 of it (S_8: 7 n products of digits of root mean square 74,
           in units of 2^-76), so six standard deviations are below 2^-55.
  extreme  digits 124 .. 127 of one sign in the planes 0 (half of that) to 5: |S_4|
           comes within 5% of its bound 2^24, where FP32 sums of integers are still
           exact, and has odd values.  Against the same sums
           formed here, the result is one rounding (S_5 above 2^24 may be off by
           one unit, 2^-6 of the result's half spacing, and the integer sum is cut
           below its 61st bit): one unit in the last place.
"""
import ctypes as C
import os
import random
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
BITS = 62


@pytest.fixture(scope="module")
def check(tmp_path_factory):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1107_2461_gb300 import build
    lib = build.build()
    out = str(tmp_path_factory.mktemp("slice") / "slice_transform_check.so")
    subprocess.run([build.nvcc()] + build.ARCH + build.NVCC_FLAGS +
                   ["-I" + build.CSRC, "-shared", os.path.join(HERE, "slice_transform_check.cu"), lib, "-o", out,
                    "-Xlinker", "-rpath," + os.path.dirname(lib)], check=True)
    so = C.CDLL(out)
    fn = so.slice_transform_check
    fn.restype = C.c_int
    fn.argtypes = [C.c_void_p, C.c_int, C.c_void_p, C.c_void_p, C.c_longlong, C.c_int, C.c_longlong, C.c_int]
    fn.prepare_status = so.slice_prepare_status
    return fn


def digits(v):
    """Signed base-256 digits, the leading one first; v any integer below 2^62 in magnitude."""
    d = []
    for _ in range(7):
        low = (v + 128) % 256 - 128
        d.append(low)
        v = (v - low) >> 8
    return [v] + d[::-1]


def to_double(v):
    """v 2^-62 as a double; v has at most 53 significant bits."""
    x = float(v)
    assert int(x) == v
    return x * 2.0**-BITS


def fit(v):
    """v cut to 53 significant bits."""
    cut = max(0, abs(v).bit_length() - 53)
    return (v >> cut) << cut


def cancel_data(rnd, n, lines, perturb_lines):
    """Rows (a, -a (1 + 2^-12 e)) against lines (x, x), or the other way round
    (the digits of the repeated factor cancel: each side takes its turn)."""
    h = n // 2

    def one():
        return fit(rnd.randrange(-(2**62) + 1, 2**62) >> rnd.randrange(10))  # the smaller ones fill the last digits

    perturbed, repeated = [], []
    for _ in range(lines if perturb_lines else n):
        a = [one() for _ in range(h)]
        perturbed.append(a + [fit(-(v - v * rnd.randrange(-256, 257) // 2**20)) for v in a] + [0] * (n - 2 * h))
    for _ in range(n if perturb_lines else lines):
        x = [one() for _ in range(h)]
        repeated.append(x + x + [0] * (n - 2 * h))
    return (repeated, perturbed) if perturb_lines else (perturbed, repeated)


def extreme_data(rnd, n, lines):
    def one(sign):
        v = rnd.randrange(62, 64)
        for _ in range(5):
            v = v * 256 + rnd.randrange(124, 128)
        return sign * v * 256**2

    T = [[one(1 if k % 2 else -1) for _ in range(n)] for k in range(n)]
    X = [[one(1 if r % 3 else -1) for _ in range(n)] for r in range(lines)]
    return T, X


# one step of 16 columns and its edges, the edges of a 128-mode tile, the largest;
# few lines (32 per item) and many (64 per item, several items per CTA)
@pytest.mark.parametrize("n,lines", [(2, 5), (16, 40), (17, 33), (128, 70), (129, 9), (256, 33), (64, 9800),
                                     (256, 5000)])
@pytest.mark.parametrize("kind", ["cancel", "extreme"])
@pytest.mark.parametrize("contiguous", [True, False])
def test_against_exact_sums(check, n, lines, kind, contiguous):
    import torch
    rnd = random.Random(n * 1000 + lines)
    distinct = min(lines, 12)
    T, X = cancel_data(rnd, n, distinct, not contiguous) if kind == "cancel" else extreme_data(rnd, n, distinct)
    # every line is one of the distinct ones, scaled by a power of two of its own
    which = np.array([rnd.randrange(distinct) for _ in range(lines)])
    power = np.array([rnd.randrange(-200, 200) for _ in range(lines)])
    which[:distinct] = np.arange(distinct)
    xd = np.array([[to_double(v) for v in x] for x in X])
    x_all = np.ldexp(xd[which], power[:, None])
    row = np.array([rnd.randrange(-30, 30) for _ in range(n)])
    t_all = np.ldexp(np.array([[to_double(v) for v in t] for t in T]), row[:, None])
    width = 7
    if contiguous:
        x_in = x_all
    else:  # [slab][n][width], the last slab padded with zero lines
        slabs = -(-lines // width)
        pad = np.zeros((slabs * width, n))
        pad[:lines] = x_all
        x_in = pad.reshape(slabs, width, n).transpose(0, 2, 1)
    x_dev = torch.from_numpy(np.ascontiguousarray(x_in)).cuda()
    t_dev = torch.from_numpy(np.ascontiguousarray(t_all)).cuda()
    y_dev = torch.full_like(x_dev, 3.0)  # overwritten
    total = lines if contiguous else x_in.shape[0] * width
    torch.cuda.synchronize()

    def apply(accumulate):
        assert check(t_dev.data_ptr(), n, x_dev.data_ptr(), y_dev.data_ptr(), total, int(contiguous), width,
                     accumulate) == 0
        y = y_dev.cpu().numpy()
        return y if contiguous else y.transpose(0, 2, 1).reshape(-1, n)[:lines]

    y = apply(0)
    # the exponents taken out again, in units of the two scales
    got = np.ldexp(y, -power[:, None] - row[None, :])
    Tm, Xm = np.array(T, dtype=object), np.array(X, dtype=object)
    if kind == "cancel":
        want = Xm @ Tm.T  # exact, in units of 2^-124
        # a row's or line's scale: the power of two above its largest entry
        scale = np.exp2(np.array([[max(map(abs, x)).bit_length() + max(map(abs, t)).bit_length() - 124 for t in T]
                                  for x in X]))
        for r in range(distinct):
            for k in range(n):
                err = abs(int(got[r, k] * 2.0**1000) - (int(want[r, k]) << 876))
                tol = 2.0**-55 * scale[r, k] + 2.0**-53 * abs(got[r, k])
                assert err <= int(tol * 2.0**1000), (r, k, err * 2.0**-1000 / scale[r, k])
    else:
        td = np.array([[digits(v) for v in t] for t in T], dtype=np.int64)  # [k][j][u]
        xg = np.array([[digits(v) for v in x] for x in X], dtype=np.int64)  # [r][j][v]
        want = np.zeros((distinct, n), dtype=object)
        for level in range(8):
            s = sum(xg[:, :, v] @ td[:, :, level - v].T for v in range(level + 1))
            assert level > 4 or np.abs(s).max() <= 2**24
            if level == 4 and n == 256:
                assert np.abs(s).max() > 0.95 * 2**24 and (s % 2).any()
            want = want + s.astype(object) * 256 ** (14 - level)
        for r in range(distinct):
            for k in range(n):
                w = float(int(want[r, k]))  # rounded to nearest
                assert abs(got[r, k] * 2.0**124 - w) <= np.spacing(abs(w)), (r, k)
    # all other lines repeat these, bit for bit
    assert np.array_equal(got, got[:distinct][which])
    # adding to what is there: 3 y after two more passes
    apply(1)
    assert np.array_equal(apply(1), (y + y) + y)


def test_out_of_memory_is_reported_once(check):
    import torch
    from paper_1107_2461_gb300 import ERR_OUT_OF_MEMORY
    assert check.prepare_status(1 << 20) == ERR_OUT_OF_MEMORY  # 17 TB
    # the next launch does not report it again
    eye = torch.eye(33, dtype=torch.float64, device="cuda")
    x = torch.randn(5, 33, dtype=torch.float64, device="cuda")
    y = torch.empty_like(x)
    torch.cuda.synchronize()
    assert check(eye.data_ptr(), 33, x.data_ptr(), y.data_ptr(), 5, 1, 1, 0) == 0
    # one product per result, one rounding of a 62-bit value
    assert (y - x).abs().max() <= 2.0**-52 * x.abs().max()
