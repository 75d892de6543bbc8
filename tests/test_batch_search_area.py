"""Batches and servers with a restricted search (Eq. 6) in the tensor-core form.

The BF16 planes of an image hold the rows that its search rectangle reads,
narrow rectangles in several folds.  On the CPU: for rectangles anywhere in an
image, the places that plane_places names for a pixel are exactly those that
the planes were filled from it, each inside the allocation.  On the GPU:
objects in the lower part of an image, three folds and more, teams of one, two
and many CTAs, as a batch and as a server; iterations, evaluations and pixels
against the oracle, tolerance 0.  The same CPU program says that the engine's
estimate takes the tensor-core form on one CTA for the images of r >= 4.
"""
import ctypes
import os
import subprocess

import numpy as np
import pytest

import oracle
from paper_1403_4238_gb300 import _lib, synth

# W, H, r, the object (x, y, w, h), search factor
CASES = [
    (512, 384, 4, (200, 200, 80, 60), 0.25),
    (480, 639, 4, (180, 380, 60, 120), 0.25),
    (420, 500, 1, (150, 330, 40, 90), 0.5),
    (400, 460, 8, (170, 250, 60, 110), 0.5),
    (640, 600, 6, (330, 420, 90, 100), 0.25),
    (500, 700, 2, (60, 600, 50, 60), 0.5),
]

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include <vector>
#include "inpaint_engine.h"
using namespace inp;

// the image pixel that a place of the planes is filled from (k_planes), -1 outside the image
static long long pixel_of(const ImgState& s, int tx, int row, int xl) {
  const int f = s.tc_f > 1 ? xl / 8 / s.tc_n1 : 0;
  if (f >= (s.tc_f > 1 ? s.tc_f : 1)) return -1;
  const int x = s.tc_xs0 + 8 * (tx * s.tc_n - f * s.tc_n1) + xl, y = s.cy0 - s.r + row + f * s.tc_h;
  return x < s.W && y < s.H ? (long long)y * s.W + x : -1;
}

int main() {
  int W, H, r, x0, x1, y0, y1, want;
  while (scanf("%d %d %d %d %d %d %d %d", &W, &H, &r, &x0, &x1, &y0, &y1, &want) == 8) {
    ImgState s{};
    s.W = W;
    s.H = H;
    s.r = r;
    s.cx0 = x0;
    s.cx1 = x1;
    s.cy0 = y0;
    s.cy1 = y1;
    const size_t bytes = tc_plane_layout(s, want);
    std::vector<uint8_t> mem(bytes);
    tc_bind_planes(s, mem.data());
    const size_t words = (size_t)s.tc_ntx * s.prows * 5 * s.tc_len;
    long long bad = (uint8_t*)(s.planes + words) > mem.data() + bytes;
    bad += s.prows < kTcRows * s.tc_nty + 2 * r;  // the last tile's last source row
    std::vector<int> named(words / 5, 0);
    for (int y = 0; y < H; ++y)
      for (int x = 0; x < W; ++x) {
        uint16_t* p[2];
        plane_places(s, x, y, p[0], p[1]);
        for (uint16_t* q : p) {
          if (!q) continue;
          const size_t o = q - s.planes, row = o / (5 * s.tc_len), xl = o % (5 * s.tc_len);
          if (o >= words || xl >= (size_t)s.tc_len ||
              pixel_of(s, (int)(row / s.prows), (int)(row % s.prows), (int)xl) != (long long)y * W + x)
            ++bad;
          else
            ++named[row * s.tc_len + xl];
        }
      }
    for (int tx = 0; tx < s.tc_ntx; ++tx)
      for (int row = 0; row < s.prows; ++row)
        for (int xl = 0; xl < s.tc_len; ++xl)
          bad += named[((size_t)tx * s.prows + row) * s.tc_len + xl] != (pixel_of(s, tx, row, xl) >= 0 ? 1 : 0);
    printf("%lld %d %d\n", bad, s.tc_f, (int)(tc_round_cycles(s, 1) < plain_round_cycles(s, 1)));
  }
  return 0;
}
"""


@pytest.fixture(scope="module")
def layout(tmp_path_factory):
    d = tmp_path_factory.mktemp("layout")
    src, exe = os.path.join(d, "layout.cu"), os.path.join(d, "layout")
    with open(src, "w") as f:
        f.write(PROGRAM)
    subprocess.run([_lib._nvcc(), _lib.ARCH, "-std=c++17", "-O1", "-I", _lib.INCLUDE, "-I", _lib.CSRC, src, "-o", exe],
                   check=True, capture_output=True)

    def ask(rows):
        text = "\n".join(" ".join(str(v) for v in row) for row in rows) + "\n"
        out = subprocess.run([exe], input=text, check=True, capture_output=True, text=True).stdout.split()
        assert len(out) == 3 * len(rows)
        return [tuple(int(v) for v in out[3 * i: 3 * i + 3]) for i in range(len(rows))]

    return ask


def case_image(W, H, r, box, seed):
    x, y, w, h = box
    m = np.zeros((H, W), np.uint8)
    m[y: y + h, x: x + w] = 1
    return synth.image(W, H, 7, 30.0, seed), m, r


def rect_of(W, H, r, box, alpha):
    x, y, w, h = box
    ex, ey = int(alpha * w), int(alpha * h)
    return (max(r, x - ex), min(W - 1 - r, x + w - 1 + ex), max(r, y - ey), min(H - 1 - r, y + h - 1 + ey))


@pytest.mark.parametrize("r", range(1, 9))
def test_every_place_of_a_pixel_is_named(layout, r):
    rng = np.random.default_rng(r)
    rows = []
    for k in range(60):
        W, H = int(rng.integers(2 * r + 1, 700)), int(rng.integers(2 * r + 1, 500))
        x0, x1 = sorted(int(v) for v in rng.integers(r, W - r, 2))
        y0, y1 = sorted(int(v) for v in rng.integers(r, H - r, 2))
        if k % 3 == 0:  # narrow and low: many folds
            x1, y1 = min(x1, x0 + int(rng.integers(1, 120))), H - 1 - r
        rows.append((W, H, r, x0, x1, y0, y1, 151 if k % 4 == 3 else 0))
    rows.append((1500, 70, r, r, 1499 - r, r, 69 - r, 0))  # several tile columns
    rows.append((1500, 70, r, r + 3, 1499 - r, 30, 69 - r, 151))
    out = layout(rows)
    assert all(o[0] == 0 for o in out), [(row, o) for row, o in zip(rows, out) if o[0]]
    assert max(o[1] for o in out) >= 4


def test_the_cases_fold_and_take_the_tensor_cores(layout):
    rows = []
    for W, H, r, box, alpha in CASES:
        x0, x1, y0, y1 = rect_of(W, H, r, box, alpha)
        m = case_image(W, H, r, box, 1)[1]
        assert oracle.search_rect(m, r, alpha) == (x0, x1, y0, y1)
        rows.append((W, H, r, x0, x1, y0, y1, 0))
    for row, (bad, folds, one) in zip(rows, layout(rows)):
        assert bad == 0 and folds >= 3 and (one or row[2] < 4), (row, folds, one)


@pytest.fixture(scope="module")
def lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return _lib.load()


@pytest.fixture(scope="module")
def cases():
    out = []
    for k, (W, H, r, box, alpha) in enumerate(CASES):
        c = case_image(W, H, r, box, 500 + k)
        ref = oracle.run(*c, alpha=alpha)
        assert ref.status == 0
        out.append((c, alpha, ref))
    return out


def option(lib, alpha):
    opt = _lib.Options()
    lib.inpaint_options_default(ctypes.byref(opt))
    opt.search_alpha = alpha
    return opt


def image_of(c):
    rgb, m, r = c
    H, W = m.shape
    return _lib.Image(rgb.ctypes.data, W, H, 3 * W, m.ctypes.data, W, r)


@pytest.mark.gpu
@pytest.mark.parametrize("alpha", [0.25, 0.5])
@pytest.mark.parametrize("copies", [1, 30, 55])  # teams of about 50, one or two, and one CTA
def test_batch_with_a_search_factor(lib, cases, alpha, copies):
    mine = [x for x in cases if x[1] == alpha] * copies
    opt, b = option(lib, alpha), ctypes.c_void_p()
    ims = (_lib.Image * len(mine))(*[image_of(x[0]) for x in mine])
    assert lib.inpaint_batch_create(ims, len(mine), ctypes.byref(opt), ctypes.byref(b)) == 0
    try:
        for again in range(2):
            assert lib.inpaint_batch_run_ctx(b, 0, None) == 0
            for i, (c, _, ref) in enumerate(mine):
                out = np.zeros_like(c[0])
                it, ev = ctypes.c_int(), ctypes.c_uint64()
                assert lib.inpaint_batch_result(b, i, out.ctypes.data, 3 * out.shape[1], ctypes.byref(it),
                                                ctypes.byref(ev)) == 0
                assert it.value == ref.iters and ev.value == ref.evals, i
                assert np.array_equal(out, ref.rgb), i
            assert lib.inpaint_batch_reset(b) == 0
    finally:
        lib.inpaint_batch_destroy(b)


@pytest.mark.gpu
@pytest.mark.parametrize("alpha", [0.25, 0.5])
def test_server_with_a_search_factor(lib, cases, alpha):
    mine = [x for x in cases if x[1] == alpha] * 20
    opt, s = option(lib, alpha), ctypes.c_void_p()
    assert lib.inpaint_server_create(8 << 30, 256, 0, ctypes.byref(opt), ctypes.byref(s)) == 0
    try:
        ids = []
        for c, _, _ in mine:
            rid = ctypes.c_uint64()
            im = image_of(c)
            assert lib.inpaint_server_submit(s, ctypes.byref(im), ctypes.byref(rid)) == 0
            ids.append(rid)
        assert lib.inpaint_server_wait_idle(s, 120.0) == 0
        for rid, (c, _, ref) in zip(ids, mine):
            out, info = np.zeros_like(c[0]), _lib.RequestInfo()
            assert lib.inpaint_server_poll(s, rid, out.ctypes.data, 3 * out.shape[1], ctypes.byref(info)) == 0
            assert info.status == 0 and info.iterations == ref.iters and info.evals == ref.evals
            assert np.array_equal(out, ref.rgb)
    finally:
        lib.inpaint_server_destroy(s)
