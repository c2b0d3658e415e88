"""The streaming kernel (csrc/stream.cu) run on the CPU under schedules in which one warp of a CTA gets
as far ahead of the others as the kernel's barriers allow (tests/emulator.h): whatever order the warps
take, every output appears once with the sum of its products, and the positions between them are
filled."""
import ctypes

import numpy as np
import pytest

import emulator

HARNESS = r"""
extern "C" int run_stream(uint32_t order, int sms, uint64_t FY, uint32_t groups, const uint32_t* goff, uint32_t* ystart,
                          uint32_t* w, uint32_t* ck, double* xv, const uint32_t* yoff, const uint32_t* yfk,
                          const double* yv, uint32_t ny, uint64_t cap, uint64_t win, int32_t* coords, double* vals, uint64_t* nnz,
                          uint64_t* holes) {
  using namespace stc;
  const uint32_t seg = FY > kDenseSeg ? kDenseSeg : [&] { uint32_t c = 64; while (c < FY) c <<= 1; return c; }();
  const uint32_t nseg = (uint32_t)((FY + seg - 1) / seg);
  std::vector<uint32_t> list(groups);
  for (uint32_t g = 0; g < groups; g++) list[g] = g;
  std::vector<StreamHole> hl(stream_max_holes(groups, nseg));
  unsigned nholes = 0;
  u64 nz = 0, total = 0, fill[2] = {0, 0};
  uint32_t status = 0;
  GroupArgs a{};
  a.goff = goff;
  a.gx = GroupedX{ystart, w, xv, ck};
  a.yfk = yfk;
  a.yv = yv;
  a.FY = FY;
  a.op.order = 2;  // the key itself, in two words
  a.op.pow2 = a.op.ident = 1;
  a.op.mod[0] = a.op.mod[1] = 1ull << 32;
  a.op.shift[1] = 32;
  a.coords = coords;
  a.vals = vals;
  a.out_cap = cap;
  a.nz = &nz;
  a.status = &status;
  StreamArgs sa{};
  sa.holes = hl.data();
  sa.nholes = &nholes;
  sa.hole_total = &total;
  sa.ny_entries = ny;
  emu::order = order;
  emu::stuck = false;
  if (launch_group_stream(a, yoff, nseg, seg, list.data(), groups, sa, sms, nullptr)) return 1;
  if (nholes > hl.size() || nz > cap) return 2;
  for (const StreamHole& h : hl)
    if (h.len >= 65536) return 3;
  std::vector<uint32_t> dst(win);
  HoleRound rd{0, win, 0, dst.data()};
  do {
    rd.base = fill[1];
    if (launch_hole_fill(hl.data(), &nholes, &nz, &total, rd, fill, coords, vals, 2, &status, sms, nullptr)) return 3;
    rd.at += win;
  } while (rd.at < total);
  if (fill[0] != fill[1]) return 6;
  *nnz = nz - total;
  *holes = total;
  return emu::stuck ? 4 : status ? 5 : 0;
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return emulator.build(tmp_path_factory.mktemp("stream"), "stream.cu", HARNESS)


def ptr(a):
    return a.ctypes.data_as(ctypes.c_void_p)


def run(lib, order, X, Y, FX, K, FY, sms=1, window=100_000):
    """X, Y: (free key, contract key, value) arrays; checks the outputs against plain sums."""
    xf, xk, xv = X
    yf, yk, yv = Y
    nseg = max(1, -(-FY // 65536))
    at = np.lexsort((yf // 65536, yk))
    yf, yk, yv = yf[at], yk[at], yv[at]
    yoff = np.searchsorted(yk * nseg + yf // 65536, np.arange(K * nseg + 1)).astype(np.uint32)
    at = np.argsort(xf, kind="stable")
    xf, xk, xv = xf[at], xk[at], xv[at]
    goff = np.searchsorted(xf, np.arange(FX + 1)).astype(np.uint32)
    ystart = yoff[xk * nseg]
    w = yoff[(xk + 1) * nseg] - ystart
    dead = 0xFFFFFFFF if FY > 65536 else FY
    want = {}
    for f, k, v in zip(xf.tolist(), xk.tolist(), xv.tolist()):
        for j in range(yoff[k * nseg], yoff[(k + 1) * nseg]):
            z = f * FY + int(yf[j])
            want[z] = want.get(z, 0.0) + v * yv[j]
    products = int(w.astype(np.int64).sum())
    coords = np.full((products, 2), -7, np.int32)
    vals = np.full(products, np.nan)
    nnz, holes = ctypes.c_uint64(), ctypes.c_uint64()
    a = [ystart.astype(np.uint32), w.astype(np.uint32), xk.astype(np.uint32), np.ascontiguousarray(xv), yoff,
         np.append(yf, dead).astype(np.uint32), np.append(yv, 0.0)]
    rc = lib.run_stream(ctypes.c_uint32(order), sms, ctypes.c_uint64(FY), ctypes.c_uint32(FX), ptr(goff), *map(ptr, a),
                        ctypes.c_uint32(len(yf)), ctypes.c_uint64(products), ctypes.c_uint64(window), ptr(coords), ptr(vals), ctypes.byref(nnz),
                        ctypes.byref(holes))
    assert rc == 0
    n = nnz.value
    got = np.ascontiguousarray(coords[:n]).view(np.uint64)[:, 0]
    order_by = np.argsort(got)
    np.testing.assert_array_equal(got[order_by], np.array(sorted(want), np.uint64))
    # Values are small integers here: every sum is exact.
    np.testing.assert_array_equal(vals[:n][order_by], np.array([want[z] for z in sorted(want)]))
    return holes.value


def tensors(rng, groups, entries, runs, length, fy, distinct):
    xf, xk = np.repeat(np.arange(groups), entries), rng.integers(0, runs, groups * entries)
    if distinct:
        yf = np.concatenate([rng.permutation(fy)[:length] for _ in range(runs)])
    else:
        yf = rng.integers(0, fy, runs * length)
    yk = np.repeat(np.arange(runs), length)
    return ((xf, xk, rng.integers(1, 9, len(xf)).astype(float)), (yf, yk, rng.integers(1, 9, len(yf)).astype(float)))


SCHEDULES = [0, 1, 7, 1234]


@pytest.mark.parametrize("order", SCHEDULES)
@pytest.mark.parametrize("entries,length,fy,distinct", [(1, 40, 1000, True),       # no repeats at all
                                                        (2, 60, 1000, False),      # some groups with, some without
                                                        (3, 400, 500, False),      # every key several times
                                                        (2, 900, 3000, True),      # around the list of 512
                                                        (2, 300, 65536, False),    # the widest single segment
                                                        (2, 200, 200_000, False)])  # several segments
def test_any_order_of_the_warps(lib, order, entries, length, fy, distinct):
    rng = np.random.default_rng(entries * 1000 + length + fy)
    X, Y = tensors(rng, 26, entries, 5, length, fy, distinct)
    run(lib, order, X, Y, 26, 5, fy)


@pytest.mark.parametrize("order", SCHEDULES[:2])
def test_groups_of_several_pieces(lib, order):
    """More than 256 X entries in a group."""
    rng = np.random.default_rng(3)
    X, Y = tensors(rng, 6, 300, 40, 4, 5000, False)
    run(lib, order, X, Y, 6, 40, 5000)


@pytest.mark.parametrize("window", [1, 31, 500, 4096])
@pytest.mark.parametrize("order", SCHEDULES[:2])
def test_holes_in_rounds(lib, order, window):
    """The holes filled a window of the output's end at a time, down to a position per round: groups
    whose products are mostly repeats, which drop positions again and again."""
    rng = np.random.default_rng(window)
    X, Y = tensors(rng, 20, 4, 3, 30, 60, False)
    holes = run(lib, order, X, Y, 20, 3, 60, window=window)
    assert holes > 500
