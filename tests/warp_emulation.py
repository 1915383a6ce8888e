"""A kernel of gts.cu on the host, one fiber per lane, under the thread sanitizer (see warp_emulation.h): the results
of a batch and the sanitizer's report."""
import os
import re
import shutil
import subprocess

import numpy as np

from paper_2607_11262_gb300 import build as B
from paper_2607_11262_gb300 import gts
from paper_2607_11262_gb300 import workloads as W

HERE = os.path.dirname(os.path.abspath(__file__))
NONE = 0xFFFFFFFF
CLASS_BITS = {W.LOAD: 2, W.SMEM: 4, W.MMA: 1, W.EW: 8, W.STORE: 2, W.BAR: 16, W.NOP: 0, W.DSMEM: 4 | 32}
STAND_INS = (("createpolicy", "pol = 0;"), ("ld.relaxed", "r = load_pair(p);"), ("st.relaxed", "store_pair(p, 0u);"),
             ("global.add", "atomicAdd(&c->x, 1u);"), ("global.max", "atomicMax(&c->y, r);"))

MAIN = r"""
static std::vector<std::vector<char>> in;
template <class T> static T *arr(int k) { return reinterpret_cast<T *>(in[k].data()); }
static DevGraph g;
static uint32_t h[16];
static bool lanes, ext, noc, pad, split;
static int32_t *st, *fi, *mk, *status, *cta_sm;
static uint64_t *digest;
static int64_t *busy;
static uint2 *scratch;
static uint32_t words, np_;
static void body() {
  const int32_t *prm = arr<int32_t>(9);
  const uint32_t f = GTS_FULL_TRACE | GTS_WANT_DIGEST | GTS_WANT_CTA_SM | GTS_WANT_BUSY;
#define ARGS g, prm, 0u, np_, f, st, fi, mk, status, digest, cta_sm, busy, scratch, 1u, words, nullptr, 0u
  if (lanes && ext) k_simulate_lanes<true>(ARGS, 0.0f, pad);
  else if (lanes) k_simulate_lanes<false>(ARGS, 0.0f, pad);
  else if (noc) k_simulate<true, true, false>(ARGS);
  else if (ext) k_simulate<true, false, false>(ARGS);
  else if (split) k_simulate<false, false, true>(ARGS);
  else k_simulate<false, false, false>(ARGS);
}
int main(int, char **argv) {
  FILE *f = fopen(argv[1], "rb");
  if (fread(h, 4, 16, f) != 16) return 2;
  for (uint64_t len; fread(&len, 8, 1, f) == 1;) {
    in.emplace_back(len + 16);
    if (fread(in.back().data(), 1, len, f) != len) return 2;
  }
  fclose(f);
  g.rec = arr<uint4>(0); g.rng = arr<uint4>(1); g.succ = arr<uint2>(2); g.stream_first = arr<uint32_t>(3);
  g.cta_cnt = arr<uint32_t>(4); g.cta_kernel = arr<uint32_t>(5); g.node_off = arr<uint32_t>(6); g.cta_off = arr<uint32_t>(7);
  g.W = h[0]; g.G = 1; g.row_nodes = h[1]; g.row_ctas = h[2]; g.cross_cta = h[3]; g.n_tiles = h[4]; g.class_mask = h[5];
  g.zero_types = h[6];
  np_ = h[7]; lanes = h[8]; ext = h[9]; noc = h[10]; pad = h[11]; split = h[13];
  words = 64;
  for (uint32_t p = 0; p < np_; p++) {
    const int32_t *row = arr<int32_t>(9) + p * GTS_NPARAM;
    Layout L;
    LaneLayout LL;
    if (check_row(row, 1, g.class_mask) != GTS_OK || !make_layout(row, g.row_ctas, g.W, g.class_mask, L)) continue;
    if (lanes && (!lane_row_ok(row, g.zero_types) || !make_lane_layout(L, pad, row[GTS_P_L2_BYTES] ? g.n_tiles : 0u, LL))) return 3;
    words = std::max(words, lanes ? LL.words : L.words);
  }
  const size_t n = g.row_nodes, row = std::max<size_t>(16, ((n + 1) & ~size_t(1)) * 8 + 16 * g.n_tiles);
  shared_words = (uint32_t *)aligned_alloc(16, words * 4);
  memset(shared_words, 0xA5, words * 4);
  scratch = (uint2 *)aligned_alloc(16, 16 + row);
  memset((void *)scratch, 0xA5, 16 + row);
  st = new int32_t[np_ * n](); fi = new int32_t[np_ * n](); mk = new int32_t[np_](); status = new int32_t[np_]();
  cta_sm = new int32_t[np_ * g.row_ctas](); digest = new uint64_t[np_](); busy = new int64_t[np_ * GTS_BUSY_CLASSES]();
  run_warp(body, h[12]);
  f = fopen(argv[2], "wb");
  fwrite(status, 4, np_, f); fwrite(mk, 4, np_, f); fwrite(st, 4, np_ * n, f); fwrite(fi, 4, np_ * n, f);
  fwrite(cta_sm, 4, np_ * g.row_ctas, f); fwrite(digest, 8, np_, f); fwrite(busy, 8, np_ * GTS_BUSY_CLASSES, f);
  fwrite((char *)scratch + 16, 1, row, f);
  fclose(f);
  return 0;
}
"""


def build(path, edit=lambda s: s):
    """Compiles the device part of gts.cu (after ``edit``) into an executable in ``path``; None without the sanitizer."""
    if shutil.which("g++") is None:
        return None
    s = edit(open(B.SRC).read())
    s = s[:s.index("\nsize_t align_up(size_t x) {")] + "\n}  // namespace\n"
    s = s.replace("#include <cuda_runtime.h>", "")
    a, b = s.index("thread_local char g_err"), s.index("// sums of work kept for the cost")  # error texts, CUDA statuses
    s = s[:a] + s[b:]
    s = s.replace("extern __shared__ __align__(16) uint32_t smem[];", "uint32_t *smem = shared_words;")

    def stand_in(m):
        return next(c for k, c in STAND_INS if k in m.group(0)) + "\n"
    s = re.sub(r"asm volatile\(.*?\);\n", stand_in, s, flags=re.S)
    src, exe = os.path.join(path, "warp.cpp"), os.path.join(path, "warp")
    with open(src, "w") as f:
        f.write('#include "warp_emulation.h"\n' + s + MAIN)
    cmd = ["g++", "-std=c++17", "-O1", "-g", "-w", "-fsanitize=thread", "-I", HERE, "-I", os.path.dirname(B.HDR)]
    probe = subprocess.run(cmd + ["-x", "c++", "-", "-o", exe], input="int main() {}", text=True, capture_output=True)
    if probe.returncode or subprocess.run([exe]).returncode:
        return None
    subprocess.check_call(cmd + ["-o", exe, src])
    return exe


def run(exe, path, g, params, lanes, pad=True, backwards=False, split=False):
    """Results of the batch, as tests.gpu_helpers.run_gpu gives them, with ``scratch``, and the sanitizer's report."""
    n, C, Wp = g.n_nodes, g.n_ctas, g.warps_per_cta
    col, cta = g.col.astype(np.int64), g.cta.astype(np.int64)
    src = np.repeat(np.arange(n), np.diff(g.row_ptr.astype(np.int64)))
    nxt, first = np.full(n, NONE, np.uint32), np.full(C * Wp, NONE, np.uint32)
    for v in range(n - 1, -1, -1):
        key = cta[v] * Wp + int(g.warp[v])
        nxt[v], first[key] = first[key], v
    rec, rng, succ = np.zeros((n, 4), np.uint32), np.zeros((n, 4), np.uint32), np.zeros((g.n_edges, 2), np.uint32)
    rec[:, 0], rec[:, 1], rec[:, 2] = g.work, g.lat_extra, nxt
    rec[:, 3] = g.type.astype(np.uint32) | (np.bincount(col, minlength=n).astype(np.uint32) << 4)
    rng[:, 2], rng[:, 3] = g.row_ptr[:-1], g.row_ptr[1:]
    n_tiles = 0
    if getattr(g, "tile", None) is not None:
        n_tiles = int(g.n_tiles)
        tiled = (g.tile != W.NO_TILE) & ((g.type == W.LOAD) | (g.type == W.STORE))
        rng[:, 0] = np.where(tiled, g.tile.astype(np.int64) + 1, 0)
    succ[:, 0] = col
    succ[:, 1] = g.ekind.astype(np.uint32) | (g.warp[col].astype(np.uint32) << 1) | (g.cta[col].astype(np.uint32) << 8)
    mask = int(np.bitwise_or.reduce([CLASS_BITS[int(t)] for t in np.unique(g.type)]))
    zero = (g.lat_extra == 0) & ((g.work == 0) | (g.type == W.NOP)) & (g.type != W.BAR)
    zero_types = sum(1 << int(t) for t in np.unique(g.type[zero]))
    prm = np.ascontiguousarray(params, np.int32)
    P = prm.shape[0]
    ext = bool(np.any(prm[:, W.P_ISSUE_POLICY]) or np.any(prm[:, W.P_L2_BYTES]))
    head = np.array([Wp, n, C, int(np.any(cta[src] != cta[col])), n_tiles, mask, zero_types, P, lanes, ext,
                     bool(mask & 32), pad, backwards, split, 0, 0], np.uint32)
    cnt = np.bincount(cta, minlength=C).astype(np.uint32)
    arrays = (rec, rng, succ, first, cnt, g.cta_kernel, g.node_off, g.cta_off, np.zeros(0, np.uint32), prm)
    a, b = os.path.join(path, "in"), os.path.join(path, "out")
    with open(a, "wb") as f:
        f.write(head.tobytes())
        for x in arrays:
            x = np.ascontiguousarray(x)
            f.write(np.uint64(x.nbytes).tobytes() + x.tobytes())
    r = subprocess.run([exe, a, b], capture_output=True, text=True, timeout=600,
                       env=dict(os.environ, TSAN_OPTIONS="halt_on_error=0 history_size=4 exitcode=66"))
    assert r.returncode in (0, 66), (r.returncode, r.stderr[-2000:])
    buf, at, res = open(b, "rb").read(), 0, {}
    for k, dt, shape in (("status", np.int32, (P,)), ("makespan", np.int32, (P,)), ("start", np.int32, (P, n)),
                         ("finish", np.int32, (P, n)), ("cta_sm", np.int32, (P, C)), ("digest", np.uint64, (P,)),
                         ("busy", np.int64, (P, gts.GTS_BUSY_CLASSES))):
        k_n = int(np.prod(shape))
        res[k] = np.frombuffer(buf, dt, k_n, at).reshape(shape)
        at += k_n * np.dtype(dt).itemsize
    res["scratch"] = np.frombuffer(buf, np.uint8, -1, at)
    return res, r.stderr
