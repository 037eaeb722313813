"""The tensor-core path's choice of a form for a layer, run on the CPU (`tests/form_host.cu`): what each form may be given."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = os.path.join(ROOT, "tests", "form_host.cu")
IN = ["N", "H", "W", "C", "Cp", "K", "R", "S", "stride", "pad", "xb", "wb", "mode", "packed", "s2d", "path"]
OUT = ["status", "s2d_ok", "planned", "rows_geom", "narrow", "use_patch", "pk", "BN", "n_groups", "overlap", "TW", "TH", "TN",
       "tiles"]


def build_harness(src):
    """A host program of this folder, compiled against the library's objects."""
    from paper_2203_12091_gb300 import build as B
    if not os.path.exists(B.nvcc()) and not shutil.which(B.nvcc()):
        pytest.skip("nvcc not available")
    B.build()
    exe = os.path.join(ROOT, "tests", "_build", os.path.basename(src)[:-3])
    objs = sorted(os.path.join(B.BUILD, f) for f in os.listdir(B.BUILD) if f.endswith(".o"))
    deps = [src] + objs + [os.path.join(B.CSRC, f) for f in os.listdir(B.CSRC) if f.endswith(".cuh")]
    if not os.path.exists(exe) or any(os.path.getmtime(d) > os.path.getmtime(exe) for d in deps):
        os.makedirs(os.path.dirname(exe), exist_ok=True)
        r = subprocess.run([B.nvcc(), *B.ARCH, "-O2", "-std=c++17", "--expt-relaxed-constexpr", f"-I{B.INCLUDE}", f"-I{B.CSRC}", src,
                            *objs, "-o", exe + ".tmp"], capture_output=True, text=True)
        assert r.returncode == 0, r.stdout + r.stderr
        os.replace(exe + ".tmp", exe)
    return exe


def choose(layers):
    """The choices for layers given as dicts (mode 1: int64 sums; missing: no padding, 8 / 7 bits, default path)."""
    exe = build_harness(SRC)
    text = ""
    for c in layers:
        c = {"W": c["H"], "S": c["R"], "Cp": (c["C"] + 7) // 8 * 8, "stride": 1, "pad": 0, "xb": 8, "wb": 7, "mode": 1, "packed": 0,
             "s2d": 0, "path": "-", **c}
        text += " ".join(str(c[k]) for k in IN) + "\n"
    r = subprocess.run([exe], input=text, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr
    rows = [dict(zip(OUT, map(int, line.split()))) for line in r.stdout.strip().splitlines()]
    assert len(rows) == len(layers)
    return rows


def test_packed_weights_stay_behind_the_space_to_depth_form():
    """The records hold the original reduction: the original layer may read them, its rewritten form may not."""
    layers = [dict(N=3, H=224, C=3, K=192, R=4, stride=4), dict(N=40, H=5, C=8, K=16384, R=5, stride=4),
              dict(N=40, H=4, C=3, K=16384, R=4, stride=4), dict(N=40, H=7, C=8, K=264, R=7, stride=2, path="tc")]
    for c, plain, s2d in zip(layers, choose([dict(c, packed=1) for c in layers]), choose([dict(c, packed=1, s2d=1) for c in layers])):
        assert s2d["s2d_ok"] and s2d["planned"] and s2d["rows_geom"] and not s2d["pk"], c
        if c["R"] == c["H"] and c["K"] > 300:
            assert plain["pk"], c


def test_overlapping_pixels_are_read_through_tensor_maps():
    """The space-to-depth form of a wide enough tap row has overlapping pixels: never gathered, over all its geometries."""
    layers = [dict(N=N, H=H, W=W, C=C, K=64, R=R, S=S, stride=st, pad=pad, xb=xb, wb=xb - 1, s2d=1, path=path)
              for st in (2, 3, 4) for R in range(st, 12) for S in range(st, 12) for C in (1, 2, 3, 5, 8)
              for N, H, W, pad in ((1, 31, 29, 0), (40, 51, 47, 0), (7, 140, 140, 3))
              for xb in (8, 16) for path in ("-", "tc_patch")]
    seen = 0
    for c, r in zip(layers, choose(layers)):
        if r["s2d_ok"] and r["planned"] and r["overlap"]:
            seen += 1
            assert r["use_patch"] or r["rows_geom"], c
    assert seen > 1000


def test_space_to_depth_maps_have_31_bit_positions():
    """The copy kernels count a rewritten map's pixels in 32 bits: larger maps keep their own codes."""
    layers = [dict(N=1, H=H, C=1, K=8, R=2, stride=2) for H in (92_000, 92_800, 131_072, 400_000)]
    assert [r["s2d_ok"] for r in choose(layers)] == [1, 0, 0, 0]


def test_patches_give_way_where_their_groups_are_too_many():
    """Patches take whole k-blocks per tap and so more exact groups than the gathered reduction: a layer that only the
    latter keeps exact is gathered, not left to the CUDA cores."""
    layers = [dict(N=4, H=30, C=48, K=64, R=10, pad=5, xb=16, wb=16), dict(N=2, H=14, C=664, K=64, R=7, pad=3, wb=8)]
    for c, r in zip(layers, choose(layers)):
        assert r["planned"] and not r["use_patch"] and r["n_groups"] <= 64, c


def _patch_shape(N, P, Q, stride):
    """Every way of cutting a map into equal counts of columns and rows, in the library's order: widest first."""
    best, ideal, span = None, (N * P * Q + 127) // 128, 255 // stride + 1
    for w in sorted({-(-Q // i) for i in range(1, Q + 1)}, reverse=True):
        for h in sorted({-(-P // j) for j in range(1, P + 1)}, reverse=True):
            if w > min(128, span) or h * w > 128 or h > span:
                continue
            tn = min(128 // (h * w), N)
            t = -(-N // tn) * -(-P // h) * -(-Q // w)
            if best is None or t < best[3] or (t == best[3] and tn < best[2]):
                best = (w, h, tn, t)
            if best[3] == ideal and best[2] == 1:
                return best
    return best


def test_patch_shapes_are_the_best_of_all():
    """The search that skips equal and hopeless shapes finds what a full one finds."""
    import random
    rng = random.Random(2)
    sizes = [(1, 1, 1, 1), (7, 1, 300, 1), (5, 300, 1, 1), (128, 7, 7, 1), (64, 56, 55, 1), (1, 1023, 511, 1), (2, 224, 222, 1), (1, 20, 4095, 8)]
    sizes += [(rng.randint(1, 200), rng.randint(1, 120), rng.randint(1, 120), rng.choice([1, 1, 2, 3, 8])) for _ in range(300)]
    layers = [dict(N=N, H=(P - 1) * st + 3, W=(Q - 1) * st + 3, C=64, K=64, R=3, stride=st) for N, P, Q, st in sizes]
    for (N, P, Q, st), r in zip(sizes, choose(layers)):
        if not r["rows_geom"]:
            assert (r["TW"], r["TH"], r["TN"], r["tiles"]) == _patch_shape(N, P, Q, st), (N, P, Q, st)
