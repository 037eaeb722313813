"""The fp32 epilogue of layers of one exact group, run on the CPU against the oracle (`tests/fepi_host.cu`): codes without
and with a Scale layer, and the fp32 image, on random formats, ties, biases finer and coarser than the accumulator and
clip levels.  A Scale layer's value may be decided by the exact arithmetic behind it only next to a rounding boundary."""
import os
import subprocess

import numpy as np

import oracle
from test_epilogue_host import NA, ORDER, ROOT, _cases, _expected
from test_form_host import build_harness


def _rows(cases):
    exe = build_harness(os.path.join(ROOT, "tests", "fepi_host.cu"))
    text = "\n".join(" ".join(str(c[k]) for k in ORDER) for c in cases) + "\n"
    r = subprocess.run([exe], input=text, capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stderr
    rows = [list(map(int, line.split())) for line in r.stdout.strip().splitlines()]
    assert len(rows) == len(cases)
    return rows


def _image(c):
    kw = dict(scale=np.array([c["m"]]), fl_scale=c["sfl"], shift=np.array([c["h"]]), fl_shift=c["hfl"]) if c["has_scale"] else {}
    v, s = oracle.cblock(np.array([c["acc"]], dtype=np.int64), c["xfl"] + c["wfl"], np.array([c["bias"]]) if c["has_bias"] else None,
                         c["bfl"], bool(c["relu"]), **kw)
    return float(oracle.to_f32(v, s)[0]) if abs(int(v[0])) < 1 << 53 else None  # (the oracle's range)


def test_fp32_epilogue_matches_the_oracle():
    cases = _cases(6000, 21)
    rng = np.random.default_rng(22)
    for c in _cases(6000, 23):  # one-plane operands and codes, sums below 2^24: where the forms apply
        c.update(xb=int(rng.integers(2, 9)), wb=int(rng.integers(2, 9)), yb=int(rng.integers(2, 9)), bb=int(rng.choice([8, 16])))
        c["has_scale"] = int(rng.random() < 0.4)
        c["acc"] = int(rng.integers(-(1 << 24) + 1, 1 << 24)) >> int(rng.integers(0, 20))
        bound = 2 ** (c["xb"] - c["xs"]) * 2 ** (c["wb"] - 1) * c["C"]
        c["acc"] = max(-bound, min(bound, c["acc"]))
        c["bias"] = int(rng.integers(-(1 << (c["bb"] - 1)), 1 << (c["bb"] - 1)))
        if rng.random() < 0.5:
            c.update(bfl=c["xfl"] + c["wfl"] + int(rng.integers(-3, 8)), yfl=c["xfl"] + c["wfl"] - int(rng.integers(1, 14)))
        cases.append(c)
    used, near_count, bad_near = {"vf": 0, "vs": 0, "image": 0}, 0, 0
    for c, (st, vf, vs, near, image) in zip(cases, _rows(cases)):
        if st != 0:
            continue
        if vf != NA:
            used["vf"] += 1
            assert vf == _expected(c), c
        if vs != NA:
            used["vs"] += 1
            near_count += near
            if not near:
                assert vs == _expected(c), c
        if image != NA:
            want = _image(c)
            if want is not None:
                used["image"] += 1
                assert float(np.uint32(image).view(np.float32)) == want, c
    assert min(used.values()) > 200, used
    assert near_count < 0.1 * used["vs"], (near_count, used)
