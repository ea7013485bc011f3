"""The table of shapes of the 5-smooth band lengths (csrc/band_shapes.cuh): index maps, shared-memory bounds and barriers of every
shape, with the stages of band_smooth.cuh restated in numpy."""
import os
import re

import numpy as np

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_29119_b200", "csrc")
LIMITS = {0: (0, 128), 1: (128, 1024), 2: (1024, 4096), 4: (13500, 27648)}
THREADS = {0: 256, 1: 256, 2: 256, 4: 1024}
SMEM_ELEMS = 227 * 1024 // 8       # of an SM


def shapes():
    group, out = None, []
    for line in open(os.path.join(CSRC, "band_shapes.cuh")):
        head, row = re.match(r"#define CQT_SHAPES_(\d)\(X\)", line), re.match(r"\s+X\(([^)]*)\)", line)
        if head:
            group = int(head.group(1))
        elif row:
            out.append((group,) + tuple(int(v) for v in row.group(1).split(",")))
    return out


def smooth(m):
    for f in (2, 3, 5):
        while m % f == 0:
            m //= f
    return m == 1


def test_every_length_has_a_shape():
    rows = shapes()
    assert sorted(r[1] for r in rows) == [m for above, upto in LIMITS.values() for m in range(above // 4 * 4 + 4, upto + 1, 4) if smooth(m)]
    for group, (above, upto) in LIMITS.items():
        own = [r[1] for r in rows if r[0] == group]
        assert own == sorted(own, reverse=True) and len(own) <= 40
        assert all(above < m <= upto for m in own)


def test_barriers_are_met_by_all_their_threads():
    """T threads per item and PER items fill the CTA: the barrier of an item counts T threads, so it has to be one of whole warps, or of
    the whole CTA, or of the lanes of one warp."""
    for group, M, *rest in shapes():
        T, per, threads = rest[5], rest[6], rest[7]
        assert threads == THREADS[group] and per * T == threads
        assert 32 % T == 0 if T <= 32 else T % 32 == 0 and per < 16, M     # named barriers 1 ... per


def test_stages_stay_in_the_buffer_and_give_the_dft():
    rng = np.random.default_rng(3)
    for group, M, R0, R1, R2, R3, R4, T, per, threads, pad, chunk, *maps in shapes():
        radices = [r for r in (R0, R1, R2, R3, R4) if r > 1]
        assert np.prod(radices) == M
        at = (lambda p: p + p // pad) if pad else (lambda p: p)
        stride, n = [], M
        for r in radices:
            n //= r
            stride.append(n)
        buf_len = R0 * chunk
        assert per * buf_len <= SMEM_ELEMS // (1 if threads == 1024 else 3)
        x = rng.standard_normal(M) + 1j * rng.standard_normal(M)
        buf = np.full(buf_len, np.nan, dtype=complex)
        dft = {r: np.exp(-2j * np.pi * np.outer(np.arange(r), np.arange(r)) / r) for r in radices}
        b = np.arange(stride[0])
        y = dft[R0] @ x[b[None, :] + np.arange(R0)[:, None] * stride[0]]
        y *= np.exp(-2j * np.pi * np.arange(R0)[:, None] * b[None, :] / M)
        where = at(b)[None, :] + np.arange(R0)[:, None] * chunk
        assert where.max() < buf_len and len(np.unique(where)) == M
        buf[where] = y
        for j in range(1, len(radices) - 1):
            R, s = radices[j], stride[j]
            w, blocks = np.arange(M // R), stride[0] // (R * s)
            if maps[j - 1]:
                k0, z = w % R0, w // R0
                np_, blk = z % s, z // s
            else:
                np_, z = w % s, w // s
                k0, blk = z // blocks, z % blocks
            where = (k0 * chunk + at(blk * (R * s) + np_))[None, :] + np.arange(R)[:, None] * at(s)
            assert where.min() >= 0 and where.max() < buf_len and len(np.unique(where)) == M
            buf[where] = (dft[R] @ buf[where]) * np.exp(-2j * np.pi * np.arange(R)[:, None] * np_[None, :] / (R * s))
        RL, NL = radices[-1], M // radices[-1]
        w = np.arange(NL)
        z, pos = w // R0, 0
        for j in range(1, len(radices) - 1):
            pos = pos + (z % radices[j]) * stride[j]
            z = z // radices[j]
        where = ((w % R0) * chunk + at(pos + 0 * w))[None, :] + np.arange(RL)[:, None]
        assert where.max() < buf_len and len(np.unique(where)) == M
        out = np.empty(M, dtype=complex)
        out[w[None, :] + np.arange(RL)[:, None] * NL] = dft[RL] @ buf[where]
        want = np.fft.fft(x)
        assert np.linalg.norm(out - want) <= 1e-11 * np.linalg.norm(want), M


def test_debug_build_checks_every_access():
    """-DCQT_DEBUG_BOUNDS: loads and stores of the spectrum, the window table, the coefficients, the planes and the buffer are behind
    a check of their index; slot_value has its own."""
    code = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, "band_smooth.cuh")).read())
    body = code[code.index("void smooth_middle("):]
    access = re.compile(r"ld_spectrum<|ld_coefficient<|__ldg\(tab|__stcs\(|\bYs\[|\bd\[")
    lines = body.split("\n")
    found = [i for i, line in enumerate(lines) if access.search(line)]
    assert len(found) == 10
    for i in found:
        assert "CQT_CHK(" in lines[i] or ("in ? ld_spectrum" in lines[i] and "CQT_CHK(" in lines[i - 1]), lines[i]
    assert re.search(r"slot_value<CHAINED>\([^;]*a\.b\.dbg\)", body)
    common = open(os.path.join(CSRC, "band_common.cuh")).read()
    slot = re.search(r"float2 slot_value\(.*?\n}", common, re.S).group(0)
    assert slot.index("CQT_CHK(dbg, 405") < slot.index("__ldg(") and slot.index("CQT_CHK(dbg, 406") < slot.index("ld_spectrum")
