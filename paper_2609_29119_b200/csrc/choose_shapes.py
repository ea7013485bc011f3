#!/usr/bin/env python3
"""Chooses the radices, their order, the threads and the shared-memory layout of every 5-smooth band length (band_smooth.cuh) and
writes band_shapes.cuh, which is under version control.

A shape is M = R0 R1 R2 R3 R4 (trailing ones: fewer stages) on T threads, PER items in a CTA of the group's THREADS.  Radices: the
fewest stages, then the smallest largest radix (fewer registers and less code per stage); among the orders of those the one
with the least work, counted in warp instructions (a warp with one active lane issues as often as a full one) and
shared-memory cycles.

Layout: position p of chunk k0 (first-stage output digit) at k0 CHUNK + p + (PAD ? p / PAD : 0).  MAP_j = 1: the chunk index
runs fastest over the threads of middle stage j (short strides), 0: the position inside the sub-transform does.
"""
import itertools
import multiprocessing
import os
import sys

import gen_codelets as gc

RADICES = (2, 3, 4, 5, 6, 8, 9, 10, 12, 15, 16)
# class: lengths above, up to, threads per CTA, largest radix, threads of an item
GROUPS = {0: (0, 128, 256, 16, lambda m: 8), 1: (128, 1024, 256, 10, lambda m: 32),
          2: (1024, 4096, 256, 12, lambda m: 128 if m <= 2304 else 256), 4: (13500, 27648, 1024, 16, lambda m: 1024)}
SMEM_ELEMS = 227 * 1024 // 8


def smooth_lengths(lo, hi):
    for m in range(lo // 4 * 4 + 4, hi + 1, 4):
        x = m
        for f in (2, 3, 5):
            while x % f == 0:
                x //= f
        if x == 1:
            yield m


def codelet_ops(r, memo={}):
    if r not in memo:
        e = gc.E()
        gc.dft(e, [((e.let("r"), 1), (e.let("i"), 1)) for _ in range(r)])
        memo[r] = len(e.lines) - 2 * r
    return memo[r]


def rows(r):
    return (r - 1).bit_length()


def twiddle_ops(r):
    return 4 * (r - 1) + 4 * (r - 1 - rows(r)) + rows(r)


def ops(r, kind):   # of one butterfly
    fixed = {"first": 14 + 11 * r, "middle": 14 + 2 * r, "last": 16 + 5 * r}[kind]
    return fixed + codelet_ops(r) + (twiddle_ops(r) if kind != "last" else 0)


def factorisations(m, most):
    if most == 0:
        return
    for r in RADICES:
        if m == r:
            yield (r,)
        elif m % r == 0:
            for rest in factorisations(m // r, most - 1):
                yield (r,) + rest


class Shape:
    def __init__(s, radices, T, per, threads):
        s.r, s.T, s.per, s.threads = radices, T, per, threads
        s.M = 1
        for x in radices:
            s.M *= x
        s.stride = []
        n = s.M
        for x in radices:
            n //= x
            s.stride.append(n)
        s.rl, s.nl = radices[-1], s.M // radices[-1]
        s.pad, s.chunk, s.maps = 0, s.stride[0], [0] * (len(radices) - 2)

    def at(s, p):
        return p + (p // s.pad if s.pad else 0)

    def chunk_min(s):
        return s.at(s.stride[0] - 1) + 1

    def buf(s):
        return s.r[0] * s.chunk

    def kinds(s):
        return ["first"] + ["middle"] * (len(s.r) - 2) + ["last"]

    def warp_rounds(s, butterflies):
        """warps with an active lane, summed over rounds, and the number of rounds"""
        rounds = -(-butterflies // s.T)
        total = 0
        for i in range(rounds):
            act = min(s.T, butterflies - i * s.T)
            if s.T % 32 == 0:
                total += s.per * -(-act // 32)
            else:
                total += len({(g * s.T + t) // 32 for g in range(s.per) for t in range(act)})
        return total, rounds

    def middle_address(s, j, w):
        n, st, blocks = s.r[j] * s.stride[j], s.stride[j], s.stride[0] // (s.r[j] * s.stride[j])
        if s.maps[j - 1]:
            k0, x = w % s.r[0], w // s.r[0]
            np_, blk = x % st, x // st
        else:
            np_, x = w % st, w // st
            k0, blk = x // blocks, x % blocks
        return k0 * s.chunk + s.at(blk * n + np_)

    def last_address(s, w):
        k0, x, pos = w % s.r[0], w // s.r[0], 0
        for j in range(1, len(s.r) - 1):
            pos += (x % s.r[j]) * s.stride[j]
            x //= s.r[j]
        return k0 * s.chunk + s.at(pos)

    def conflicts(s, butterflies, address):
        """average shared-memory cycles per 64-bit access of 16 lanes, 1 without conflicts"""
        total = n = 0
        for first in (0, 64, 96):
            for half in (0, 16):
                banks = {}
                for x in range(first + half, first + half + 16):
                    g, t = x // s.T, x % s.T
                    if g >= s.per or t >= butterflies:
                        continue
                    a = g * s.buf() + address(t)
                    banks.setdefault(a % 16, set()).add(a)
                if banks:
                    total += max(len(v) for v in banks.values())
                    n += 1
        return total / max(1, n)

    def layout(s):
        """CHUNK, PAD and the maps with the fewest shared-memory cycles"""
        best = None
        room = SMEM_ELEMS // (s.per * (1 if s.threads == 1024 else 3 if s.per >= 8 else 4))
        for pad in ([0, s.rl] if len(s.r) > 2 else [0]):
            s.pad = pad
            for extra in range(0, 17):
                s.chunk = s.chunk_min() + extra
                if s.buf() > room:
                    continue
                cost = s.r[0] * s.conflicts(s.stride[0], lambda b: s.at(b)) * (s.M / s.r[0])
                for j in range(1, len(s.r) - 1):
                    opts = []
                    for m in (0, 1):
                        s.maps[j - 1] = m
                        opts.append((s.conflicts(s.M // s.r[j], lambda w: s.middle_address(j, w)) * (1.0 if m == 0 else 1.02), m))
                    c, s.maps[j - 1] = min(opts)
                    cost += 2 * c * s.M
                cost += s.conflicts(s.nl, s.last_address) * s.M
                cost = cost / s.M / (2 * (len(s.r) - 1)) + 1e-3 * extra + (5e-3 if pad else 0)
                if best is None or cost < best[0]:
                    best = (cost, s.pad, s.chunk, list(s.maps))
        if best is None:
            return None
        s.cycles, s.pad, s.chunk, s.maps = best
        return s.cycles

    def estimate(s, cycles=1.1):
        """per item and SM: issue slots of the four schedulers and shared-memory cycles, half hidden behind one another"""
        instr = lsu = 0.0
        for x, kind in zip(s.r, s.kinds()):
            w, _ = s.warp_rounds(s.M // x)
            instr += w * ops(x, kind)
            lsu += w * {"first": 1, "middle": 2, "last": 1}[kind] * x * 2 * cycles
        return (instr / 4 + 0.5 * lsu) / s.per


def choose(m, group):
    _, _, threads, cap, t_of = GROUPS[group]
    T = t_of(m)
    sets = {tuple(sorted(f)) for f in factorisations(m, 5) if len(f) >= 2 and max(f) <= cap}
    fewest = min(len(f) for f in sets)
    smallest = min(max(f) for f in sets if len(f) == fewest)
    best = None
    for f in {o for s in sets if len(s) == fewest and max(s) == smallest for o in itertools.permutations(s)}:
        s = Shape(f, T, threads // T, threads)
        c = s.layout()
        if c is None:
            continue
        e = s.estimate(c)
        if best is None or (e, f) < best[:2]:
            best = (e, f, s)
    return best[0], best[2]


def row(job):
    m, group = job
    e, s = choose(m, group)
    r = list(s.r) + [1] * (5 - len(s.r))
    maps = s.maps + [0] * (3 - len(s.maps))
    print(group, m, s.r, "T", s.T, "per", s.per, "pad", s.pad, "chunk", s.chunk, s.maps, "cyc %.2f est %.0f per elem %.3f" % (s.cycles, e, e / m), flush=True)
    return f"    X({m}, {', '.join(map(str, r))}, {s.T}, {s.per}, {s.threads}, {s.pad}, {s.chunk}, {', '.join(map(str, maps))})"


def main(path):
    out = ["// Written by choose_shapes.py: the shapes of the 5-smooth band lengths (band_smooth.cuh), longest first.",
           "// X(M, R0, R1, R2, R3, R4, T, PER, THREADS, PAD, CHUNK, MAP1, MAP2, MAP3)", "#pragma once", ""]
    with multiprocessing.Pool() as pool:
        for group, (lo, hi, _, _, _) in sorted(GROUPS.items()):
            lines = pool.map(row, [(m, group) for m in sorted(smooth_lengths(lo, hi), reverse=True)], chunksize=1)
            out.append(f"#define CQT_SHAPES_{group}(X) \\")
            out.append(" \\\n".join(lines))
            out.append("")
    open(path, "w").write("\n".join(out))


if __name__ == "__main__":
    here = os.path.dirname(os.path.abspath(__file__))
    main(sys.argv[1] if len(sys.argv) > 1 else os.path.join(here, "band_shapes.cuh"))
