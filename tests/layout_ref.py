"""A restatement of the packer's plan (which slab width a matrix gets) and of a
layout's size, so that a test can say which kernel path its shape reaches:
check() compares the size with what the library allocated, which depends on the
slab width, so a changed plan cannot silently empty a test."""

from __future__ import annotations

import numpy as np
import torch

import paper_2607_02893_gb300 as vbq

RB, MAX_BLOB, UNIT_MAX_GROUPS = 128, 41 * 1024, 200_000


def sm_count() -> int:
    return torch.cuda.get_device_properties(0).multi_processor_count


def _tasks(ends, w):
    """Warp tasks of one width of a unit, from its column ends."""
    span, most = (64, 1) if w == 0 else (32, 3)
    n, start, count = int(ends[-1]), 0, 0
    while start < n:
        first = start & ~1 if w == 0 else start
        end = min(first + span, n)
        inside = ends[(ends > start) & (ends < end)]
        for e, mult in zip(*np.unique(inside, return_counts=True)):
            if mult > most:
                end = int(e)
                break
        count += 1
        start = end
    return count


def unit_sizes(widths, c):
    """Blob sizes (16-byte units) of every unit of slabs of c columns."""
    n, g = widths.shape
    sizes = []
    for s0 in range(0, g, c):
        for r0 in range(0, n, RB):
            part = widths[r0:r0 + RB, s0:s0 + c]
            size = 3 + -(-8 * c // 16)
            for w in range(4):
                ends = np.cumsum((part == (1 << w)).sum(axis=0))
                k = int(ends[-1])
                size += -(-k * (8 << w) // 16) + -(-2 * k // 16) + -(-k // 16) + _tasks(ends, w)
            sizes.append(size)
    return sizes


def unit_plan_fits(c, s, units, groups, sms):
    return c <= 8 and s <= 16 and groups < UNIT_MAX_GROUPS and 4 * units <= (7 if s <= 8 else 5) * sms


def unit_neighbours(g):
    return 64 * g * g < UNIT_MAX_GROUPS


def plan(widths, sms):
    """(columns per slab, slabs, units, allocated bytes)"""
    n, g = widths.shape
    nrb = -(-n // RB)
    cands = []
    for most in (8, 16):
        for c in (2, 4, 8):
            s = -(-g // c)
            if c <= g and not cands and s <= most and unit_plan_fits(c, s, nrb * s, n * g, sms):
                cands.append(c)
    widest = True
    for c in (16, 8, 4, 2, 1):
        if c != 1 and (c > g or 2 * nrb * -(-g // c) < sms):
            continue
        if widest and cands and c < cands[0] and not unit_neighbours(g):
            cands = []
        widest = False
        if not cands or cands[0] != c:
            cands.append(c)
    for c in cands:
        sizes = unit_sizes(widths, c)
        if 16 * max(sizes) <= MAX_BLOB:
            break
    up = lambda v: -(-v // 256) * 256
    blobs = up(16 * sum(sizes) + 256)
    return c, -(-g // c), len(sizes), up(blobs + 4 * (len(sizes) + 1)) + 4 * (2 + 2 * nrb)


def check(layout, widths):
    """The layout's (columns per slab, slabs, units), after comparing its size with the plan's."""
    c, s, units, size = plan(widths, sm_count())
    assert sum(vbq.vbq_packed_bytes(layout)) == size, "the packer planned this matrix differently"
    return c, s, units


def runs_unit_per_block(widths, c, s, units):
    n, g = widths.shape
    return unit_neighbours(g) and unit_plan_fits(c, s, units, n * g, sm_count())


def pair_view(widths, c):
    """(columns per slab, slabs, units) as the two-row table kernel takes a layout of c columns
    per slab: several slabs as one while there are at least half as many units as SMs and the
    slabs' blobs fit one stage."""
    n, g = widths.shape
    nrb, wide = -(-n // RB), 16
    while wide > 1 and (wide > g or 2 * nrb * -(-g // wide) < sm_count()):
        wide //= 2
    sub, blob = wide // c, 16 * max(unit_sizes(widths, c))
    while sub > 1 and sub * blob > MAX_BLOB:
        sub //= 2
    wide = c * max(sub, 1)
    return wide, -(-g // wide), nrb * -(-g // wide)
