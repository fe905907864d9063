"""Shapes within a few KB of the shared-memory limit have an expansion plan (host only): the converter kernel's
plans are charged for the rows that its MMAs read behind a last sub-tile, and for no more.  Each of these, and
every shape around it with smaller ranks, fits; the limit itself is still respected."""
import itertools

import pytest

import paper_2401_04189_gb300 as P

LIMIT = 226 * 1024        # dynamic shared memory that a plan may ask for

NEAR = [
    ("tf32", (40, 192, 84), (20, 89, 71), 0),
    ("tf32", (129, 140, 120), (108, 45, 98), 1),
    ("tf32", (174, 222, 200), (174, 124, 38), 0),
    ("bf16", (13, 128, 236), (3, 106, 196), 0),
    ("bf16", (51, 215, 128), (45, 190, 108), 0),
    ("tf32x3", (20, 60, 232), (16, 40, 128), 0),
    ("tf32x3", (31, 52, 228), (2, 35, 126), 0),
    ("bf16x3", (60, 223, 136), (33, 185, 95), 0),
    ("bf16x3", (76, 219, 140), (74, 183, 91), 0),
]


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2401_04189_gb300 import build
    build.build()


@pytest.mark.parametrize("prec,n,r,form", NEAR)
def test_shapes_near_the_limit_have_a_plan(prec, n, r, form):
    for d2, d3 in itertools.product((0, 1, 3, 8), (0, 1, 3, 8)):
        rr = (r[0], r[1] - d2, r[2] - d3)
        d = P.tx_describe_expansion_plan(n, rr, 20, prec, form)
        assert 0 < d["smem_bytes"] <= LIMIT, (rr, d)


def pad(v, m):
    return (v + m - 1) // m * m


def test_plans_hold_every_row_that_is_read():
    """The rings, one converted operand and the rows an MMA reads past them, recomputed from the plan's own
    numbers for whole-slab plans of one plane."""
    seen = 0
    for prec, n2, n3, r2, r3 in itertools.product(("tf32x3", "bf16x3"), (40, 64, 65, 96, 100, 116, 130, 200),
                                                  (60, 64, 120), (5, 16, 33, 64), (3, 8, 17, 40)):
        if r2 > n2:
            continue
        d = P.tx_describe_expansion_plan((2, n2, n3), (1, r2, r3), 4, prec, 0)
        if d["kernel"] != "converter" or d["planes"] != 1 or d["z_parts"]:
            continue
        seen += 1
        mk = 8 if prec == "tf32x3" else 16
        ks2, ks3, ny = -(-r2 // mk), -(-r3 // mk), -(-n2 // 128)
        rows = pad(n2, 16) if ny == 1 else 128 * ny                    # rows kept per K step of A_t2
        ya, zb, b3 = ks2 * rows * 32, ks2 * pad(r3, 8) * 32, ks3 * pad(n3, 16) * 32
        load, load_b = pad(2 * (ya + zb), 1024), pad(2 * b3, 1024)
        last = load * (d["stages2"] - 1)
        a_end = last + 2 * ya + (128 * ny - rows) * 32                 # 128-row MMAs
        z_end = last + 2 * (ya + zb) + (pad(r3, 16) - pad(r3, 8)) * 32      # pad16(r3) columns of Z
        end = load * d["stages2"] + load_b * d["stages3"]
        if not (prec == "tf32x3" and n2 > 64):                         # converted operand in shared memory
            end += 2 * ks3 * rows * 32 + (128 * ny - rows) * 32
        assert d["smem_bytes"] - 1024 >= max(a_end, z_end, end), (prec, n2, n3, r2, r3, d)
    assert seen > 50
