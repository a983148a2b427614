"""The barrier protocol of the weight-gradient kernel (k_wgrad), modelled on the host.

Its roles -- the producer copying X and dZ rows into two rings (one TMA copy a row, landing in any
order), the issuer multiplying each X row with the three dZ rows it meets, the four bias warps
adding up each dZ row, the tensor pipe completing products and commits in order after they were
issued -- meet only at mbarriers, and a parity wait is right only when its barrier is at the awaited
phase or the one after it.  The model walks the kernel's chunks and rows, with the ring sizes and
barrier counts read from the source, under random interleavings, and checks that:
  - no role waits forever, and every parity wait finds its barrier at the awaited phase or the next;
  - every product reads the X row and the three dZ rows it means to, landed, from its issue until it
    completes, and every bias warp the dZ row it means to;
  - over an image each X row meets its dZ rows once and each dZ row is added to the bias once;
  - every copy has landed and every product completed when the block ends.
A block's slots and phases run on from one chunk to the next: blocks of one to five chunks."""
import inspect
import pathlib
import random
import re

import pytest

from test_conv_protocol import Barrier, conv_chunk

SRC = pathlib.Path(__file__).resolve().parents[1] / "paper_2312_06827_gb300" / "csrc" / "svgf_kpn.cu"


def rings():
    m = re.search(r"kWgXRing\s*=\s*(\d+)\s*,\s*kWgDRing\s*=\s*(\d+)\s*;", SRC.read_text())
    return int(m.group(1)), int(m.group(2))


X_RING, D_RING = rings()
BIAS_WARPS = 4


def simulate(heights, seed):
    """One block over chunks of the given heights."""
    rnd = random.Random(seed)
    full_x, free_x = [Barrier() for _ in range(X_RING)], [Barrier() for _ in range(X_RING)]
    full_d, free_d = [Barrier() for _ in range(D_RING)], [Barrier(1 + BIAS_WARPS) for _ in range(D_RING)]
    slot_x, slot_d = {}, {}
    copies, pipe, met = [], [], []                # copies in flight, the tensor pipe's queue, products done
    biased = [[] for _ in range(BIAS_WARPS)]

    def producer():
        nx = nd = 0
        used_x, used_d = set(), set()
        phase_x, phase_d = [0] * X_RING, [0] * D_RING
        for c, rows in enumerate(heights):
            order = [("d", -1), ("d", 0)]
            for i in range(rows):
                order += [("x", i), ("d", i + 1)]
            for kind, row in order:
                if kind == "x":
                    sl, nx = nx % X_RING, nx + 1
                    if sl in used_x:
                        while not free_x[sl].done(phase_x[sl]):
                            yield
                        phase_x[sl] += 1
                    used_x.add(sl)
                    slot_x[sl] = ("in flight", c, row)
                else:
                    sl, nd = nd % D_RING, nd + 1
                    if sl in used_d:
                        while not free_d[sl].done(phase_d[sl]):
                            yield
                        phase_d[sl] += 1
                    used_d.add(sl)
                    slot_d[sl] = ("in flight", c, row)
                copies.append((kind, sl))
                yield
        while copies:                             # its copies land before the block ends
            yield

    def copy_engine():
        while True:
            if copies:
                kind, sl = copies.pop(rnd.randrange(len(copies)))
                slots, full = (slot_x, full_x) if kind == "x" else (slot_d, full_d)
                slots[sl] = ("landed",) + slots[sl][1:]
                full[sl].arrive()
            yield

    def tensor_pipe():
        """Products and commits complete in the order they were issued."""
        while True:
            if pipe:
                op = pipe.pop(0)
                if op[0] == "commit":
                    op[1].arrive()
                else:
                    _, c, i, sx, sd = op
                    assert slot_x[sx] == ("landed", c, i), ("X restaged under a product", op, slot_x[sx])
                    for j in range(3):
                        assert slot_d[sd[j]] == ("landed", c, i - 1 + j), ("dZ under a product", op, slot_d[sd[j]])
                    met.append((c, i))
            yield

    def issuer():
        nx = nd = 0
        phase_x, phase_d = [0] * X_RING, [0] * D_RING
        for c, rows in enumerate(heights):
            for i in range(rows):
                for j in range(0 if i == 0 else 2, 3):
                    sl = (nd + i + j) % D_RING
                    while not full_d[sl].done(phase_d[sl]):
                        yield
                    phase_d[sl] += 1
                sl = nx % X_RING
                while not full_x[sl].done(phase_x[sl]):
                    yield
                phase_x[sl] += 1
                s0 = (nd + i) % D_RING
                first = min(D_RING - s0, 3)                  # rows up to the ring's end, then from slot 0
                sd = [s0 + j for j in range(first)] + list(range(3 - first))
                assert slot_x[sl] == ("landed", c, i)
                pipe.append(("product", c, i, sl, sd))
                pipe.append(("commit", free_x[sl]))
                pipe.append(("commit", free_d[s0]))
                if i == rows - 1:
                    pipe.append(("commit", free_d[(nd + i + 1) % D_RING]))
                    pipe.append(("commit", free_d[(nd + i + 2) % D_RING]))
                nx += 1
                yield
            nd += rows + 2
        while pipe:                                # the last commit, before the sums are read
            yield

    def bias(g):
        nd, phase_d = 0, [0] * D_RING
        for c, rows in enumerate(heights):
            for j in range(rows + 2):
                sl, nd = nd % D_RING, nd + 1
                while not full_d[sl].done(phase_d[sl]):
                    yield
                phase_d[sl] += 1
                assert slot_d[sl] == ("landed", c, j - 1), (slot_d[sl], c, j)
                yield                              # its reads
                assert slot_d[sl] == ("landed", c, j - 1), "dZ restaged under a bias warp"
                if 1 <= j <= rows:
                    biased[g].append((c, j - 1))
                free_d[sl].arrive()
                yield

    roles = [copy_engine(), tensor_pipe(), producer(), issuer()] + [bias(g) for g in range(BIAS_WARPS)]
    alive = [True] * len(roles)
    weights = [rnd.choice((1, 1, 4, 16)) for _ in roles]
    for _ in range(3000 * (sum(heights) + 3)):
        if not any(alive[2:]):
            break
        i = rnd.choices(range(len(roles)), weights)[0]
        if alive[i]:
            try:
                next(roles[i])
            except StopIteration:
                alive[i] = False
    else:
        raise AssertionError(f"no progress: {heights}, seed {seed}")
    assert not copies and not pipe
    want = [(c, i) for c, rows in enumerate(heights) for i in range(rows)]
    assert met == want and all(b == want for b in biased)


def chunks_of_blocks(B, H, W, sms=152):
    """The chunk heights of each block of a launch, as wgrad() sizes its grid."""
    chunk = conv_chunk(B, H, W, sms)
    cols = B * -(-W // 128)
    per = -(-H // chunk)
    total = cols * per
    grid = min(total, 2 * sms)
    h = [min(chunk, H - y * chunk) for y in range(per)]
    return [[h[c % per] for c in range(b, total, grid)] for b in range(grid)]


@pytest.mark.parametrize("rows", [1, 2, 3, 4, 5, 6, 7, 20, 54])
@pytest.mark.parametrize("chunks", [1, 2, 5])
def test_protocol_under_random_schedules(rows, chunks):
    for seed in range(10):
        simulate([rows] * chunks, seed)


def test_protocol_over_uneven_chunks():
    rnd = random.Random(0)
    for seed in range(60):
        simulate([rnd.randint(1, 9) for _ in range(rnd.randint(2, 6))], seed)


@pytest.mark.parametrize("B,H,W", [(16, 256, 256), (51, 17, 257), (40, 3, 260), (700, 2, 20), (330, 9, 40), (110, 2, 300),
                                   (1300, 1, 17)])
def test_every_row_of_a_launch_is_taken_once(B, H, W):
    blocks = chunks_of_blocks(B, H, W)
    assert sum(map(sum, blocks)) == B * -(-W // 128) * H
    # one chunk a block, unless the columns alone are more than the grid's blocks
    assert (max(map(len, blocks)) > 1) == (B * -(-W // 128) > 304)
    simulate(max(blocks, key=len), seed=B)


def test_kernel_text_matches_the_model():
    src = SRC.read_text()
    for line in ("mbar_init(&free_d[i], 1 + 4);", "nd += (unsigned)k.rows + 2;",
                 "for (int j = i == 0 ? 0 : 2; j <= 2 && ok; ++j) {",
                 "first = kWgDRing - s0 < 3 ? kWgDRing - s0 : 3;", "const int chunk = conv_chunk(B, H, W, sm_count);"):
        assert line in src, line


@pytest.mark.parametrize("old,new", [
    # a row is copied into a slot before the products of its previous row completed
    ("while not free_x[sl].done(phase_x[sl]):", "while False:"),
    ("while not free_d[sl].done(phase_d[sl]):", "while False:"),
    # the chunk's last two dZ rows are never released
    ("if i == rows - 1:", "if False:"),
    # the halo rows are left out of the running count from one chunk to the next
    ("            nd += rows + 2\n", "            nd += rows\n"),
    # the issuer waits for its newest dZ row only on the first X row
    ("range(0 if i == 0 else 2, 3)", "range(0 if i == 0 else 3, 3)"),
    # the ring's end is not looked at
    ("first = min(D_RING - s0, 3) ", "first = 3 "),
    # the bias warps do not release the rows they read
    ("                free_d[sl].arrive()\n                yield\n", "                yield\n"),
])
def test_model_catches_planted_protocol_mistakes(old, new):
    src = inspect.getsource(simulate)
    assert src.count(old) == 1, old
    ns = dict(globals())
    exec(src.replace(old, new), ns)
    failures = 0
    for seed in range(24):
        try:
            ns["simulate"]([17, 3, 8], seed)
        except (AssertionError, KeyError):
            failures += 1
    assert failures > 0
