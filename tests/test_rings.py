"""Host logic of the tensor-core kernels: lengths of the rings that their roles hand blocks round in (csrc/bpdq_rings.h).

A role that waits on an mbarrier by parity is let through at once when the barrier's phase BEFORE the awaited one is still
open.  So for every wait that phase has to be over, by what the waiting role has itself waited for, whatever the copies' and the
other roles' delays.  The kernels' order constraints are laid out as a graph, and the end of the phase before must be reachable
from every wait; a copy may land arbitrarily late, also later than copies that were requested after it."""
import glob
import os
import re
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HEADER_DIR = os.path.join(ROOT, "paper_2602_04163_b200", "csrc")

DRIVER = r"""
#include <cstdio>
#include <cstdlib>
#include "bpdq_rings.h"
int main(int argc, char** argv) {
    if (argc == 5) {
        const bpdq::TsSplit w = bpdq::ts_split(atoi(argv[1]), atoi(argv[2]), atoi(argv[3]), atoi(argv[4]));
        printf("%d %d %d %d %d\n", w.grid, w.whole, w.cut_begin, w.cut_units, w.cut_step);
        return 0;
    }
    if (argc == 6) {
        printf("%d\n", bpdq::wide_half(atoi(argv[1]), atoi(argv[2]), atoi(argv[3]), atoi(argv[4]), atoi(argv[5])));
        return 0;
    }
    if (argc == 4) {
        printf("%d\n", bpdq::gather_tokens(atoi(argv[1]), atoi(argv[2]), 148, atoi(argv[3])));
        return 0;
    }
    for (int K = 1; K <= 4; ++K)
        for (int half = 16; half <= 256; half += 16) {
            const int bkw = half <= bpdq::kWideLongHalf ? 64 : 32;
            const bpdq::WideRings r = bpdq::wide_rings(K, bkw, half);
            const int groups = bpdq::wide_groups(K, half);
            printf("wide %d %d %d %d %d %d %d %d\n", K, half, 128 / bkw, r.stages, r.sp,
                   bpdq::kWideSmem - r.stages * bpdq::wide_stage_bytes(bkw, half) - r.sp * bpdq::wide_block_bytes(K), groups, bpdq::wide_releases(groups));
        }
    for (int K = 1; K <= 4; ++K)
        for (int cols = 16; cols <= 128; cols += 16) {
            const bpdq::TsRings r = bpdq::ts_rings(K, cols);
            printf("ts %d %d %d %d %d\n", K, cols, r.sx, r.sp, bpdq::kTsSmem - r.sx * cols * 256 - r.sp * bpdq::ts_slot_bytes(K));
        }
    printf("release %d %d\n", bpdq::wide_release_stage(4), bpdq::wide_release_stage(2));
    return 0;
}
"""


@pytest.fixture(scope="module")
def driver(tmp_path_factory):
    d = tmp_path_factory.mktemp("rings")
    src, exe = d / "driver.cpp", d / "driver"
    src.write_text(DRIVER)
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", HEADER_DIR, str(src), "-o", str(exe)], check=True)
    return str(exe)


@pytest.fixture(scope="module")
def rings(driver):
    rows = [line.split() for line in subprocess.run([driver], check=True, capture_output=True, text=True).stdout.splitlines()]
    return [(r[0], [int(v) for v in r[1:]]) for r in rows]


class Order:
    """Events with what must have happened before them; waits with the event that ends the phase before the awaited one."""

    def __init__(self):
        self.before, self.waits = {}, []

    def event(self, name, *after):
        self.before[name] = {a for a in after if a is not None}

    def wait(self, role, after, previous):
        """`role` begins to wait once `after` has happened; `previous` must be over then."""
        self.waits.append((role, after, previous))

    def _happened(self, name):
        seen, todo = set(), [name]
        while todo:
            e = todo.pop()
            if e in seen or e is None:
                continue
            seen.add(e)
            todo += self.before[e]
        return seen

    def open_waits(self):
        return [(role, previous) for role, after, previous in self.waits
                if previous in self.before and (after is None or previous not in self._happened(after))]


def ts_order(sx, sp, blocks, groups=4, issuers=2):
    """gemm_ts_kernel: packed producer, x producer, decode groups (group q mod 4 takes block q), issuers (issuer q mod 2)."""
    o = Order()

    def ev(kind, q):
        return (kind, q) if q >= 0 else None
    for q in range(blocks):
        # producers: one thread each, in block order; a slot is free once the block before in it has been decoded / multiplied
        o.event(("packed asked", q), ev("packed asked", q - 1), ev("decoded", q - sp))
        o.wait("packed producer", ev("packed asked", q - 1), ev("decoded", q - 2 * sp))
        o.event(("packed landed", q), ("packed asked", q))
        o.event(("x asked", q), ev("x asked", q - 1), ev("multiplied", q - sx))
        o.wait("x producer", ev("x asked", q - 1), ev("multiplied", q - 2 * sx))
        o.event(("x landed", q), ("x asked", q))
        # a group: waits for the packed block, decodes into registers, waits for its A slot, stores and arrives
        o.wait("group, packed", ev("decoded", q - groups), ev("packed landed", q - sp))
        o.wait("group, A slot", ev("decoded", q - groups), ev("multiplied", q - 2 * groups))
        o.event(("decoded", q), ev("decoded", q - groups), ("packed landed", q), ev("multiplied", q - groups))
        # an issuer: waits for x, then for the A slot; its commits complete in order
        o.wait("issuer, x", ev("issued", q - issuers), ev("x landed", q - sx))
        o.wait("issuer, A slot", ev("issued", q - issuers), ev("decoded", q - groups))
        o.event(("issued", q), ev("issued", q - issuers), ("x landed", q), ("decoded", q))
        o.event(("multiplied", q), ("issued", q), ev("multiplied", q - issuers))
    return o


def test_rings_up_to_128_tokens(rings):
    """Every K and number of token columns: no wait can pass by a phase that is still open, and the rings fit shared memory."""
    seen = 0
    for kind, r in rings:
        if kind != "ts":
            continue
        K, cols, sx, sp, left = r
        seen += 1
        assert left >= 1024 + 8 * (2 * 4 + 4 + 2 * sx + 2 * sp) + 16, r      # alignment slack, barriers, TMEM address and flags
        assert 4 <= sx <= 8 and 8 <= sp <= 24, r
        assert ts_order(sx, sp, 2 * sp + 40).open_waits() == [], r
    assert seen == 32


def test_the_order_model_sees_an_odd_ring():
    """The model itself: nine packed slots beside four of x (K = 4 with 128 tokens, were the length not rounded) leave a group's
    wait for its packed block open."""
    assert {role for role, _ in ts_order(4, 9, 60).open_waits()} == {"group, packed"}
    assert ts_order(8, 23, 100).open_waits() == []           # an odd ring that the x ring covers


def wide_order(stages, sp, per_block, blocks, groups, releases, issuers, release, tile=5, accs=2):
    """gemm_wide_kernel: x producer, packed producer, decode groups (group b mod groups takes block b), issuers that all multiply every
    stage, epilogue.  A stage slot's uses are released through `releases` barriers in turn, so the phase before the awaited one is
    releases + 1 uses back; tiles of `tile` blocks take `accs` accumulators with barriers of their own in turn."""
    o = Order()

    def ev(kind, q):
        return (kind, q) if q >= 0 else None
    for b in range(blocks):
        o.event(("packed asked", b), ev("packed asked", b - 1), ev("stored", (b - sp) * per_block + release) if b >= sp else None)
        o.wait("packed producer", ev("packed asked", b - 1), ev("stored", (b - 2 * sp) * per_block + release) if b >= 2 * sp else None)
        o.event(("packed landed", b), ("packed asked", b))
        j = b // tile
        for it in range(b * per_block, (b + 1) * per_block):
            o.event(("x asked", it), ev("x asked", it - 1), ev("multiplied", it - stages))
            o.wait("x producer", ev("x asked", it - 1), ev("multiplied", it - (releases + 1) * stages))
            o.event(("x landed", it), ("x asked", it))
            before = ev("stored", it - 1) if it % per_block else ev("stored", (b - groups + 1) * per_block - 1)    # the group's stage before
            if it % per_block == 0:
                o.wait("group, packed", before, ev("packed landed", b - sp))
            o.wait("group, stage", before, ev("multiplied", it - (releases + 1) * stages))
            o.event(("stored", it), before, ("packed landed", b), ev("multiplied", it - stages))
            for i in range(issuers):
                last = ev(f"issued {i}", it - 1)
                if it == j * tile * per_block:              # a tile's first stage: its accumulator has been drained of tile j - accs
                    o.wait("issuer, accumulator", last, ev("drained", j - 2 * accs))
                    o.event((f"accumulator {i}", j), last, ev("drained", j - accs))
                    last = (f"accumulator {i}", j)
                o.wait("issuer", last, ev("full", it - stages))
                o.event((f"issued {i}", it), last, ("full", it))
            o.event(("full", it), ("stored", it), ("x landed", it))
            o.event(("multiplied", it), *((f"issued {i}", it) for i in range(issuers)), ev("multiplied", it - 1))
        if b % tile == tile - 1:                            # the tile's last commits fill its accumulator, the epilogue drains it
            o.event(("filled", j), ("multiplied", (b + 1) * per_block - 1))
            o.wait("epilogue", ev("drained", j - 1), ev("filled", j - accs))
            o.event(("drained", j), ev("drained", j - 1), ("filled", j))
    return o


def test_rings_of_the_prefill_kernel(rings):
    """Every K and half tile, with the groups and issuers that it has, tiles of one block and of several: no wait can pass by a phase that is
    still open, the rings and barriers fit shared memory, and the release barriers of a slot are no more than the shortest ring takes."""
    (release,) = [r for kind, r in rings if kind == "release"]
    seen, needed = 0, set()
    for kind, r in rings:
        if kind != "wide":
            continue
        K, half, per_block, stages, sp, left, groups, releases = r
        seen += 1
        assert groups == 4 or releases == 1, r
        assert groups in (2, 4) and sp % groups == 0 and (K < 4 or groups == 2), r
        assert left >= 1024 + 8 * ((1 + releases) * stages + 2 * sp + 4) + 8, r     # alignment slack, barriers, TMEM address and flag
        whole = half <= 128                                  # one issuer and two accumulators, else two and one
        shape = (stages, sp, per_block, 2 * sp + 3 * stages + 8, groups)
        last = (1 if whole else 2, release[0 if per_block == 4 else 1])
        for tile in (1, 5):
            assert wide_order(*shape, releases, *last, tile, 2 if whole else 1).open_waits() == [], r
        if releases > 1 and wide_order(*shape, releases - 1, *last).open_waits():
            needed.add(groups)
    assert seen == 64 and needed == {4}


def test_the_order_model_of_the_prefill_kernel_sees_what_would_not_do():
    assert wide_order(4, 2, 4, 20, 2, 1, 2, 2).open_waits()                     # four stages of 32 columns
    assert wide_order(3, 4, 2, 40, 4, 2, 1, 1).open_waits()                     # three of 64 with four groups
    assert wide_order(6, 6, 2, 40, 4, 2, 1, 1).open_waits()                     # a packed ring that is no multiple of the groups
    assert {role for role, _ in wide_order(6, 4, 2, 40, 4, 1, 1, 1).open_waits()} == {"group, stage"}     # one release barrier


@pytest.mark.parametrize("M,nrt,nblocks,K", [(129, 28, 28, 2), (777, 28, 148, 2), (777, 4, 28, 2), (4096, 231, 64, 3), (4096, 1, 1, 4), (513, 148, 32, 4),
                                             (131, 64, 231, 1), (8192, 64, 64, 3), (17, 192, 1, 2), (128, 256, 8, 4), (300, 1, 8, 2)])
def test_half_tiles(driver, M, nrt, nblocks, K):
    """A half tile is a multiple of 16 tokens, at most 256, and one of the equal cuts of M."""
    half = int(subprocess.run([driver, *map(str, (M, nrt, nblocks, K, 148))], check=True, capture_output=True, text=True).stdout)
    assert half % 16 == 0 and 16 <= half <= 256
    assert half in [min(256, -(-(-(-M // n)) // 32) * 16) for n in range(-(-M // 512), -(-M // 32) + 1)]


# (tokens, rows, columns, K, {half: us of the launch}) on a B200, back to back under its power limit: halves within 1.6 of the best
MEASURED_TILES = [
    (786, 29568, 8192, 2, {48: 485.4, 64: 409.8, 80: 322.4, 112: 324.6, 144: 359.7, 208: 308.1}),
    (576, 29568, 8192, 2, {48: 342.3, 64: 294.8, 80: 272.6, 96: 219.8, 144: 273.9}),
    (639, 29568, 8192, 3, {48: 391, 64: 315.8, 80: 303.6, 112: 248.8, 160: 276.2}),
    (839, 29568, 8192, 3, {48: 533, 64: 440.8, 80: 429, 96: 369.4, 112: 356.8, 144: 369.4, 224: 337.1}),
    (3156, 29568, 8192, 3, {80: 1651.1, 96: 1460.6, 112: 1400.1, 128: 1269.3, 144: 1509.4, 160: 1337.8, 176: 1189.5, 208: 1239.6, 240: 1166.9}),
    (2306, 8192, 29568, 2, {64: 1254.2, 80: 1087.7, 96: 1026.7, 112: 905.3, 128: 944.8, 144: 1092.8, 160: 966.6, 176: 1014.9, 208: 888.5, 240: 990.2}),
    (1055, 8192, 29568, 3, {48: 616.1, 64: 548.9, 80: 576, 96: 474.8, 112: 495.7, 144: 494.3, 176: 455.2}),
    (3772, 8192, 29568, 2, {80: 1887.3, 96: 1626.1, 112: 1594.4, 128: 1399.9, 144: 2004.1, 160: 1523.5, 176: 1466.9, 192: 1474.6, 224: 1341, 240: 1468.8}),
    (1386, 18944, 3584, 2, {64: 184.8, 80: 168.4, 96: 165.3, 112: 153.5, 128: 141.6, 144: 148.9, 176: 138.7, 240: 125.7}),
    (1560, 18944, 3584, 3, {64: 238.9, 80: 199.1, 96: 188.6, 112: 166.1, 144: 193.2, 160: 168.7, 208: 153.2}),
    (2796, 3584, 18944, 2, {80: 358.7, 96: 304.5, 112: 314.1, 128: 327.9, 144: 311.6, 160: 292.6, 176: 317.9, 208: 335.1, 240: 375.5}),
    (184, 3584, 18944, 1, {32: 69.2, 48: 67.5, 96: 78}),
    (290, 29568, 8192, 4, {80: 220.1, 160: 152.9}),
    (1323, 4096, 4096, 4, {80: 61.8, 96: 65.9, 176: 41.6, 224: 46.4}),
    (1220, 1024, 8192, 4, {48: 59.1, 64: 59.9, 80: 54.5, 96: 59.8, 112: 60.6, 128: 61.3, 160: 66.3, 208: 68.5}),
    (438, 4096, 4096, 1, {32: 31.6, 48: 31.3, 64: 19.9, 80: 20.4, 112: 22.8}),
    (258, 512, 3584, 4, {16: 22.9, 32: 24.7, 48: 24.7, 80: 24.2, 144: 30.2}),
]


@pytest.mark.parametrize("M,out,in_,K,us", MEASURED_TILES)
def test_the_half_tile_that_is_taken_is_measured_fast(driver, M, out, in_, K, us):
    """Against measured launches, not against the rule's own model: no more than 5 % over the best half (two runs of a launch differ by up to
    3 % under the power limit)."""
    half = int(subprocess.run([driver, *map(str, (M, -(-out // 128), in_ // 128, K, 148))], check=True, capture_output=True, text=True).stdout)
    assert half in us and us[half] <= 1.05 * min(us.values())


def test_launches_of_several_tiles_per_cta_are_what_their_gpu_test_says(driver, rings):
    """The GPU test of CTAs that walk over tiles is only worth something while the rules give its launches these tiles."""
    from tests import gpu_util as G
    groups_of = {(r[0], r[1]): r[6] for kind, r in rings if kind == "wide"}
    nrt = -(-G.TILE_WALK_ROWS // 128)
    for K, g, in_, M, half, groups in G.TILE_WALKS:
        out = subprocess.run([driver, *map(str, (M, nrt, in_ // 128, K, 148))], check=True, capture_output=True, text=True).stdout
        assert int(out) == half and groups_of[K, half] == groups, (K, g, in_, M)
        assert nrt * -(-M // (2 * half)) > 4 * 148
        # not a call of the kernel for up to 128 tokens (ts_drain_bound)
        assert M > 128 or (M > 16 and in_ // 128 <= (8 if M > 64 else 2))
    assert {(half > 128, groups) for _, _, _, _, half, groups in G.TILE_WALKS} == {(False, 4), (False, 2), (True, 2)}


def test_prefill_slots_are_given_back_after_the_last_use(rings):
    """The stage behind which a decode group of the prefill kernel gives a packed slot back: by then every plane word and every
    coefficient group that it has loaded is part of a stored stage, for both stage widths and for one or two groups per block."""
    (release,) = [r for kind, r in rings if kind == "release"]
    for stages, at in zip((4, 2), release):
        words = 4 // stages                                   # 32-column words per stage
        for groups in (1, 2):
            need = {("plane", k) for k in range(4)} | {("coefficients", c) for c in range(groups)}
            for st in range(at + 1):
                for q in range(st * words, (st + 1) * words):
                    need -= {("plane", q), ("plane", (q + 3) % 4), ("coefficients", q // 2 if groups == 2 else 0)}
            assert not need, (stages, groups, need)
        assert at < stages


def guarded_waits(text):
    """(line, inside a block that one thread runs) for every per-thread wait whose answer decides what the thread does next."""
    text = re.sub(r"//[^\n]*", "", text)
    headers, at, found = [], 0, []
    for m in re.finditer(r"[;{}]|\bmbar_wait\(", text):
        if m.group() == "{":
            headers.append(text[at:m.start()])
        elif m.group() == "}":
            headers.pop()
        elif m.group() != ";":
            statement = text[at:m.start()].strip()
            if re.sub(r"[\w]+::", "", statement):          # a bare call's answer goes nowhere
                one = any(re.search(r"elect_one\(\)|threadIdx\.x == 0|\blane == 0", h) for h in headers)
                found.append((text.count("\n", 0, m.start()) + 1, one))
            continue
        at = m.end()
    return found


def test_warps_leave_a_wait_together():
    """A bounded wait that ran out ends the role that waited.  Lanes that each decide for themselves may part there, some at the CTA's
    last barrier and some in a warp-wide instruction, for good: code that a whole warp runs uses mbar_wait_warp (one answer for all
    lanes), the per-thread wait stands only where a single thread runs."""
    seen = 0
    for path in glob.glob(os.path.join(HEADER_DIR, "*.cu*")):
        if path.endswith("bpdq_tma.cuh"):
            continue                                        # where the waits are defined
        with open(path) as f:
            for line, one in guarded_waits(f.read()):
                assert one, f"{os.path.basename(path)}:{line}: a wait that lanes leave one by one"
                seen += 1
    assert seen >= 6


def test_landing_areas_are_refilled_behind_a_fence():
    """The few-token kernel's warps copy the next task over the one they have just loaded: every copy but a warp's very first is asked
    for behind a proxy fence of all its lanes."""
    with open(os.path.join(HEADER_DIR, "bpdq_gemv_mma.cu")) as f:
        text = re.sub(r"//[^\n]*", "", f.read())
    calls = re.findall(r"([^;{}]*)\bissue_task\(", text)
    assert len(calls) == 2 and sum("early &&" in c for c in calls) == 1       # the first copy, and the one in refill
    assert re.search(r"auto refill = [^;]*\{\s*bpdq::tma::fence_proxy_async\(\);\s*__syncwarp\(\);\s*issue_task\(", text)


@pytest.mark.parametrize("tiles,nb0,sms", [(4, 28, 148), (28, 28, 148), (36, 28, 148), (32, 32, 148), (1, 16, 148), (9, 17, 148), (8, 64, 148),
                                           (231, 64, 148), (64, 231, 148), (148, 28, 148), (296, 28, 148), (256, 4, 148), (3, 1, 148),
                                           (149, 15, 148), (37, 31, 132), (1, 1, 1)])
def test_the_work_split_covers_every_block_once(driver, tiles, nb0, sms):
    """Shares of the cut units and whole tiles together are all blocks, once each; every CTA has work; where every tile can be cut into
    shares of eight blocks at most, no share lies across two tiles."""
    units = tiles * nb0
    out = subprocess.run([driver, str(tiles), str(units), str(nb0), str(sms)], check=True, capture_output=True, text=True).stdout
    grid, whole, cut_begin, cut_units, step = (int(v) for v in out.split())
    assert 1 <= grid <= sms
    taken = [(b + grid * f) * nb0 + k for b in range(grid) for f in range(whole) for k in range(nb0)]
    shares = [cut_begin + cut_units // step * s // grid * step for s in range(grid + 1)]
    assert shares[0] == cut_begin and shares[-1] == units
    taken += range(shares[0], shares[-1])
    assert sorted(taken) == list(range(units))
    assert whole > 0 or all(a < b for a, b in zip(shares, shares[1:]))
    per_tile = -(-nb0 // 8)
    if nb0 >= 16 and tiles * per_tile <= sms:
        assert grid == tiles * per_tile
        assert all(a // nb0 == (b - 1) // nb0 for a, b in zip(shares, shares[1:]))
    if nb0 < 16:
        assert all(a % nb0 == 0 for a in shares)                # short rows are not cut


@pytest.mark.parametrize("blocks,sms", [([64, 9, 5], 148), ([28, 231], 148), ([1], 4), ([200, 17], 3)])
def test_the_work_split_of_rows_of_different_lengths(driver, blocks, sms):
    units = sum(blocks)
    out = subprocess.run([driver, str(len(blocks)), str(units), "0", str(sms)], check=True, capture_output=True, text=True).stdout
    grid, whole, cut_begin, cut_units, step = (int(v) for v in out.split())
    assert (whole, cut_begin, cut_units, step) == (0, 0, units, 1) and 1 <= grid <= min(sms, (units + 7) // 8)


def test_a_cta_that_gave_up_outlives_its_copies():
    """The last thing every kernel with bounded waits and copies does: in the tensor-core kernels once all roles have met, in the few-token
    kernel, whose warps wait for their own copies only, in each warp."""
    for name in ("bpdq_gemm_ts.cuh", "bpdq_gemm_wide.cuh"):
        with open(os.path.join(HEADER_DIR, name)) as f:
            text = f.read()
        assert re.search(r"__syncthreads\(\);\s*if \(warp == 1\) \{[^}]*\}\s*if \(\*abort_flag\) linger\(\);\s*\}\s*$", text), name
    with open(os.path.join(HEADER_DIR, "bpdq_gemv_mma.cu")) as f:
        assert re.search(r"pend_nsl\);\s*if \(\*abort_flag\) bpdq::tma::linger\(\);\s*\}\s*template", f.read())


BARRIERS = r"""
#include <cstdio>
#include "bpdq_rings.h"
constexpr int kWideEpiWarps = %(epi)s;
template <int BKW, int NG> struct Cfg {
    %(config)s
};
static void mbar_init(unsigned addr, int count) { printf("init %%u %%d\n", addr, count); }
static void fence_barrier_init() {}
template <int BKW, int NG> void layout(int K, int half) {
    using C = Cfg<BKW, NG>;
    constexpr bool kWhole = C::kWhole;
    (void)kWhole;
    const bpdq::WideRings r = bpdq::wide_rings(K, BKW, half);
    const int S = r.stages, SP = r.sp, tid = 0;
    const unsigned bar_base = 0;
    int aborted = 0, *abort_flag = &aborted;
    printf("tile %%d %%d\n", K, half);
    %(names)s
    %(init)s
    // what the roles use: three uses of every stage slot, both packed barriers, the accumulators of six tiles
    for (int n = 0; n < 3; ++n)
        for (int s = 0; s < S; ++s) printf("use %%u\nuse %%u\nuse %%u\n", full(s), empty(s, n), released(s, n));
    for (int s = 0; s < SP; ++s) printf("use %%u\nuse %%u\n", full_p(s), empty_p(s));
    for (int j = 0; j < 6; ++j) printf("use %%u\nuse %%u\nacc %%u %%u %%u\n", acc_full(j), acc_empty(j), acc_full(j), acc_empty(j), acc_parity(j));
    printf("end %%d\n", %(end)s);
}
int main() {
    for (int K = 1; K <= 4; ++K)
        for (int half = 16; half <= bpdq::kWideMaxHalf; half += 16)
            if (half > bpdq::kWideLongHalf) layout<32, 2>(K, half);
            else if (bpdq::wide_groups(K, half) == 4) layout<64, 4>(K, half);
            else layout<64, 2>(K, half);
    return 0;
}
"""


def test_every_barrier_of_the_prefill_kernel_is_initialised_once(tmp_path):
    """The kernel's own lines that lay out and initialise its barriers, run on the host: every address that a role uses is initialised, none
    twice (a second initialisation of a live mbarrier is undefined), all lie below the TMEM address, and one accumulator's barriers serve every
    tile, or two sets serve tiles in turn."""
    with open(os.path.join(HEADER_DIR, "bpdq_gemm_wide.cuh")) as f:
        text = f.read()
    kernel = text[text.index("gemm_wide_kernel(const"):]
    parts = {
        "epi": re.search(r"kWideEpiWarps = (\d+);", text).group(1),
        "config": "\n".join(re.findall(r"static constexpr (?:bool kWhole|int kIssuers|int kAccs|int kReleases) = [^;]*;", text)),
        "names": kernel[kernel.index("auto full ="):kernel.index("unsigned* tmem_slot")],
        "init": re.search(r"if \(tid == 0\) \{.*?fence_barrier_init\(\);\s*\}", kernel, re.S).group(),
        "end": re.search(r"\(bar_base - base\) \+ (8 \* \([^;]*\))\);", kernel).group(1),
    }
    src, exe = tmp_path / "barriers.cpp", tmp_path / "barriers"
    src.write_text(BARRIERS % parts)
    subprocess.run(["g++", "-O1", "-std=c++17", "-I", HEADER_DIR, str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout
    tiles = out.split("tile ")[1:]
    assert len(tiles) == 64
    for tile in tiles:
        rows = [line.split() for line in tile.splitlines()]
        half = int(rows[0][1])
        inits = [int(r[1]) for r in rows if r[0] == "init"]
        used = {int(r[1]) for r in rows if r[0] == "use"}
        (end,) = [int(r[1]) for r in rows if r[0] == "end"]
        assert len(set(inits)) == len(inits) and used == set(inits), rows[0]
        assert all(a % 8 == 0 and a + 8 <= end for a in used), rows[0]
        acc = [tuple(int(v) for v in r[1:]) for r in rows if r[0] == "acc"]
        sets = 2 if half <= 128 else 1
        assert [a[:2] for a in acc] == [acc[j % sets][:2] for j in range(6)] and len({a[:2] for a in acc}) == sets
        assert [a[2] for a in acc] == [j // sets % 2 for j in range(6)]


@pytest.mark.parametrize("in_,M,smem_optin", [(128, 295, 232448), (128, 296, 232448), (18944, 777, 232448), (24576, 4096, 232448), (28928, 4096, 232448),
                                              (29056, 4096, 232448), (29568, 4096, 232448), (51200, 4096, 232448), (102400, 500, 232448),
                                              (102528, 500, 232448), (24576, 500, 101376)])
def test_a_gather_that_stages_two_tokens_leaves_room_for_a_second_cta(driver, in_, M, smem_optin):
    """Rows that a CTA of the gather holds fit its shared memory, and two tokens are staged only where two such CTAs share an SM (whose shared
    memory is a CTA's largest opt-in and the 1 KB that every CTA costs beside its own)."""
    tokens = int(subprocess.run([driver, str(in_), str(M), str(smem_optin)], check=True, capture_output=True, text=True).stdout)
    cta = 2 * in_ * tokens
    two_ctas = 2 * (4 * in_ + 1024) <= smem_optin + 1024
    assert tokens == (2 if M >= 296 and two_ctas else 1 if 2 * in_ <= 200 * 1024 and 2 * in_ <= smem_optin else 0)
    assert cta <= smem_optin and (tokens < 2 or 2 * (cta + 1024) <= smem_optin + 1024)
    if in_ == 29568:
        assert tokens == 1                                   # the 72B-shaped down projection: 142 us with one, 191 with two
