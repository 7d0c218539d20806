"""CPU checks of the launch shapes of the tensor-core GEMM: rings, issuers and shared memory as the library would launch
them, held against a model of the kernel's barrier protocol."""
import ctypes
import functools
import os
import random
import re

import pytest

from paper_2206_07446_b200 import binding as nb

CSRC = os.path.join(os.path.dirname(nb.LIB_PATH), "csrc")
FIELDS = ("BN", "splits", "rows", "m_tiles", "issuers", "ring", "tmem_cols", "bar_off", "recv_off", "stage_off", "smem",
          "stage_bytes", "threads")
X3, BF16_CVT, ROUNDED = 2, 3, 8


def shape(mode, M, N, batch, nkb, tma_out, addend):
    out = (ctypes.c_int32 * len(FIELDS))()
    st = ctypes.CDLL(nb.LIB_PATH).nnv_internal_gemm_shape(mode, M, N, batch, nkb, int(tma_out), int(addend), out)
    return None if st else dict(zip(FIELDS, out))


def cases(n, seed):
    """Kernel mode, M, N, batch, K blocks, write-out by TMA, residual: shapes of layers from 1 x 1 to 224 x 224."""
    rng = random.Random(seed)
    for _ in range(n):
        mode = rng.randrange(9)
        side, wide = rng.choice((7, 10, 14, 21, 28, 42, 56, 84, 112, 169, 224)), rng.random() < 0.5
        M = side * side if wide else max(1, int(2 ** rng.uniform(0, 15.7)))
        N = rng.choice((16, 24, 64, 96, 128, 160, 256, 512, 1024)) if wide else max(1, int(2 ** rng.uniform(0, 11)))
        yield (mode, M, N, rng.choice((16, 36, 64)) if mode == X3 else rng.choice((1, 1, 1, 16)) if mode < 2 else 1,
               max(1, int(2 ** rng.uniform(0, 8))), rng.random() < 0.7, rng.random() < 0.3)


@functools.lru_cache(maxsize=None)
def early_pass(ring, issuers, nkb, converted, groups=1):
    """True if an issuer can take a ring slot for full before the block it wants has arrived, for some block whose load takes
    longer than all others'.  Barriers are phase counters; a wait for parity p passes while the current phase's parity is not p.
    converted: the issuers wait for `groups` groups of warps that convert the blocks in turn."""
    for late in range(min(nkb, 3 * ring)):
        full, conv, empty = [0] * ring, [0] * ring, [0] * ring
        loads, converts, nxt, held = 0, list(range(groups)), list(range(issuers)), False
        moved = True
        while moved:
            moved = False
            if loads < nkb and (loads < ring or empty[loads % ring] >= loads // ring):
                if loads == late:
                    held = True
                else:
                    full[loads % ring] += 1
                loads += 1
                moved = True
            for k in range(groups):
                it = converts[k]
                if converted and it < nkb and (full[it % ring] & 1) != (it // ring & 1):
                    if full[it % ring] <= it // ring:
                        return True
                    conv[it % ring] += 1
                    converts[k] += groups
                    moved = True
            ready = conv if converted else full
            for k in range(issuers):
                it = nxt[k]
                if it < nkb and (ready[it % ring] & 1) != (it // ring & 1):
                    if ready[it % ring] <= it // ring:
                        return True
                    empty[it % ring] += 1
                    nxt[k] += issuers
                    moved = True
            if not moved and held:
                held, moved = False, True
                full[late % ring] += 1
    return False


def test_the_model_finds_the_hazard():
    # a ring of three that two issuers share: block 0 late, block 1 in time, and the slot of block 3 looks full
    assert early_pass(3, 2, 8, False) and early_pass(7, 2, 18, False) and early_pass(1, 2, 2, False) and early_pass(1, 2, 2, True)
    assert early_pass(3, 2, 8, True, 2) and early_pass(3, 1, 8, True, 2)           # two groups of converting warps on an odd ring
    # one issuer, an even ring, a ring that is never refilled, blocks converted in order
    assert not any(early_pass(*a) for a in ((3, 1, 8, False), (4, 2, 40, False), (3, 2, 3, False), (7, 2, 7, False), (3, 2, 40, True), (4, 2, 40, True, 2)))


@pytest.mark.parametrize("tuning", ["", "gemm_ring=3", "gemm_ring=5", "gemm_ring=7", "gemm_tile=128,2", "gemm_tile=64,1;gemm_ring=7"])
def test_no_issuer_runs_ahead_of_a_load(tuning):
    nb.nnv_tuning_set(tuning)
    try:
        seen = 0
        for c in cases(4000, 7):
            s = shape(*c)
            if s is None:
                continue
            seen += 1
            assert s["issuers"] in (1, 2) and (c[0] != BF16_CVT or s["issuers"] == 1)
            for nkb in {c[4] // s["splits"], -(-c[4] // s["splits"])}:
                assert not early_pass(s["ring"], s["issuers"], min(nkb, 6 * s["ring"]), c[0] in (X3, ROUNDED),
                                      s["issuers"] if c[0] == ROUNDED else 1), (c, s)
        assert seen > 3000
    finally:
        nb.nnv_tuning_set("")


@pytest.mark.parametrize("tuning", ["", "gemm_tile=128,8", "gemm_tile=96,2;gemm_ring=2"])
def test_clusters_that_fit_an_sm_find_their_tmem_columns(tuning):
    """A cluster's CTA takes at least the share of an SM's 228 KB of shared memory (1 KB of it the system's) that its TMEM
    columns are of 512: tcgen05.alloc then never waits for a CTA that waits for a member of its own cluster."""
    nb.nnv_tuning_set(tuning)
    try:
        split = 0
        for c in cases(4000, 11):
            s = shape(*c)
            if s is None or s["splits"] == 1:
                continue
            split += 1
            assert (s["smem"] + 1024) * 512 >= 228 * 1024 * s["tmem_cols"], (c, s)
        assert split > 500
    finally:
        nb.nnv_tuning_set("")


def test_no_arrival_without_a_waiter():
    """A tcgen05.commit arrives on its own time: on a slot's "empty" barrier only where the slot is refilled, that is, where a
    producer waits for it before the CTA can leave."""
    found = 0
    for f in sorted(os.listdir(CSRC)):
        if f.endswith((".cu", ".cuh")):
            for line in open(os.path.join(CSRC, f)):
                if re.search(r"umma_commit\(\w*empty", line):
                    found += 1
                    assert re.search(r"if \(.*(\+ .* < |refill_[ab]-- > 0).*\) umma_commit", line), (f, line)
    assert found >= 9


def test_the_next_kernel_is_let_in_after_the_tmem_allocation():
    """CTAs let in earlier could take columns that this grid's still need, and keep them until this grid is done."""
    kernels = 0
    for f in sorted(os.listdir(CSRC)):
        if f.endswith((".cu", ".cuh")):
            for body in open(os.path.join(CSRC, f)).read().split("__global__")[1:]:
                if "tcgen05.alloc" in body:
                    kernels += 1
                    assert body.index("tcgen05.alloc") < body.rindex("pdl_wait();", 0, body.index("pdl_trigger();")), (f, body[:200])
    assert kernels == 7


def test_warp_wide_instructions_follow_a_reconvergence():
    """tcgen05.ld and the cluster barriers are .aligned: one instruction of a whole warp, whose lanes may just have left a loop or
    a branch on their own."""
    for f in sorted(os.listdir(CSRC)):
        if f.endswith((".cu", ".cuh")):
            src = open(os.path.join(CSRC, f)).read()
            for m in re.finditer(r"void (tmem_ld\w+)\(uint32_t", src):
                assert src[m.end():].split("{", 1)[1].lstrip().startswith("__syncwarp();"), (f, m.group(1))
            lines = [ln.split("//")[0].strip() for ln in src.split("\n")]
            code = [ln for ln in lines if ln]
            for i, ln in enumerate(code):
                own = re.match(r"(asm volatile\(.barrier\.cluster\.arrive|cluster_arrive\w*\(\);|cluster_sync_all\(\);)", ln)
                if own and "cluster_arrive();" not in ln:
                    back = code[max(0, i - 3):i]
                    assert any("__syncwarp();" in b or "__syncthreads();" in b for b in back) or "cluster_arrived" in code[i + 1], (f, ln, back)


def halo_shape(C, H, W, N):
    out = (ctypes.c_int32 * 9)()
    assert ctypes.CDLL(nb.LIB_PATH).nnv_internal_conv3x3_shape(C, H, W, N, out) == 0
    return dict(zip(("use", "MT", "BN", "splits", "na", "nb", "tmem_cols", "smem", "gemm_waves"), out))


def test_split_halo_layers_run_in_one_wave_of_whole_clusters():
    """A second wave costs the split 3x3 kernel as much as the first.  Clusters of 2 / 4 / 8 CTAs that run at once with one, two and
    three CTAs to an SM, as the occupancy API reports them on this GPU (132 ... 416 for four: GPCs hold no whole number of them)."""
    slots = {1: (148, 296, 444), 2: (148, 296, 444), 4: (132, 284, 416), 8: (120, 264, 384)}
    rng, used, split = random.Random(3), 0, 0
    layers = [(32 * rng.randrange(1, 25), rng.randrange(7, 240), rng.randrange(7, 240), rng.randrange(1, 520)) for _ in range(4000)]
    layers += [(384, 48, 48, 512), (512, 40, 56, 512), (384, 80, 80, 256), (512, 160, 160, 64)]
    for C, H, W, N in layers:
        t = halo_shape(C, H, W, N)
        if not t["use"]:
            assert t["gemm_waves"] == 1
            continue
        used += 1
        tiles = -(-H // 16) * -(-W // 8) * -(-N // t["BN"])
        occ = min(3, 227 * 1024 // (t["smem"] + 1024), 512 // t["tmem_cols"])
        assert t["splits"] <= -(-C // 32) and t["smem"] <= 200 * 1024
        if t["splits"] > 1:
            split += 1
            assert tiles * t["splits"] <= slots[t["splits"]][occ - 1], (C, H, W, N, t)
    assert used > 1000 and split > 100


@pytest.mark.parametrize("C,N,H,W,splits", [
    (64, 64, 224, 224, 1), (128, 256, 112, 112, 1), (512, 512, 72, 72, 1), (512, 256, 56, 56, 4), (384, 256, 80, 80, 4),   # the halo kernel's
    (128, 128, 112, 112, 0), (64, 64, 180, 180, 0), (384, 512, 48, 48, 0), (512, 512, 40, 56, 0), (256, 512, 56, 56, 0)])  # the GEMM's
def test_halo_kernel_takes_the_layers_it_was_measured_to_win(C, N, H, W, splits):
    t = halo_shape(C, H, W, N)
    assert (t["splits"] if t["use"] else 0) == splits
