"""The order in which the chain kernel's roles take tiles and blocks.

On the CPU: its barriers (a ring of four per kind, one parity bit each), with the roles as coroutines that
take random times, for passes of one to three blocks: no role passes a barrier early (it would write over
a slot that is still to be read), and none waits for good.  On the GPU: passes of two blocks over scattered
qubits, whose stores are slow, against the same circuit by another method, and bit for bit again."""
import heapq
import os
import random
import shutil
import subprocess

import numpy as np
import pytest

import workloads as W
from conftest import ROOT

RING = 4


class Barrier:
    def __init__(self, count):
        self.count = self.missing = count
        self.phase = 0

    def arrive(self):
        self.missing -= 1
        assert self.missing >= 0
        if self.missing == 0:
            self.phase += 1
            self.missing = self.count

    def passed(self, parity):
        return (self.phase & 1) != parity


def simulate(nblk, tiles, group, seed):
    """None, or the waits of the roles that are left when nothing moves; AssertionError when a slot is written
    over before it has been read.  Threads of a warp as one, the four warps of a role apart."""
    r = random.Random(seed)
    nload, nstore = {1: (3, 3), 2: (2, 2), 3: (2, 1)}[nblk]   # chain_pass_desc
    ring = lambda c: [Barrier(c) for _ in range(RING)]   # noqa: E731
    full, lread, done, stored = ring(1), ring(4), ring(4), ring(1)
    mfull, mread = [ring(4), ring(4)], [ring(4), ring(4)]
    halves = lambda c: [[[Barrier(c) for _ in range(2)] for _ in range(2)] for _ in range(2)]   # noqa: E731
    afull, aempty = halves(4), halves(1)
    dfull, dempty, nsum = [Barrier(1), Barrier(1)], [Barrier(4), Barrier(4)], [Barrier(4), Barrier(4)]
    took = {k: r.choice([0.1, 1, 5] + ([30] if k in ("load", "store") else [])) for k in ("prod", "epi", "mma", "load", "store")}
    read, stores = {}, [-1]

    def items(g):
        it = 0
        for step in range(tiles + nblk - 1):
            for b in range(nblk):
                if 0 <= step - b < tiles and group[step, nblk, b] == g:
                    yield step - b, b, it
                    it += 1

    def producer(g):
        for t, b, it in items(g):
            yield (full if b == 0 else mfull[b - 1])[t % RING], t // RING & 1, ("producer", g, t, b)
            yield took["prod"]
            for h in range(2):
                yield aempty[g][it & 1][h], (it >> 1 & 1) ^ 1, ("operand", g, t, b, h)
                yield took["prod"]
                afull[g][it & 1][h].arrive()
            read[t, b] = read.get((t, b), 0) + 1
            (lread if b == 0 else mread[b - 1])[t % RING].arrive()

    def epilogue(g):
        turn = 0
        for t, b, it in items(g):
            yield dfull[g], it & 1, ("accumulator", g, t, b)
            yield took["epi"]
            dempty[g].arrive()
            last = b + 1 == nblk
            if last:
                nsum[g].arrive()
                yield nsum[g], turn & 1, ("norm", g, t)
                turn += 1
            back = nstore if last else 1
            if t >= back:
                yield (stored if last else mread[b])[(t - back) % RING], (t - back) // RING & 1, ("slot", g, t, b)
                assert stores[0] >= t - back if last else read.get((t - back, b + 1)) == 4, ("written over", t, b)
            yield took["epi"]
            (done if last else mfull[b])[t % RING].arrive()

    def issuer(g):
        for t, b, it in items(g):
            yield dempty[g], (it & 1) ^ 1, ("issue", g, t, b)
            for h in range(2):
                yield afull[g][it & 1][h], it >> 1 & 1, ("operand full", g, t, b, h)
            m = took["mma"]
            later.extend([(now[0] + m * r.random(), aempty[g][it & 1][0]), (now[0] + m, aempty[g][it & 1][1]), (now[0] + 1.1 * m, dfull[g])])
            yield 0.1

    def loader():
        for t in range(tiles):
            if t >= nload:
                yield lread[(t - nload) % RING], (t - nload) // RING & 1, ("load", t)
                assert read.get((t - nload, 0)) == 4, ("loaded over", t)
            later.append((now[0] + took["load"] * r.random(), full[t % RING]))
            yield 0.1

    def storer():
        for t in range(tiles):
            yield done[t % RING], t // RING & 1, ("store", t)
            yield took["store"]
            stores[0] = t
            stored[t % RING].arrive()

    now, later, waiting = [0.0], [], {}
    roles = [f(g) for f in (producer, epilogue) for g in (0, 1) for _ in range(4)] + [issuer(0), issuer(1), loader(), storer()]
    ready = [(0.0, i) for i in range(len(roles))]
    left = len(roles)
    while left:
        for i in [i for i, w in waiting.items() if w[0].passed(w[1])]:
            del waiting[i]
            heapq.heappush(ready, (now[0] + 0.05 * r.random(), i))
        if not ready and not later:
            return sorted(w[2] for w in waiting.values())
        now[0] = max(now[0], min([x[0] for x in ready[:1]] + [x[0] for x in later]))
        for x in [x for x in later if x[0] <= now[0]]:
            later.remove(x)
            x[1].arrive()
        while ready and ready[0][0] <= now[0]:
            i = heapq.heappop(ready)[1]
            try:
                w = next(roles[i])
            except StopIteration:
                left -= 1
                continue
            if isinstance(w, tuple):
                waiting[i] = w
            else:
                heapq.heappush(ready, (now[0] + w * r.random() * (10 if r.random() < 0.02 else 1), i))
    return None


@pytest.fixture(scope="module")
def group(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("g++ not available")
    exe = tmp_path_factory.mktemp("order") / "chain_order_dump"
    cuda_inc = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
    subprocess.run(["g++", "-O1", "-std=c++17", os.path.join(ROOT, "tests", "chain_order_dump.cpp"), "-I",
                    os.path.join(ROOT, "paper_2008_13490_gb300", "csrc"), "-I", os.path.join(ROOT, "include"), "-I", cuda_inc,
                    "-o", str(exe)], check=True, capture_output=True, text=True)
    rows = subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.split()
    x = np.array(rows, dtype=int).reshape(-1, 4)
    return {(int(s), int(k), int(b)): int(g) for s, k, b, g in x}


@pytest.mark.parametrize("nblk", [1, 2, 3])
@pytest.mark.parametrize("tiles", [1, 2, 3, 5, 7, 8, 9, 10, 11, 12, 13, 25])
def test_barriers(group, nblk, tiles):
    for seed in range(40):
        assert simulate(nblk, tiles, group, 1000 * seed + tiles) is None, seed


def test_the_simulation_sees_a_pipeline_that_comes_early(group):
    # the order counted over the items alone: the last tile's last block falls to the other pipeline
    tiles, counted, k = 9, {}, 0
    for step in range(tiles + 1):
        for b in range(2):
            if 0 <= step - b < tiles:
                counted[step, 2, b] = k & 1
                k += 1
    with pytest.raises(AssertionError, match="written over"):
        for seed in range(200):
            assert simulate(2, tiles, counted, seed) is None


@pytest.mark.gpu
@pytest.mark.parametrize("n", [22, 24])
def test_passes_of_two_blocks_over_scattered_qubits(qs, n):
    # two dense blocks on every other qubit from 4 on: single positions in the tile (64 copies a tile), 6 to 27
    # tiles a CTA
    g = W.rng(n)
    qubits = [4, 6, 8, 10, 12, 14, 16, 18]
    ops = []
    for block in (qubits[:5], qubits[3:8]):
        for layer in range(4):
            ops += [("MAT1", (q,), (), W.haar_su2(g)) for q in block]
            ops += [("CZ", (block[i], block[i + 1]), (), None) for i in range(layer % 2, len(block) - 1, 2)]
    psi = W.random_state(n, g).astype(np.complex64)
    outs = []
    for method in [qs.METHOD_TILED] + [qs.METHOD_AUTO] * 12:
        st = qs.State(n, qs.QS_C64)
        qs.sv_copy_in(st, psi)
        stats = qs.sv_apply_circuit(st, ops, method)
        outs.append(qs.sv_copy_out(st))
        st.close()
    assert stats["passes"] == 1 and stats["ops_fused"] == 2 and stats["tile_launches"] == 0
    assert np.linalg.norm(outs[1] - outs[0]) <= 4 * np.sqrt(len(ops)) * 2.0 ** -23
    for out in outs[2:]:
        assert np.array_equal(out.view(np.uint64), outs[1].view(np.uint64))
