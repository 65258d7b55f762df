"""Order of the halo exchange between the tiles of the shared-memory SOR solve,
on the CPU: a model of the kernel's schedule (load the halo, update, publish the
rim, one grid barrier per sweep, the whole tile to phi at the end) with the copies
that ekl_rim.h names, over every interleaving of the blocks' loads and stores.
A block held up behind the barrier must still load what its neighbour published
in the sweep before, not what it publishes now."""
import ctypes
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "..", "paper_1710_09421_gb300", "csrc")


@pytest.fixture(scope="module")
def copies(tmp_path_factory):
    d = tmp_path_factory.mktemp("rim")
    src, so = d / "rim.cpp", d / "librim.so"
    src.write_text('#include "ekl_rim.h"\n'
                   'extern "C" int load(int k) { return ekl::rim_load_copy(k); }\n'
                   'extern "C" int store(int k) { return ekl::rim_store_copy(k); }\n')
    subprocess.run(["g++", "-shared", "-fPIC", "-I", CSRC, str(src), "-o", str(so)], check=True)
    lib = ctypes.CDLL(str(so))
    return lib.load, lib.store


def _program(load, store, tiles, me, sweeps, converged):
    """What block `me` of a ring does, as steps on the two copies of each rim:
    ("load", copy, block, wanted) and ("store", copy, value); values count the
    sweeps a rim has seen."""
    nbrs = sorted({(me - 1) % tiles, (me + 1) % tiles})
    prog = [("load", 0, b, 0) for b in nbrs]  # the starting guess, from phi
    for k in range(sweeps):
        if k > 0:
            prog += [("load", load(k), b, k) for b in nbrs]
        prog += [("store", store(k), k + 1), ("barrier",)]
    if converged:  # found at the top of one more sweep, after its halo loads
        prog += [("load", load(sweeps), b, sweeps) for b in nbrs]
    prog.append(("store", 0, sweeps))
    return prog


@pytest.mark.parametrize("tiles", [2, 3])
@pytest.mark.parametrize("sweeps", [1, 2, 3, 4])
@pytest.mark.parametrize("converged", [False, True])
def test_every_interleaving_loads_the_sweep_before(copies, tiles, sweeps, converged):
    progs = [_program(*copies, tiles, b, sweeps, converged) for b in range(tiles)]
    start = (tuple([0] * tiles), tuple([(0, None)] * tiles))
    seen, todo = {start}, [start]
    while todo:
        pc, mem = todo.pop()
        at = [progs[b][pc[b]] if pc[b] < len(progs[b]) else None for b in range(tiles)]
        nxt = []
        if all(a == ("barrier",) for a in at):
            nxt.append((tuple(p + 1 for p in pc), mem))
        for b, a in enumerate(at):
            if a is None or a == ("barrier",):
                continue
            m = mem
            if a[0] == "load":
                assert mem[a[2]][a[1]] == a[3], (b, pc, mem)
            else:
                rim = list(mem[b])
                rim[a[1]] = a[2]
                m = mem[:b] + (tuple(rim),) + mem[b + 1:]
            nxt.append((pc[:b] + (pc[b] + 1,) + pc[b + 1:], m))
        for s in nxt:
            if s not in seen:
                seen.add(s)
                todo.append(s)
    # every block reached its end and phi holds the last sweep
    done = [m for p, m in seen if all(p[b] == len(progs[b]) for b in range(tiles))]
    assert done and all(rim[0] == sweeps for m in done for rim in m)
