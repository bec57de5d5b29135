"""A handle whose step was aborted steps on correctly once a state is loaded.

A step that runs out of room for its pairs is aborted in the compaction, which puts the step's counters
back.  A fused launch whose waits run out stops at a barrier and leaves them, with the tallies and cell
counts, as they then are; what such a step can leave is written into the handle's memory from the host
here (the control block's words and the arrays, found by the order of the handle's allocations), between
steps.  The recovered handle must continue exactly like a fresh one."""
import ctypes
import os
import re

import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_1107_0270_gb300 as pkg  # noqa: E402
from test_gpu_parity import dense_reversible  # noqa: E402

RD_ETIMEOUT = 4


def source(name):
    return open(os.path.join(os.path.dirname(pkg.__file__), "csrc", name)).read()


def control_words():
    """Word index of each leading 32-bit field of the control block, from its declaration."""
    at, words = 0, {}
    for line in source("rd_internal.cuh").split("struct DevCtl {")[1].split("};")[0].splitlines():
        m = re.match(r"\s*u?int32_t (\w+)(?:\[(\d+)\])?;", line)
        if m:
            words[m.group(1)] = at
            at += int(m.group(2) or 1)
        elif line.strip():
            break
    return words


class Memory:
    """Named allocations of a handle (without drift) and words written to them from the host."""

    def __init__(self, allocs):
        body = source("rd_capi.cu").split("const size_t vs = h->vsize;")[1].split("if (!ok) {")[0]
        names = [n for n in re.findall(r"^\s*(?:h->|L\.)(\w+(?:\[\d\])?) = [^;]*\bA\(", body, re.M) if n != "x0d"]
        self.at = dict(zip(names, allocs))
        self.rt = ctypes.CDLL(f"libcudart.so.{torch.version.cuda.split('.')[0]}")
        self.words = control_words()

    def write(self, name, first, values):
        ptr, size = self.at[name]
        buf = np.ascontiguousarray(values, np.uint32)
        assert 4 * first + buf.nbytes <= size
        torch.cuda.synchronize()
        assert self.rt.cudaMemcpy(ctypes.c_void_p(ptr + 4 * first), buf.ctypes.data_as(ctypes.c_void_p),
                                  ctypes.c_size_t(buf.nbytes), 1) == 0

    def read(self, name, count):
        buf = np.zeros(count, np.uint32)
        torch.cuda.synchronize()
        assert self.rt.cudaMemcpy(buf.ctypes.data_as(ctypes.c_void_p), ctypes.c_void_p(self.at[name][0]),
                                  ctypes.c_size_t(buf.nbytes), 2) == 0
        return buf


def continues_like_a_fresh_handle(sim, system, precision, start, **options):
    fresh = pkg.Simulation(system, precision=precision, **options)
    for s in (sim, fresh):
        s.set_state(start["x"], start["species"], start["ids"], None, start["next_id"], start["step"])
    for _ in range(6):
        sim.step()
        fresh.step()
        a, b = sim.get_state(), fresh.get_state()
        for key in ("ids", "species", "next_id", "x"):
            assert np.array_equal(a[key], b[key]), key
        assert np.array_equal(sim.observables()["counts"], fresh.observables()["counts"])
    assert fresh.observables()["stats"]["fired"] > 0
    fresh.close()


def membrane():
    return W.membrane_2d(n_each=600, L=0.6, dt=1e-4, equilibrium_start=True)


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("make", [dense_reversible, membrane])
def test_after_a_pair_list_overflow(make, precision):
    system = make()
    big = pkg.Simulation(system, precision=precision)
    big.step()
    fired = len(big.last_fired()["id_a"])
    big.close()
    sim = pkg.Simulation(system, precision=precision, pair_capacity=fired - 1)
    start = sim.get_state()
    sim.step()
    with pytest.raises(pkg.RDError):
        sim.sync()
    # the same handle, on a state with fewer pairs: half of the particles
    keep = np.flatnonzero(start["ids"] % 2 == 0)
    half = {"x": start["x"][keep], "species": start["species"][keep], "ids": start["ids"][keep],
            "next_id": start["next_id"], "step": 0}
    continues_like_a_fresh_handle(sim, system, precision, half)
    sim.close()


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("launch", ["fused", "separate"])
@pytest.mark.parametrize("make", [dense_reversible, membrane])
def test_after_a_step_that_left_its_lists_and_tallies(make, launch, precision, monkeypatch):
    system = make()
    allocs = []
    real = torch.cuda.caching_allocator_alloc

    def alloc(nbytes, device=None, stream=None):
        ptr = real(nbytes, device, stream)
        allocs.append((ptr, nbytes))
        return ptr

    monkeypatch.setattr(torch.cuda, "caching_allocator_alloc", alloc)
    sim = pkg.Simulation(system, precision=precision, step_launch=launch)
    monkeypatch.undo()
    start = sim.get_state()
    sim.run(2)
    sim.sync()
    n, cap, cells = len(start["ids"]), sim.info()["capacity"], sim.info()["cells"]
    mem = Memory(allocs)
    assert mem.read("ctl", 2).tolist() == [2, 0] and not mem.read("cell_count", cells).any()
    assert not mem.read("deg", cap).any()
    assert precision == "fp64" or (mem.read("best_key", 2 * cap) == 0xFFFFFFFF).all()
    w = mem.words
    for name in ("fired", "n_conflict", "n_decay", "n_accept", "n_round_acc", "n_ang", "n_ev", "done_blocks", "done_res",
                 "bar_count", "bar2_count"):
        mem.write("ctl", w[name], [3])
    mem.write("ctl", w["live"], [2, 2])
    mem.write("rep_cons", 0, [4])
    mem.write("rep_prod", 0, [2])
    mem.write("cell_count", 0, np.arange(cells) % 3)
    mem.write("deg", 0, np.arange(n) % 2)
    mem.write("best_key", 0, np.zeros(2 * n))
    mem.write("best_pid", 0, np.zeros(2 * n))
    mem.write("ctl", w["status"], [RD_ETIMEOUT])
    assert sim.get_state(allow_error=True)["status"] == RD_ETIMEOUT
    continues_like_a_fresh_handle(sim, system, precision, start, step_launch=launch)
    sim.close()
