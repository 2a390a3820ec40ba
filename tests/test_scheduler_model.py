"""The protocol of the one-launch brick scheduler as a host model
(tests/host/scheduler_model.cpp: warps take turns at random, one atomic
operation a turn) with the ring sizes and the claims of csrc/fmm_ring.h: it must always
end, with every chunk of a scan taken once."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SEEDS = 20


@pytest.fixture(scope="module")
def model(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("model") / "scheduler_model")
    subprocess.run(["g++", "-O2", "-std=c++17", "-Wall", "-I",
                    os.path.join(ROOT, "paper_1502_07303_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "host", "scheduler_model.cpp"), "-o", exe], check=True)

    def run(bricks, waiting, warps, levels=40, release=1, slots=0, any_raise=0, keep=0):
        args = (bricks, waiting, warps, levels, release, SEEDS, slots, any_raise, keep)
        r = subprocess.run([exe, *map(str, args)], capture_output=True, text=True, timeout=300)
        return r.returncode, r.stdout
    return run


# bricks, bricks that wait, warps: chunks of a scan of one and of many warp
# loads, half of the bricks waiting and all of them
GRIDS = [(1, 1, 4), (33, 33, 4), (64, 64, 4), (512, 400, 4), (512, 512, 4), (1000, 800, 12),
         (4096, 2600, 32), (4096, 4096, 32)]


@pytest.mark.parametrize("bricks,waiting,warps", GRIDS)
def test_appends_never_wait_for_the_scan(model, bricks, waiting, warps):
    rc, out = model(bricks, waiting, warps)
    assert rc == 0, out


def test_one_slot_per_brick_would_stall(model):
    """The model does find a ring that is too small."""
    rc, out = model(512, 512, 4, slots=512)
    assert rc == 2, out


# (few bricks wait at first: scans of one to a few chunks, and more of them later)
@pytest.mark.parametrize("bricks,waiting,warps", [(300, 20, 16), (1000, 20, 32), (4000, 40, 64)])
def test_late_claims_take_no_chunk(model, bricks, waiting, warps):
    rc, out = model(bricks, waiting, warps)
    assert rc == 0, out


def test_claims_of_any_raise_would_take_chunks_twice(model):
    """The model does find a claim that is taken for a later scan's."""
    rc, out = model(1000, 20, 32, any_raise=1)
    assert rc == 3 and "twice" in out, out


@pytest.mark.parametrize("bricks,waiting,warps", GRIDS)
@pytest.mark.parametrize("levels,release", [(1, 100), (3, 2)])
def test_raises_that_queue_every_brick(model, bricks, waiting, warps, levels, release):
    """Scanning warps hold queue tickets while the queue fills."""
    rc, out = model(bricks, waiting, warps, levels=levels, release=release)
    assert rc == 0, out


def test_a_kept_ticket_entry_would_stall(model):
    """The model does find a warp that waits for a slot only it can empty."""
    rc, out = model(512, 512, 4, levels=1, release=100, keep=1)
    assert rc == 2, out
