"""The host rules that choose a launch shape, called in the built library (no
GPU): a small program is compiled against the engine's header."""
import os
import subprocess

import pytest

from paper_1006_0252_gb300 import build

# Prints, for a class given as (kind, size, alone, R0 ...): threads a block,
# threads a replica, replicas a thread, shared memory asked for, slots of an item.
PROGRAM = r"""
#include "pa_engine.h"
int main(int n, char** a) {
  LatticeClass c;
  const std::string kind = a[1];
  if (kind == "resample") {
    printf("%lld 0 0 0 0\n", (long long)boot_resample(strtoul(a[2], 0, 10), 128, atoi(a[3]), 8));
    return 0;
  }
  c.model = kind[0] == 'g';
  c.dim = kind.back() == 'c' ? 1 : 3;
  c.L = atoi(a[2]);
  c.sms = atoi(getenv("SMS"));
  c.capacity = atoll(getenv("CAPACITY"));
  c.Wr = (c.L + 31) / 32;
  c.W = (c.Wr + 3) / 4 * 4;
  std::vector<int64_t> R0;
  for (int i = 4; i < n; ++i) R0.push_back(atoll(a[i]));
  set_default_launch(c, 0, 0, R0);
  spread_blocks(c, R0, atoi(a[3]) != 0);
  printf("%d %d %d %d %d\n", c.tpb, c.split, c.rp, c.min_smem, c.item);
}
"""
SM_SMEM, BLOCK_RESERVED, NUM_SMS = 228 * 1024, 1024, 152


@pytest.fixture(scope="module")
def shape(tmp_path_factory):
    lib = build.build_library()
    d = tmp_path_factory.mktemp("shape")
    src, exe = d / "shape.cu", d / "shape"
    src.write_text(PROGRAM)
    where = os.path.dirname(lib)
    p = subprocess.run([build.nvcc(), *build.ARCH, "-std=c++17", "--expt-relaxed-constexpr", "-I", build.CSRC, "-I",
                        build.INCLUDE, str(src), "-o", str(exe), "-L", where, "-l:" + os.path.basename(lib), "-Xlinker",
                        "-rpath=" + where], capture_output=True, text=True)
    assert p.returncode == 0, p.stderr

    def call(kind, size, *R0, alone=True, sms=NUM_SMS, capacity=0):
        out = subprocess.run([str(exe), kind, str(size), str(int(alone)), *map(str, R0)], capture_output=True, text=True,
                             env={**os.environ, "SMS": str(sms), "CAPACITY": str(capacity)})
        assert out.returncode == 0, out.stderr
        return dict(zip(("tpb", "split", "rp", "min_smem", "item"), map(int, out.stdout.split())))

    return call


# (kind, size): pm / gpm cubic, c / gc chains.
SPREAD = [("pm", 4), ("pm", 6), ("pm", 8), ("pm", 10), ("pm", 12), ("pm", 14), ("pm", 16), ("c", 256), ("c", 4096),
          ("gc", 256)]


@pytest.mark.parametrize("sms", [132, 148, 152])
def test_rules_follow_the_number_of_multiprocessors(shape, sms):
    """As many replicas as fill sms blocks: one an SM, nothing to even out, on a
    device that has that many; work items of the threshold tables fill one round."""
    R0 = 16 * sms - 150
    assert shape("pm", 8, R0, sms=sms)["min_smem"] == 0
    assert shape("pm", 8, 2 * R0, sms=sms)["min_smem"] > 0
    for R0 in range(900, 3000, 100):
        item = shape("gpm", 8, R0, sms=sms)["item"]
        assert -(-R0 // item) <= sms and (item <= 4 or -(-(R0 + 3 * R0 ** 0.5 + 1) // (item - 4)) > sms), (R0, item)


def _blocks(sh, R0):
    per = sh["tpb"] // sh["split"] * sh["rp"]
    return -(-(R0 + int(3 * R0 ** 0.5)) // per)


@pytest.mark.parametrize("kind,size", SPREAD)
def test_no_shared_memory_is_held_where_it_evens_nothing(shape, kind, size):
    """At most one block an SM, or blocks that leave a tenth of their places
    free: nothing that would keep the blocks of other handles out."""
    for R0 in (100, 300, 1000, 1500, 2000, 2300, 3400, 5600, 8000, 16000):
        sh = shape(kind, size, R0)
        blocks = _blocks(sh, R0)
        most = -(-blocks // NUM_SMS)
        if most == 1 or blocks < 0.9 * most * NUM_SMS:
            assert sh["min_smem"] == 0, (R0, sh)


@pytest.mark.parametrize("kind,size", SPREAD)
def test_shared_memory_keeps_one_block_more_out(shape, kind, size):
    for R0 in range(3000, 16000, 700):
        sh = shape(kind, size, R0)
        blocks = _blocks(sh, R0)
        most = -(-blocks // NUM_SMS)
        if most > 1 and blocks >= 0.9 * most * NUM_SMS:
            held = sh["min_smem"] + BLOCK_RESERVED
            assert most * held <= SM_SMEM < (most + 1) * held, (R0, sh)
        # a capacity far above the population: from 0.7 of the places on
        if blocks >= 0.7 * most * NUM_SMS:
            held = shape(kind, size, R0, capacity=200 * R0)["min_smem"] + BLOCK_RESERVED
            assert most * held <= SM_SMEM < (most + 1) * held, (R0, sh)
        # classes of one step share the SMs
        assert shape(kind, size, R0, alone=False, capacity=200 * R0)["min_smem"] == 0


# Eight threads a resample, so a block of 128 threads takes 16: the thread's
# number in the grid passes 2^32 from 2^29 resamples on.
@pytest.mark.parametrize("block", [0, (1 << 25) - 1, 1 << 25, (1 << 27) - 1])
def test_bootstrap_resample_of_a_thread(shape, block):
    for thread in (0, 1):
        assert shape("resample", block, alone=thread)["tpb"] == 16 * block


# Chains: the words' places of the split that a large population gets are within a
# quarter of the words (the finest split of 9 words has 16).
@pytest.mark.parametrize("kind", ["c", "gc"])
def test_chain_splits_leave_few_places_idle(shape, kind):
    for words in range(5, 60):
        sh = shape(kind, 32 * words, 300000)
        places = -(-words // sh["split"]) * sh["split"]
        assert places <= 1.25 * words, (words, sh)


# Several runs: the blocks of their unused capacity lie between the others.
def test_unused_capacity_between_runs_is_spread(shape):
    sh = shape("pm", 16, *[500] * 7, capacity=7 * 794)
    assert 2 * (sh["min_smem"] + BLOCK_RESERVED) <= SM_SMEM < 3 * (sh["min_smem"] + BLOCK_RESERVED)
    assert shape("pm", 16, 3500, capacity=4156)["min_smem"] == 0
