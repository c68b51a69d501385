"""The pool of idle blocks (csrc/block_pool.h) on a runtime of two devices that only counts: a device's idle bytes are its
own, blocks are handed out on their device only, a failed allocation trims the device it was made on, blocks released since
the last synchronisation wait for one, the bounds hold, a small one with no object alive, and the last object empties the pool."""
import subprocess
from pathlib import Path

CSRC = Path(__file__).resolve().parents[1] / "paper_1810_06760_gb300" / "csrc"

PROGRAM = r'''
#include <cstdio>
#include <cstdlib>
#include <set>
#include "block_pool.h"

static int current = 0, syncs = 0, host_frees = 0;
static std::set<long> freed;
struct Rt {
    static int device() { return current; }
    static bool synchronize() { syncs++; return true; }
    static void free_device(void *p) { if (!freed.insert((long)p).second) std::abort(); }
    static void free_host(void *) { host_frees++; }
};
#define CHECK(c) do { if (!(c)) { std::printf("line %d: %s\n", __LINE__, #c); return 1; } } while (0)
static void *blk(long i) { return (void *)i; }

int main() {
    std::atomic<int64_t> used{0};
    const size_t MB = 1 << 20;
    fga::BlockPool<Rt> pool(100 * MB, 25 * MB, 10 * MB, used);
    pool.object(1);
    size_t got = 0;
    // two blocks on device 0, one on device 1
    used = 60 * MB;
    pool.put_device(blk(1), 10 * MB, 0);
    pool.put_device(blk(2), 20 * MB, 0);
    pool.put_device(blk(3), 30 * MB, 1);
    CHECK(used == 0 && pool.idle_bytes(0) == 30 * MB && pool.idle_bytes(1) == 30 * MB && pool.idle_bytes(2) == 0);
    // a fitting block of the other device is not taken; the own one is, after a synchronisation
    CHECK(!pool.take_device(0, 30 * MB, &got) && syncs == 0);
    CHECK(pool.take_device(0, 20 * MB, &got) == blk(2) && got == 20 * MB && syncs == 1 && used == (int64_t)(20 * MB));
    CHECK(pool.take_device(0, 10 * MB, &got) == blk(1) && syncs == 1);   // idle since the same synchronisation
    CHECK(pool.idle_bytes(0) == 0 && pool.idle_bytes(1) == 30 * MB);
    // nothing much larger than asked for
    pool.put_device(blk(2), 20 * MB, 0);
    CHECK(!pool.take_device(0, 10 * MB, &got));
    // a failed allocation on device 0 leaves device 1's blocks
    pool.trim_device(0);
    CHECK(freed == std::set<long>{2} && pool.idle_bytes(0) == 0 && pool.idle_bytes(1) == 30 * MB);
    current = 1;
    CHECK(pool.take_device(1, 29 * MB, &got) == blk(3) && got == 30 * MB && syncs == 2);
    // the bound holds over all devices, the largest go first; what exceeds it alone is freed
    pool.put_device(blk(3), 30 * MB, 1);
    pool.put_device(blk(4), 50 * MB, 0);
    pool.put_device(blk(5), 40 * MB, 1);
    CHECK(freed == (std::set<long>{2, 4}) && pool.idle_bytes(0) == 0 && pool.idle_bytes(1) == 70 * MB);
    pool.put_device(blk(6), 101 * MB, 1);
    CHECK(freed.count(6) && pool.idle_bytes(1) == 70 * MB);
    pool.trim(30 * MB);
    CHECK(freed.count(5) && !freed.count(3) && pool.idle_bytes(1) == 30 * MB);
    // host blocks: bounded
    pool.put_host(blk(7), 6 * MB, 1);
    pool.put_host(blk(8), 6 * MB, 1);
    CHECK(host_frees == 1);
    // on request everything goes, whatever is alive; the bytes in use do not change
    pool.put_device(blk(12), 5 * MB, 0);
    const int64_t before = used;
    pool.release();
    CHECK(freed.count(3) && freed.count(12) && host_frees == 2 && pool.idle_bytes(0) + pool.idle_bytes(1) == 0 && used == before);
    pool.put_device(blk(13), 30 * MB, 1);
    // the last object empties the pool
    pool.object(1);
    pool.object(-1);
    CHECK(!freed.count(13));
    pool.object(-1);
    CHECK(freed.count(13) && pool.idle_bytes(1) == 0);
    // with none alive a small bound holds
    pool.put_device(blk(9), 10 * MB, 0);
    pool.put_device(blk(10), 26 * MB, 0);
    CHECK(freed.count(10) && !freed.count(9) && pool.idle_bytes(0) == 10 * MB);
    pool.put_device(blk(11), 16 * MB, 1);
    CHECK(freed.count(9) && pool.idle_bytes(0) == 0 && pool.idle_bytes(1) == 16 * MB);
    std::printf("ok\n");
    return 0;
}
'''


def test_block_pool(tmp_path):
    src, exe = tmp_path / "pool.cpp", tmp_path / "pool"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-Wall", "-Werror", "-pthread", "-I", str(CSRC), str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout == "ok\n", r.stdout
