"""What ends up in an index file, and what is accepted as one, when file accesses fail: the GPU builder writes the
two large arrays of a regular file from several threads, the loader reads all four that way.  The failures are
made on the host, by a stand-in for pread, pwrite and operator new that a child process is started with."""
import os
import subprocess
import sys
import threading
from pathlib import Path

import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

pytest.importorskip("torch")

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# The access at file offset FAULT_OFFSET, if it is a large one, waits until the others are through and fails:
# a write with ENOSPC, a read as at the end of the file.  FAULT_OP = new<i>: the i-th request for exactly FAULT_OFFSET
# bytes is refused.
STAND_IN = r"""
#ifndef _GNU_SOURCE
#define _GNU_SOURCE
#endif
#include <atomic>
#include <new>
#include <dlfcn.h>
#include <errno.h>
#include <stdlib.h>
#include <string.h>
#include <sys/types.h>
#include <unistd.h>
static int hit(const char* op, size_t n, off_t off) {
    const char *w = getenv("FAULT_OP"), *o = getenv("FAULT_OFFSET");
    if (!w || strcmp(w, op) || n < 4096 || off != (off_t)atoll(o)) return 0;
    usleep(700000);
    return 1;
}
extern "C" ssize_t pwrite(int fd, const void* p, size_t n, off_t off) {
    auto real = (ssize_t (*)(int, const void*, size_t, off_t))dlsym(RTLD_NEXT, "pwrite");
    if (hit("write", n, off)) { errno = ENOSPC; return -1; }
    return real(fd, p, n, off);
}
extern "C" ssize_t pread(int fd, void* p, size_t n, off_t off) {
    auto real = (ssize_t (*)(int, void*, size_t, off_t))dlsym(RTLD_NEXT, "pread");
    return hit("read", n, off) ? 0 : real(fd, p, n, off);
}
extern "C" ssize_t __pread_chk(int fd, void* p, size_t n, off_t off, size_t) { return pread(fd, p, n, off); }
void* operator new(size_t n) {
    static std::atomic<int> seen{0};
    const char *w = getenv("FAULT_OP"), *o = getenv("FAULT_OFFSET");
    if (w && !strncmp(w, "new", 3) && n == (size_t)atoll(o) && ++seen == atoi(w + 3)) throw std::bad_alloc();
    void* p = malloc(n ? n : 1);
    if (!p) throw std::bad_alloc();
    return p;
}
void operator delete(void* p) noexcept { free(p); }
void operator delete(void* p, size_t) noexcept { free(p); }
"""

CHILD = r"""
import sys
import numpy as np
import paper_2608_16491_b200 as frog
do, data, path = sys.argv[1:]
try:
    if do == "build":
        x = np.load(data)
        frog.build_index_gpu(x["base"], x["attrs"], path, ef_c=16, n_inv=8)
    else:
        frog.Index.load(path)
    print("code 0")
except frog.FrogError as e:
    print("code %d" % e.code)
"""


@pytest.fixture(scope="module")
def files(libs, tmp_path_factory):
    """Vectors and attributes of an index whose arrays take several chunks of 2 MB, its file, the stand-in."""
    tmp = tmp_path_factory.mktemp("files")
    rng = np.random.default_rng(3)
    base = rng.standard_normal((20000, 96)).astype(np.float32)
    attrs = rng.integers(0, 5000, 20000).astype(np.int32)
    np.savez(tmp / "data.npz", base=base, attrs=attrs)
    good = str(tmp / "good.idx")
    libs.build_index_gpu(base, attrs, good, ef_c=16, n_inv=8)
    (tmp / "stand_in.cpp").write_text(STAND_IN)
    subprocess.check_call(["g++", "-shared", "-fPIC", "-O1", "-o", str(tmp / "stand_in.so"), str(tmp / "stand_in.cpp"), "-ldl"])
    return tmp, base, attrs, good


def _child(files, do, path, op=None, offset=0):
    env = dict(os.environ, PYTHONPATH=ROOT, LD_PRELOAD=str(files[0] / "stand_in.so"), FAULT_OFFSET=str(offset))
    if op:
        env["FAULT_OP"] = op
    out = subprocess.run([sys.executable, "-c", CHILD, do, str(files[0] / "data.npz"), path], env=env, cwd=ROOT,
                         stdout=subprocess.PIPE, text=True, timeout=300)
    return int(out.stdout.split("code ")[1]) if out.returncode == 0 else -1


def _offsets(path):
    return [int(x) for x in np.frombuffer(Path(path).read_bytes()[72:112], np.uint64)]   # attr, id, vec, enc, end


def test_a_build_that_fails_late_leaves_nothing_that_loads(libs, files):
    """The first chunk of the vectors fails after all others have been written."""
    tmp, good = files[0], files[3]
    path = str(tmp / "hole.idx")
    assert _child(files, "build", path) == 0
    assert Path(path).read_bytes() == Path(good).read_bytes()
    assert _child(files, "build", path, "write", _offsets(good)[2]) == 2
    with pytest.raises(libs.FrogError) as e:
        libs.Index.load(path)
    assert e.value.code == 3
    libs.build_index_gpu(files[1], files[2], path, ef_c=16, n_inv=8)
    assert Path(path).read_bytes() == Path(good).read_bytes()


@pytest.mark.parametrize("which", [1, 2, 3])
def test_a_build_without_host_memory_says_so(files, which):
    """Arrays of one integer per object: their order, the sorted attributes, the ranks."""
    assert _child(files, "build", str(files[0] / "none.idx"), "new%d" % which, 4 * 20000) == 4


@pytest.mark.parametrize("section", [0, 2, 3])
def test_a_file_that_ends_early_while_it_is_read(libs, files, section):
    assert _child(files, "load", files[3]) == 0
    assert _child(files, "load", files[3], "read", _offsets(files[3])[section]) == 2


def test_a_pipe_gets_the_same_bytes(libs, files):
    tmp, base, attrs, good = files
    fifo = str(tmp / "pipe")
    os.mkfifo(fifo)
    got = []
    reader = threading.Thread(target=lambda: got.append(Path(fifo).read_bytes()))
    reader.start()
    libs.build_index_gpu(base, attrs, fifo, ef_c=16, n_inv=8)
    reader.join()
    assert got[0] == Path(good).read_bytes()
