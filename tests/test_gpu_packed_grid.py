"""The memory of the packed grid that single-scenario runs in a cloud-in-cell field take from the
electron species' allocator: which blocks they accept and when they take one."""
import ctypes as C

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1311_5551_gb300 import build as qbuild  # noqa: E402
from paper_1311_5551_gb300 import qed  # noqa: E402

N, ORG, SPC = (13, 11, 9), (-20.0, 5.0, 100.0), (3.0e4, 2.5e4, 4.0e4)


@pytest.fixture(scope="module")
def tables():
    qbuild.build()
    return qed.Tables()


class Pool:
    """A qed_allocator over torch's: blocks start `shift` bytes after a 256-byte boundary; after `blocks`
    of them it refuses."""

    def __init__(self, shift=0, blocks=1 << 30):
        self.shift, self.live, self.log, self.freed, self.refused = shift, {}, [], [], 0

        @C.CFUNCTYPE(C.c_void_p, C.c_size_t, C.c_void_p, C.c_void_p)
        def alloc(nbytes, stream, user):
            if len(self.log) >= blocks:
                self.refused += 1
                return None
            t = torch.empty(int(nbytes) + 512, dtype=torch.uint8, device="cuda")
            ptr = ((t.data_ptr() + 255) & ~255) + self.shift
            self.live[ptr] = t
            self.log.append((int(nbytes), int(stream or 0)))
            return ptr

        @C.CFUNCTYPE(None, C.c_void_p, C.c_size_t, C.c_void_p, C.c_void_p)
        def free(ptr, nbytes, stream, user):
            del self.live[int(ptr)]
            self.freed.append((int(nbytes), int(stream or 0)))

        self._keep = (alloc, free)
        self.allocator = qed.Allocator(alloc, free, None)


def grid(n, seed):
    rng = np.random.default_rng(seed)
    return torch.tensor(rng.normal(size=(6, n[2], n[1], n[0])) * 1e-3, dtype=torch.float32, device="cuda")


def field(g):
    return qed.Field(kind=qed.FIELD_GRID, grid=g, shape=1, origin=ORG, spacing=SPC)


def fresh(n, seed, allocator=None):
    rng = np.random.default_rng(seed)
    x = np.stack([rng.uniform(ORG[a] - 3 * SPC[a], ORG[a] + (N[a] + 2) * SPC[a], n) for a in range(3)], axis=1)
    u = rng.normal(size=(n, 3)) * 300.0
    sp = [qed.Species(qed.ELECTRON, qed.MIXED, 4 * n + 64, 4 * n + 64, allocator=allocator),
          qed.Species(qed.POSITRON, qed.MIXED, 4 * n + 64, 4 * n + 64, allocator=allocator),
          qed.Species(qed.PHOTON, qed.MIXED, 30 * n + 64, 8 * n + 64, allocator=allocator)]
    sp[0].upload(x, u)
    sp[0].init_tau(seed)
    sp[2].upload(rng.permutation(x), rng.normal(size=(n, 3)) * 10.0 ** rng.uniform(-1, 4, (n, 1)))
    sp[2].init_tau(seed)
    return sp


def params(g):
    return qed.StepParams(dt=2.0e3, seed=2, field=field(g))


@pytest.mark.parametrize("shift", [16, 48, 240])
def test_blocks_aligned_to_16_bytes(tables, shift):
    # an allocator promises no more than the 16 bytes that the tile copies need
    g = grid(N, 1)
    out = []
    for pool in (None, Pool(shift)):
        sp = fresh(3001, 5, pool.allocator if pool else None)
        qed.run(tables, sp, params(g), 0, 5)
        qed.check(sp)
        out.append([s.save() for s in sp])
    assert all(np.array_equal(a, b) for a, b in zip(*out))
    assert len(pool.log) == 4  # three species and the packed grid


@pytest.mark.parametrize("shape", [1, 2])
@pytest.mark.parametrize("steps", [1, 3])
def test_grid_updated_between_calls(tables, shape, steps):
    # the loop of a PIC code: the caller's kernels rewrite one grid in place between calls; the same
    # particles as with every call's fields in a tensor of their own
    out = []
    for in_place in (False, True):
        sp = fresh(3001, 6)
        g = grid(N, 9)
        keep = []
        for k in range(12):
            p = params(g)
            p.field.shape = shape
            qed.run(tables, sp, p, k * steps, steps)
            keep.append(g)
            if in_place:
                g.mul_(-0.75)
            else:
                g = g * -0.75
        qed.check(sp)
        out.append([s.save() for s in sp])
    assert all(np.array_equal(a, b) for a, b in zip(*out))


def test_packed_grid_is_released_on_the_species_stream(tables):
    # a run may use a stream that is destroyed before the species: the room it took for the packed grid
    # is given back on the stream the species was created on
    pool = Pool()
    sp = fresh(3001, 7, pool.allocator)
    home = torch.cuda.current_stream().cuda_stream
    other = torch.cuda.Stream()
    g = grid(N, 1)
    torch.cuda.synchronize()
    qed.run(tables, sp, params(g), 0, 2, stream=other)
    other.synchronize()
    nbytes, stream = pool.log[3]
    assert stream == other.cuda_stream != home
    del other
    for s in sp:
        s.close()
    assert not pool.live and (nbytes, home) in pool.freed
    assert all(s == home for _, s in pool.freed)


def test_refused_packed_grid_is_no_error(tables):
    # an allocator that gives no room for the packed grid: the run gathers from the grid itself, with the
    # same particles, and the thread's last error message stays what it was
    g = grid(N, 1)
    out = []
    for pool in (Pool(), Pool(blocks=3)):
        sp = fresh(3001, 8, pool.allocator)
        with pytest.raises(qed.QedError):
            qed.Species(7, qed.MIXED, 10, 10)
        message = qed.lib().qed_last_error()
        qed.run(tables, sp, params(g), 0, 5)
        assert qed.lib().qed_last_error() == message
        qed.check(sp)
        out.append([s.save() for s in sp])
    assert pool.refused >= 1
    assert all(np.array_equal(a, b) for a, b in zip(*out))


def test_refusing_allocator_is_asked_once(tables):
    pool = Pool(blocks=3)
    sp = fresh(3001, 9, pool.allocator)
    g = grid(N, 1)
    for k in range(6):
        qed.run(tables, sp, params(g), k, 1)
    qed.check(sp)
    assert pool.refused == 1
    big = qed.StepParams(dt=2.0e3, seed=2, field=field(grid((20, 20, 20), 1)))
    qed.run(tables, sp, big, 6, 1)
    assert pool.refused == 1  # no more than was refused before
    small = qed.StepParams(dt=2.0e3, seed=2, field=field(grid((4, 4, 4), 1)))
    qed.run(tables, sp, small, 7, 1)
    assert pool.refused == 2


def test_no_room_is_taken_where_packing_cannot_pay(tables):
    # packing pays from a third of a particle-step per cell on: species that cannot hold as many take no
    # room in a one-step call, and do in a longer one
    g = grid((40, 40, 40), 1)
    cap = 2000
    for steps, blocks in ((1, 3), (3, 3), (4, 4)):  # 41^3 / 3 cells against 3 x 2000 particles a step
        pool = Pool()
        sp = [qed.Species(k, qed.MIXED, cap, 100, allocator=pool.allocator)
              for k in (qed.ELECTRON, qed.POSITRON, qed.PHOTON)]
        rng = np.random.default_rng(1)
        sp[0].upload(rng.uniform(0, 1e6, (50, 3)), rng.normal(size=(50, 3)) * 10)
        sp[0].init_tau(1)
        qed.run(tables, sp, params(g), 0, steps)
        qed.check(sp)
        assert len(pool.log) == blocks, (steps, pool.log)
