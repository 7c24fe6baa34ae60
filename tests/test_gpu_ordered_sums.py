"""GPU: the grouped block products on their own.  Ordered sums (what steers a Davidson run) are
one chain of fused multiply-adds per element, over the tasks and columns in table order with
alpha multiplied into A first: the lane kernel, the kernel in rounds, staged tiles and the
uploader's choice of them must all give the bits of that chain computed on the host.  Shared sums may round
differently: 1e-13 of sum |alpha A B| per element (lists of at most ~2,000 terms: 2e3 x 1.1e-16).

Blocks of one row or column up to several 32-lane slices, one to 300 tasks, inner sizes with
every remainder of four, transposes, identities, unit and other alphas, padded rows."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
ORDERED, SHARED, OVERWRITE, LANES, ROUNDS, TILES = 1, 2, 4, 8, 16, 32


@pytest.fixture(scope="module")
def hook():
    import torch
    assert torch.cuda.is_available()
    from paper_1312_2415_gb300 import binding
    return binding


def table(seed, shapes, alphas):
    """Blocks in one array: (tasks, alpha, groups, data, per group: slice of C and its terms)."""
    rng = np.random.default_rng(seed)
    data, tasks, alpha, groups = [], [], [], []
    size = 0

    def block(rows, cols):
        nonlocal size
        ld = cols + int(rng.integers(0, 3))
        data.append(rng.normal(size=rows * ld))
        size += rows * ld
        return size - rows * ld, ld
    for m, n, nt, kmax, *kmin in shapes:
        c, ldc = block(m, n)
        first = len(tasks)
        for _ in range(nt):
            k = int(rng.integers(*(kmin or [1]), kmax + 1))
            ta, tb = (int(v) for v in rng.integers(0, 2, 2))
            if rng.random() < 0.15:
                k, a, lda, ta = m, -1, 0, 0
            else:
                a, lda = block(*((k, m) if ta else (m, k)))
            b, ldb = block(*((n, k) if tb else (k, n)))
            tasks.append((a, b, lda, ldb, k, ta, tb))
            alpha.append(rng.choice(alphas))
        groups.append((c, ldc, m, n, first, len(tasks)))
    return np.array(tasks), np.array(alpha), np.array(groups), np.concatenate(data)


def host(tasks, alpha, groups, data, over):
    """The chain (fused multiply-adds of libm) and the magnitude of every element's sum."""
    libm = ctypes.CDLL("libm.so.6")
    fma = libm.fma
    fma.restype, fma.argtypes = ctypes.c_double, [ctypes.c_double] * 3
    out, mag = data.copy(), np.zeros_like(data)
    for c, ldc, m, n, t0, t1 in groups:
        if t0 == t1:
            continue
        for i in range(m):
            for j in range(n):
                acc, s = 0.0, 0.0
                for (a, b, lda, ldb, k, ta, tb), al in zip(tasks[t0:t1], alpha[t0:t1]):
                    if a < 0:
                        v = data[b + j * ldb + i] if tb else data[b + i * ldb + j]
                        acc = fma(al, v, acc)
                        s += abs(al * v)
                        continue
                    x = data[a + i + lda * np.arange(k)] if ta else data[a + i * lda:a + i * lda + k]
                    y = data[b + j * ldb:b + j * ldb + k] if tb else data[b + j + ldb * np.arange(k)]
                    x = x * al
                    s += np.abs(x * y).sum()
                    for u, v in zip(x.tolist(), y.tolist()):
                        acc = fma(u, v, acc)
                e = c + i * ldc + j
                out[e] = acc if over else data[e] + acc
                mag[e] = s + abs(data[e])
    return out, mag


EDGES = [(1, 1, 1, 9), (1, 1, 40, 3), (3, 5, 2, 7), (4, 8, 3, 8), (5, 7, 0, 1), (5, 7, 13, 6), (8, 4, 300, 4), (31, 1, 4, 5),
         (1, 33, 4, 5), (16, 2, 17, 3), (33, 3, 12, 4), (2, 65, 6, 9), (6, 11, 20, 11), (32, 32, 2, 6), (70, 3, 5, 33),
         (36, 20, 3, 12)]
SHORT = [(m, n, 1 + (m + n) % 3, 5) for m in (1, 2, 7, 9) for n in (1, 4, 31, 40)]
LONG = [(m, n, 12 + m + n, 5) for m in (1, 3, 8) for n in (2, 5, 13)]


@pytest.mark.parametrize("shapes", [EDGES, SHORT, LONG], ids=["edges", "short lists", "long lists"])
@pytest.mark.parametrize("alphas", [(1.0, -1.0), (0.37, -2.5, 1.0, -1.0, 0.0), (-0.81,)], ids=["unit", "mixed", "scaled"])
@pytest.mark.parametrize("over", [False, True])
def test_sums(hook, shapes, alphas, over):
    tab = table(len(shapes) + 7 * len(alphas), shapes, alphas)
    want, mag = host(*tab, over)
    flag = OVERWRITE if over else 0
    for kind in (ORDERED, ORDERED | LANES, ORDERED | ROUNDS, ORDERED | TILES, ORDERED | SHARED, ORDERED | SHARED | ROUNDS):
        got = hook.test_block_products(*tab, kind | flag, ORDERED)
        assert np.array_equal(got.view(np.int64), want.view(np.int64)), (kind, np.abs(got - want).max())
    for kind in (SHARED, ORDERED | SHARED, SHARED | TILES):
        got = hook.test_block_products(*tab, kind | flag, SHARED)
        assert (np.abs(got - want) <= 1e-13 * mag).all(), kind


def test_a_run_of_another_kind_is_an_error(hook):
    tab = table(1, SHORT[:4], (1.0,))
    for upload, run in ((ORDERED, SHARED), (SHARED, ORDERED)):
        with pytest.raises(hook.DMRGError) as e:
            hook.test_block_products(*tab, upload, run)
        assert e.value.code == hook.EINTERNAL


def test_large_blocks(hook):
    """Blocks that the uploader's rule gives to staged tiles (at least 160 rows and columns with
    little padding, enough of them), and blocks beside them that it gives to lanes (one row
    less, much padding, small)."""
    tab = table(3, [(192, 160, 2, 16, 15), (159, 160, 1, 3), (161, 161, 1, 4), (5, 7, 13, 6)], (0.37, -1.0))
    want, mag = host(*tab, False)
    for kind in (ORDERED, ORDERED | LANES, ORDERED | TILES, ORDERED | SHARED):
        got = hook.test_block_products(*tab, kind, ORDERED)
        assert np.array_equal(got.view(np.int64), want.view(np.int64)), (kind, np.abs(got - want).max())
    for kind in (SHARED, SHARED | TILES):
        assert (np.abs(hook.test_block_products(*tab, kind, SHARED) - want) <= 1e-13 * mag).all(), kind
    # the first group 200 times over (6,000 tiles): the rule's own choice, on copies of its C
    tasks, alpha, groups, data = tab
    c, ldc, m, n, t0, t1 = groups[0]
    copies = 200
    many = np.array([(data.size + i * m * ldc, ldc, m, n, t0, t1) for i in range(copies)] + groups[1:].tolist())
    block = data[c:c + m * ldc]
    wide = np.concatenate([data] + [block] * copies)
    for kind, run in ((ORDERED | SHARED, ORDERED), (SHARED, SHARED), (ORDERED | LANES, ORDERED)):
        got = hook.test_block_products(tasks, alpha, many, wide, kind, run)
        for i in range(copies):  # ordered in either kind where the rule takes tiles
            part = got[data.size + i * m * ldc:][:m * ldc]
            assert np.array_equal(part.view(np.int64), want[c:c + m * ldc].view(np.int64)), (kind, i)
        rest = np.r_[got[:c], got[c + m * ldc:data.size]]
        assert (np.abs(rest - np.r_[want[:c], want[c + m * ldc:]]) <= 1e-13 * np.r_[mag[:c], mag[c + m * ldc:]]).all()


def test_rounds_without_room_for_their_table(hook):
    """Under a device-memory cap that the lanes' tables fit under and the rounds' chunks do not,
    the uploader takes lanes: nothing that fits is refused, and the bits are the same."""
    tab = table(5, [(4, 8, 60, 64, 40)] * 3, (0.37, 1.0))
    used = hook.device_memory_in_use()
    want = hook.test_block_products(*tab, ORDERED, ORDERED)

    def run(kind, cap):
        hook.set_device_memory_cap(cap)
        try:
            return hook.test_block_products(*tab, kind, ORDERED)
        except hook.DMRGError as e:
            assert e.code == hook.ENOMEM and hook.device_memory_in_use() == used
            return None
        finally:
            hook.set_device_memory_cap(0)
    between = 0
    for room in range(0, 64 * 1024, 512):
        cap = used + 8 * tab[3].size + room
        rule, lanes, rounds = run(ORDERED, cap), run(ORDERED | LANES, cap), run(ORDERED | ROUNDS, cap)
        assert (rule is None) == (lanes is None)
        between += lanes is not None and rounds is None
        for got in (rule, lanes, rounds):
            assert got is None or np.array_equal(got.view(np.int64), want.view(np.int64))
    assert between > 0 and rule is not None and rounds is not None
