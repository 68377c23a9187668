"""The waits of the SSD run kernel (csrc/k2_run.cu), restated: copy warp, product warp and two compute warps as
programs over mbarriers, run in random order with every copy and product completing as late or as early as it
likes (products and tensor-memory copies in the order of issue where PTX promises that).  A wait names the phase it means; the hardware compares one parity bit, so a barrier that has gone
more than one phase past it would be waited for until the limit.  Everything in flight holds the memory it reads
and writes: nobody may touch that before a wait has seen it complete.

A change to the kernel's waits is made here too: what this shows is the order of the waits as restated, not the
compiled kernel."""
import random

import pytest

X_SLOTS = Y_BARS = 3
WARPS = 2                      # compute warps (16 there): enough for one to run ahead of the other


def copy_warp(nt, n_pre):
    def load_x(j):
        yield "copy", ("x_full", j % X_SLOTS), (), (("x", j % X_SLOTS),)

    def load_rec(j):
        yield "copy", ("x_full", j % X_SLOTS), (), (("rec",),)

    def load_b(j):
        yield "wait", ("b_empty", j & 1), (j >> 1) - 1
        yield "copy", ("b_full", j & 1), (), (("b", j & 1),)

    def load_c(j):
        yield "wait", ("c_empty",), j - n_pre - 1
        yield "copy", ("c_full",), (), (("c",),)

    def store_y(j):
        jf = j - n_pre
        yield "wait", ("y_staged", jf % Y_BARS), jf // Y_BARS
        yield "copy", None, (("x", j % X_SLOTS),), ()

    for j in range(min(X_SLOTS, nt)):
        yield from load_x(j)
    yield from load_rec(0)
    yield from load_b(0)
    if n_pre == 0:
        yield from load_c(0)
    if nt > 1:
        yield from load_b(1)
        yield "wait", ("rec_free",), 0
        yield from load_rec(1)
    for j in range(nt):
        if j + 1 < nt and j + 1 >= n_pre:
            yield from load_c(j + 1)
        if j > n_pre:
            yield from store_y(j - 1)
        if j + 2 < nt:
            yield from load_b(j + 2)
        if j > 0 and j - 1 + X_SLOTS < nt:
            yield ("drain",)                                   # bulk_wait_read_all
            yield from load_x(j - 1 + X_SLOTS)
        if j + 2 < nt:
            yield "wait", ("rec_free",), j + 1
            yield from load_rec(j + 2)
    if nt > n_pre:
        yield from store_y(nt - 1)


def product_warp(nt, n_pre):
    def copy_c(j):
        yield "wait", ("c_full",), j - n_pre
        yield "tc", "cp", None, (("c",),), ("C",)
        yield "commit", ("c_empty",)

    def issue_g(j):
        yield "wait", ("b_full", j & 1), j >> 1
        yield "tc", "mma", ("G", 128), (("b", j & 1), "C"), ("G",)
        yield "commit", ("g_full",)

    if n_pre == 0:
        yield from copy_c(0)
        yield from issue_g(0)
    for j in range(nt):
        full, jf = j >= n_pre, j - n_pre
        if not full:
            yield "wait", ("b_full", j & 1), j >> 1
        yield "wait", ("xp_full", j & 1), j >> 1
        yield "tc", "mma", ("DH", 128), (("b", j & 1), "Y" if not full and j & 1 else "XP"), ("DH",)
        if j == n_pre - 1:
            yield "commit", ("dh_full",)
        if not full:
            yield "commit", ("xp_free", j & 1)
        yield "commit", ("b_empty", j & 1)
        if full:
            if jf > 0:
                yield "wait", ("y_staged", (jf - 1) % Y_BARS), (jf - 1) // Y_BARS
            yield "tc", "mma", ("Y", 128), ("C", ("h",)), ("Y",)
            yield "commit", ("dh_full",)
            yield "wait", ("dh_full",), jf + (n_pre > 0)
            if j + 1 < nt:
                yield from copy_c(j + 1)
            yield "wait", ("m_full",), jf
            yield "tc", "mma", ("Y", 64), ("G", ("x", j % X_SLOTS)), ("Y",)
            yield "commit", ("yd_full",)
            if j + 1 < nt:
                yield "wait", ("yd_full",), jf
        if j + 1 < nt and j + 1 >= n_pre:
            if not full:
                yield from copy_c(j + 1)
            yield from issue_g(j + 1)


def compute_warp(nt, n_pre, scale):
    def take_rec():
        yield "touch", (("rec",),), ()
        yield "arrive", ("rec_free",)

    def scale_x(j):
        lead = j < n_pre
        if lead and j > 1:
            yield "wait", ("xp_free", j & 1), (j >> 1) - 1
        yield "touch", (("x", j % X_SLOTS),), ("Y" if lead and j & 1 else "XP",)
        yield "arrive", ("xp_full", j & 1)

    yield "wait", ("x_full", 0), 0
    if n_pre == 0:
        yield "touch", (), (("h",),)
    yield from take_rec()
    yield from scale_x(0)
    for j in range(nt):
        full, jf = j >= n_pre, j - n_pre
        dh = jf + (1 if n_pre > 0 else 0) if full else 0
        if full:
            yield "wait", ("g_full",), jf
            yield "touch", ("G",), ("G",)
            if scale:
                yield "wait", ("dh_full",), dh
                yield "touch", ("Y",), ("Y",)
            yield "arrive", ("m_full",)
        if j + 1 < nt:
            yield "wait", ("x_full", (j + 1) % X_SLOTS), (j + 1) // X_SLOTS
        if full or j == n_pre - 1:
            yield "wait", ("dh_full",), dh
            yield "touch", ("DH",), (("h",),) if j + 1 < nt else ()
        if j + 1 < nt:
            yield from take_rec()
            yield from scale_x(j + 1)
        if full:
            yield "wait", ("yd_full",), jf
            yield "touch", ("Y", ("x", j % X_SLOTS)), (("x", j % X_SLOTS),)
            yield "arrive", ("y_staged", jf % Y_BARS)


NEEDED = {"x_full": 2, "rec_free": WARPS, "xp_full": WARPS, "m_full": WARPS, "y_staged": WARPS}   # arrivals a phase


def clash(a_reads, a_writes, b_reads, b_writes):
    return bool(set(a_writes) & (set(b_reads) | set(b_writes)) or set(a_reads) & set(b_writes))


def in_order(before, op):
    """Whether two tensor-core operations of one thread are promised to run in the order of issue."""
    return op[1] == "mma" and (before[1] == "cp" or before[2] == op[2])


def simulate(nt, n_pre, rng):
    agents = [copy_warp(nt, n_pre), product_warp(nt, n_pre)]
    agents += [compute_warp(nt, n_pre, scale) for scale in (rng.random() < 0.3,) for _ in range(WARPS)]
    todo = [next(a) for a in agents]
    phases, arrived = {}, {}
    copies, queue = [], []     # in flight: copies complete in any order, products and commits in theirs

    def arrive(bar):
        arrived[bar] = arrived.get(bar, 0) + 1
        if arrived[bar] == NEEDED.get(bar[0], 1):
            arrived[bar], phases[bar] = 0, phases.get(bar, 0) + 1

    def free(who, reads, writes, ordered=lambda op: False):
        for op in copies:
            assert not clash(reads, writes, op[2], op[3]), f"{who}: {op} is in flight"
        for op in queue:
            if op[0] == "tc" and not ordered(op):
                assert not clash(reads, writes, op[3], op[4]), f"{who}: {op} is in flight"

    def blocked(op):
        if op[0] == "wait":
            done = phases.get(op[1], 0)
            assert done <= op[2] + 1, f"{op[1]}: phase {op[2]} is waited for when {done} have completed"
            return done <= op[2]
        return op[0] == "drain" and any(c[1] is None for c in copies)

    def step(i):
        op = todo[i]
        if op[0] == "touch":
            free(op, op[1], op[2])
        elif op[0] == "arrive":
            arrive(op[1])
        elif op[0] == "copy":
            free(op, op[2], op[3])
            copies.append(op)
        elif op[0] == "tc":
            free(op, op[3], op[4], lambda before: in_order(before, op))
            queue.append(op)
        elif op[0] == "commit":
            queue.append(op)
        todo[i] = next(agents[i], None)

    while any(t is not None for t in todo):
        moves = [i for i, t in enumerate(todo) if t is not None and not blocked(t)]
        if copies:
            moves.append("copy")
        if queue:
            moves.append("queue")
        assert moves, f"nobody can go on: {todo}"
        move = rng.choice(moves)
        if move == "copy":
            done = copies.pop(rng.randrange(len(copies)))
            if done[1] is not None:
                arrive(done[1])
        elif move == "queue":
            done = queue.pop(0)
            if done[0] == "commit":
                arrive(done[1])
        else:                  # one agent runs ahead for a while
            for _ in range(rng.choice([1, 1, 3, 10])):
                if todo[move] is None or blocked(todo[move]):
                    break
                step(move)


@pytest.mark.parametrize("nt,n_pre", [(1, 0), (2, 0), (3, 0), (6, 0), (9, 0), (6, 1), (6, 2), (7, 3), (9, 5), (10, 9)])
def test_waits_of_the_run_kernel(nt, n_pre):
    rng = random.Random(100 * nt + n_pre)
    for _ in range(400):
        simulate(nt, n_pre, rng)
