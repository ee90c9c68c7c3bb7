"""The codebook builder takes package-merge's lengths where no other code costs as little, else those of its dynamic programme, which
goes on from its least-cost states only; the lengths must be those of the programme over all states, ties included (a blob's
bytes depend on them).  CPU only."""
import numpy as np
import pytest

INF = 1 << 62


def lengths_over_all_states(counts, cap):
    """State = (symbols placed, most frequent first; budget spent in units of 2^-cap).  Among equal costs the shortest last
    length, at the end the least budget."""
    used = sorted((s for s in range(len(counts)) if counts[s]), key=lambda s: -counts[s])
    out = [0] * len(counts)
    if len(used) == 1:
        out[used[0]] = 1
        return out
    U = 1 << cap
    if U < len(used):
        return None
    cost, choice = [0] + [INF] * U, []
    for s in used:
        to, pick = [INF] * (U + 1), [0] * (U + 1)
        for b in range(U + 1):
            for l in range(1, cap + 1) if cost[b] < INF else ():
                nb = b + (U >> l)
                if nb <= U and cost[b] + counts[s] * l < to[nb]:
                    to[nb], pick[nb] = cost[b] + counts[s] * l, l
        cost = to
        choice.append(pick)
    b = cost.index(min(cost))
    for s, pick in zip(reversed(used), reversed(choice)):
        out[s] = pick[b]
        b -= U >> pick[b]
    return out


def draw(kind, n, rng):
    if kind == "equal":
        return [7] * n
    if kind == "few values":
        return [int(v) for v in rng.integers(0, 4, n)]
    if kind == "few symbols":
        return [int(v) if rng.random() < 0.2 else 0 for v in rng.integers(1, 1000, n)]
    if kind == "powers of two":                              # sums that equal other counts: ties between symbols and pairs
        return [1 << int(v) for v in rng.integers(0, 9, n)]
    if kind == "fibonacci":                                  # every length there is, equal costs of different codes
        f = [1, 1]
        while len(f) < n:
            f.append(f[-1] + f[-2] if len(f) < 40 else 1)
        return [f[i] for i in rng.permutation(n)]
    if kind == "beyond 2^40":                                # (left to the programme)
        return [int(v) for v in rng.integers(1, 1 << 41, n)]
    if kind == "halving":
        return [int(1e8 * 0.5 ** abs(i - 11)) for i in range(n)]
    return [int(2.0 ** v) for v in rng.uniform(0, 30, n)]


KINDS = ["equal", "few values", "few symbols", "halving", "wide", "powers of two", "fibonacci", "beyond 2^40"]


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("limit", [7, 8, 9])
def test_fp16_field_lengths(kind, limit):
    import paper_2502_00922_b200 as hl
    rng = np.random.default_rng(limit)
    fields = [draw(kind, 32, rng) for _ in range(3)]
    for f in fields:
        f[5] += 1                                            # (an empty field has no code)
    cb = hl.build_codebook_from_counts(np.array(sum(fields, []), dtype=np.uint64), hl.FP16, limit)
    for i, f in enumerate(fields):
        assert list(cb.get(i)[2][:32]) == lengths_over_all_states(f, limit)
    cb.free()


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("budget", [8, 9, 12])
def test_bf16_nibble_lengths_over_every_split_of_the_budget(kind, budget):
    import paper_2502_00922_b200 as hl
    counts = draw(kind, 256, np.random.default_rng(budget))
    counts[121] += 1
    hi = [sum(counts[16 * h:16 * h + 16]) for h in range(16)]
    lo = [sum(counts[l::16]) for l in range(16)]
    best = None
    for c0 in range(1, budget):                              # least cost, ties to the smaller cap of the upper nibble
        a, b = lengths_over_all_states(hi, c0), lengths_over_all_states(lo, budget - c0)
        if a and b:
            cost = sum(x * y for x, y in zip(hi, a)) + sum(x * y for x, y in zip(lo, b))
            if best is None or cost < best[0]:
                best = (cost, a, b)
    cb = hl.build_codebook_from_counts(np.array(counts, dtype=np.uint64), hl.BF16, budget)
    assert list(cb.get(0)[2][:16]) == best[1] and list(cb.get(1)[2][:16]) == best[2]
    cb.free()

STACK_PROGRAM = r"""
#include <pthread.h>
#include <cstdio>
#include <vector>
#include "huffllm.h"
static int failures = 0;
static void *work(void *) {
    static uint64_t counts[256];
    for (int i = 0; i < 256; ++i) counts[i] = 1000003ull * (i + 1) * (i % 7 + 1);
    for (uint32_t limit = 8; limit <= 12; ++limit)
        for (int kind = 0; kind < 3; ++kind) {
            huffllm_codebook *cb = nullptr;
            const huffllm_status st = huffllm_build_codebook_from_counts(counts, kind == 2 ? HUFFLLM_FP16 : HUFFLLM_BF16,
                                                                         kind == 1 ? HUFFLLM_SPLIT_WHOLE_EXPONENT : HUFFLLM_SPLIT_PAPER, limit, &cb);
            if (st != HUFFLLM_OK) ++failures;
            huffllm_codebook_free(cb);
        }
    return nullptr;
}
int main() {
    pthread_attr_t a;
    pthread_t t;
    if (pthread_attr_init(&a) || pthread_attr_setstacksize(&a, 64 << 10) || pthread_create(&t, &a, work, nullptr)) return 2;
    pthread_join(t, nullptr);
    printf("%d", failures);
    return 0;
}
"""


def test_codebooks_on_a_thread_with_a_small_stack(tmp_path):
    """Every kind of codebook from counts, longest lists included, on a thread with 64 KB of stack."""
    import os
    import subprocess
    import paper_2502_00922_b200.binding as binding
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    so = binding._SO
    (tmp_path / "s.cpp").write_text(STACK_PROGRAM)
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-I" + os.path.join(root, "include"), "-o", str(tmp_path / "s"), str(tmp_path / "s.cpp"),
                           so, "-Wl,-rpath," + os.path.dirname(so), "-lpthread"])
    r = subprocess.run([str(tmp_path / "s")], capture_output=True, text=True, timeout=60)
    assert (r.returncode, r.stdout) == (0, "0"), r
