"""How the backward shares its KV tiles among blocks, and the workspace that this takes: a slot of fp32 dK, dV per block of
a shared tile.  The rule is restated here from the tile schedule; the sizes are those the library asks for (148 SMs)."""
import random

import pytest

import paper_2609_32704_b200 as cowa
from oracle import cowa_oracle as orc

SMS = 148


def bwd_plan(B, Nq, Nk, Hkv, G, windows):
    """[(tiles, parts)] of the three classes (sink tiles, body, last wave) and the steps of one QO head in every tile."""
    dump = cowa.cowa_schedule_dump(cowa.SCHED_BWD, Nq, Nk, Hkv, cowa.make_params(windows=windows, softmax_scale=1.0, block_q=64, block_k=128))
    steps, i = [], 0
    while i < len(dump):
        steps.append((dump[i + 1], dump[i + 2] * G))  # KV tile, steps of the group
        i += 3 + 2 * dump[i + 2]
    sink_tiles = max((min(w[0], Nk) + 127) // 128 for w in windows)
    total = sum(n for _, n in steps) * B
    sinks = sum(n for j, n in steps if j < sink_tiles) * B
    longest_sink = max([n for j, n in steps if j < sink_tiles], default=0)
    share = total / SMS
    nsink = B * Hkv * sink_tiles
    rest = B * Hkv * (-(-Nk // 128) - sink_tiles)
    avg = (total - sinks) / rest if rest else 0.0
    parts0 = max(1, min(32, int(longest_sink / max(share / 3, 4.0) + 0.999))) if longest_sink * 4 > 3 * share else 1
    cls = [[nsink, parts0], [rest, 1], [0, 1]]
    if rest <= 2 * SMS:
        cls[1][1] = max(1, min(16, int(avg / max(share / 5, 4.0) + 0.999)))
    elif rest <= 8 * SMS and avg >= 16:
        cls[1][0], cls[2] = rest - SMS, [SMS, 4 if avg >= 32 else 2]
    ntiles, longest = B * Hkv * -(-Nk // 128), max(n for _, n in steps)
    heads = next((p for p in range(1, G) if G % p == 0 and ntiles * p >= 2 * SMS and longest * 4 * SMS <= 3 * total * p), G)
    room = ntiles * heads if heads > 1 else 0
    while slots(cls) > (room if heads >= 4 else max(room, 4 * SMS)):
        max(cls, key=lambda c: c[1])[1] -= 1
    return cls, {h: steps[h * -(-Nk // 128):(h + 1) * -(-Nk // 128)] for h in range(Hkv)}


def blocks_of(B, Nq, Nk, Hkv, G, windows, deterministic=False):
    """(blocks of the main kernel, table): how the tiles are in fact cut.  table: None, or the parts of every tile of one batch
    element, KV tiles ascending, heads within them, where few tiles are shared out by their length instead."""
    (sinks, rest, tail), steps = bwd_plan(B, Nq, Nk, Hkv, G, windows)
    nkv, run = -(-Nk // 128), [sinks[1], rest[1], tail[1]]
    per_tile = [[n for _, n in steps[h]] for h in range(Hkv)]
    nsink = sinks[0] // (B * Hkv)
    total, n_rest = B * sum(map(sum, per_tile)), B * Hkv * (nkv - nsink)
    avg = B * sum(sum(x[nsink:]) for x in per_tile) / n_rest if n_rest else 0.0
    if not deterministic:  # not all parts of body tiles that there is room for
        best = None
        for p in range(1, rest[1] + 1):
            n = sinks[0] * sinks[1] + rest[0] * p + tail[0] * tail[1]
            t = (4 + avg / 2 / p) * (max(n / SMS, 1.0) + 0.5) + (0.02 * rest[0] * p if p > 1 else 0)
            if best is None or t < best:
                best, run[1] = t, p
    blocks = sinks[0] * run[0] + rest[0] * run[1] + tail[0] * run[2]
    longest = [max([n for x in per_tile for n in x[a:b]], default=0) for a, b in ((0, nsink), (nsink, nkv))]
    rows, share = B * Hkv * G * Nq, total / SMS
    uneven = max(longest[0] / run[0], longest[1] / run[1]) > 1.2 * share
    if deterministic or nkv * Hkv * B > 2 * SMS or rows > 131072 or not (uneven or Nq <= 4096 and rows <= 81920):
        return blocks, None
    cnt = [per_tile[h][j] for j in range(nkv) for h in range(Hkv)]
    room, best, x = min(slots([sinks, rest, tail]), 65535 * B), None, max(longest + [4])
    while True:
        n = B * sum(max(-(-c // x), 1) for c in cnt)
        if n > room:
            break
        t = 10 + x
        if n > SMS:
            t = max(t, 5 + (total + 5 * n) / SMS + 0.4 * (5 + x))
        if n > len(cnt) * B:
            t += 0.04 * n
        if best is None or t < best[0]:
            best = t, x, n
        if x == 4:
            break
        x = max(x * 7 // 8, 4)
    if best is None:
        return blocks, None
    return best[2], [max(-(-c // best[1]), 1) for c in cnt]


def slots(cls):
    return sum(t * p for t, p in cls if p > 1)


def slots_asked_for(B, T, Hq, Hkv, D, params):
    """Slots in the workspace that cowa_bwd asks for."""
    extra = cowa.cowa_bwd_workspace_bytes(B, T, Hq, Hkv, D, params) - B * Hq * (-(-T // 64) * 64) * (D + 2) * 4
    assert extra % (2 * 128 * D * 4) == 0
    return extra // (2 * 128 * D * 4)


CASES = [
    (1, 3000, 8, 1, 128, 40, 200, 8, 5),     # one rank of eight
    (4, 2048, 16, 2, 64, 16, 256, 2, 0),
    (1, 20001, 8, 1, 128, 128, 896, 8, 3),
    (1, 65536, 8, 1, 128, 128, 2048, 8, 7),
    (1, 131072, 8, 1, 128, 128, 4096, 8, 0),
    (1, 16384, 16, 4, 128, 128, 1024, 4, 0),
    (1, 8192, 8, 8, 64, 100, 1024, 8, 0),    # a shared last wave
    (2, 700, 3, 1, 128, 0, 64, 1, 0),        # an odd group
]


@pytest.mark.parametrize("B,T,Hq,Hkv,D,sink,local,hg,off", CASES)
def test_workspace_holds_the_shared_tiles_and_no_more(B, T, Hq, Hkv, D, sink, local, hg, off):
    p = cowa.make_params(sink=sink, local=local, softmax_scale=0.1, hkv_global=hg, hkv_offset=off)
    cls, _ = bwd_plan(B, T, T, Hkv, Hq // Hkv, orc.default_windows(T, hg, sink, local)[off:off + Hkv])
    assert slots_asked_for(B, T, Hq, Hkv, D, p) == slots(cls) <= 7 * SMS


@pytest.mark.parametrize("B,T,Hq,Hkv,D,sink,local,hg,off", CASES)
def test_blocks_fit_the_slots(B, T, Hq, Hkv, D, sink, local, hg, off):
    windows = orc.default_windows(T, hg, sink, local)[off:off + Hkv]
    cls, steps = bwd_plan(B, T, T, Hkv, Hq // Hkv, windows)
    for deterministic in (False, True):
        blocks, table = blocks_of(B, T, T, Hkv, Hq // Hkv, windows, deterministic)
        if table is None:
            assert blocks <= sum(t * p for t, p in cls)
        else:  # a slot per block, whether it needs one or not
            assert not deterministic and blocks == B * sum(table) <= slots(cls)
            assert all(p <= max(n, 1) for p, n in zip(table, (steps[h][j][1] for j in range(-(-T // 128)) for h in range(Hkv))))


def test_packed_workspace_without_parameters_is_enough_for_all():
    rng = random.Random(5)
    for _ in range(300):
        B, Hkv, G, D = rng.randint(1, 40), rng.choice([1, 2, 8]), rng.choice([1, 3, 4, 8]), rng.choice([64, 128])
        total = max(B, int(2 ** rng.uniform(5, 17)))
        args = (B, total, Hkv * G, Hkv, D)
        most = cowa.lib().cowa_bwd_varlen_workspace_bytes(*args, None)
        p = cowa.make_params(sink=rng.choice([0, 4, 128, 3000]), local=rng.choice([1, 100, 2048, 10 ** 6]), softmax_scale=0.1,
                             full_attn=rng.random() < 0.2)
        need = cowa.cowa_bwd_varlen_workspace_bytes(*args, p)
        assert need <= most <= cowa.lib().cowa_bwd_varlen_workspace_bytes(*args, None)
        base = Hkv * G * (total // 64 + B) * 64 * (D + 2) * 4
        assert most - base <= 14 * SMS * 2 * 128 * D * 4
