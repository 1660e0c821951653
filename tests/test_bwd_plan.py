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
