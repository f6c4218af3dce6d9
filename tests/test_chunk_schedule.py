"""Host model of the tile list of the backward over chunks (no GPU).

lmhead_bwd_chunk.cu walks one list of tiles: in step s the dhidden tiles of chunk
s - lag, the logit tiles of chunk s, the dW tiles of chunk s - lag.  CTA pairs claim
them in list order; a tile waits for the logit tiles of its chunk (dhidden, dW), for
every reader of the chunk that held its buffer before (logits), for the first
contribution to its sum, or for the contribution before it (reproducible sums).

The model takes each size's plan from the library and checks that the list holds every
tile once, that a chunk fits its buffer and begins where a reproducible sum's term of
512 does, and that whatever a tile waits for stands earlier in the list, so that the
pair that holds it can always be waited for.  It restates the list, not the kernel.
"""
import pytest

import paper_2607_21653_gb300 as molt

TERM = 2   # 256-row tiles to a reproducible sum's term


@pytest.fixture(scope="module", autouse=True)
def _lib():
    molt.build()
    molt.load()


def spans(n, chunk, align):
    """First tiles of n tiles cut into chunks, and n at the end."""
    parts, blocks = -(-n // chunk), -(-n // align)
    return [min(n, i * blocks // parts * align) for i in range(parts + 1)]


def tile_list(rows, H, V, plan, det):
    """(kind, chunk, i, j): dhidden tile (t, h), logit tile (t, v), dW tile (v, h)."""
    align = TERM if det else 1
    n_h = -(-H // 256)
    ts = spans(-(-rows // 256), plan["chunk_tokens"] // 256, align)
    vs = spans(-(-V // 256), plan["chunk_columns"] // 256, align)
    chunks = [(ts[a], ts[a + 1], vs[b], vs[b + 1]) for a in range(len(ts) - 1) for b in range(len(vs) - 1)]
    tiles = []
    for s in range(len(chunks) + plan["lag"]):
        c = s - plan["lag"]
        if 0 <= c < len(chunks):
            t0, t1, v0, v1 = chunks[c]
            tiles += [("dh", c, t, h) for h in range(n_h) for t in range(t0, t1)]
        if s < len(chunks):
            t0, t1, v0, v1 = chunks[s]
            tiles += [("z", s, t, v) for v in range(v0, v1) for t in range(t0, t1)]
        if 0 <= c < len(chunks):
            t0, t1, v0, v1 = chunks[c]
            tiles += [("dw", c, v, h) for h in range(n_h) for v in range(v0, v1)]
    return tiles, chunks, len(vs) - 1


# each kind of ring (4 x up to 8 tiles in sixteen buffers, 8 x 4 in sixteen, 8 x 8 in
# eight, 16 x 16 in two), with fewer and with more chunks than buffers, and remainders
@pytest.mark.parametrize("det", [False, True])
@pytest.mark.parametrize("T,H,V", [(1, 640, 1), (513, 512, 4133), (769, 256, 8200), (520, 320, 66000), (1000, 768, 9000),
                                   (2305, 256, 17000), (5003, 320, 50257), (2100, 640, 14700), (3000, 1024, 9001),
                                   (5121, 1536, 32769), (4300, 2176, 8300), (16384, 4096, 65536)])
def test_every_wait_reaches_back(T, H, V, det):
    if det and H % 128:
        pytest.skip("reproducible sums need H % 128 == 0")
    plan = molt.backward_plan(T, H, V, det)
    assert plan["kernel"] == "lmhead_bwd_chunk_kernel"
    assert 1 <= plan["lag"] < plan["buffers"]
    cap_t, cap_v = -(-T // 256), -(-V // 256)
    fit_t, fit_v = min(cap_t, plan["chunk_tokens"] // 256), min(cap_v, plan["chunk_columns"] // 256)
    # the rows with a gradient are known on the device only: anything from 1 to T
    for rows in sorted({1, T, max(1, T - 255), max(1, T // 2), max(1, T // 3)}):
        tiles, chunks, n_vc = tile_list(rows, H, V, plan, det)
        at = {x: i for i, x in enumerate(tiles)}
        n_t, n_h = -(-rows // 256), -(-H // 256)
        assert len(at) == len(tiles)
        assert {x[2:] for x in tiles if x[0] == "z"} == {(t, v) for t in range(n_t) for v in range(cap_v)}
        last = {}   # (chunk, writes or reads its buffer) -> last place in the list
        for i, (kind, c, *_) in enumerate(tiles):
            last[c, kind == "z"] = i
        for c, (t0, t1, v0, v1) in enumerate(chunks):
            assert 0 < t1 - t0 <= fit_t and 0 < v1 - v0 <= fit_v
            assert not det or (t0 % TERM == 0 and v0 % TERM == 0)
        for i, (kind, c, a, b) in enumerate(tiles):
            if kind == "z":
                assert c < plan["buffers"] or last[c - plan["buffers"], False] < i
                continue
            assert last[c, True] < i
            order = c % n_vc if kind == "dh" else c // n_vc
            step = 1 if kind == "dh" else n_vc
            if order:
                assert at[kind, c - step, a, b] < i            # the contribution before
                assert at[kind, c - order * step, a, b] < i    # the first one
        assert sum(x[0] == "dh" for x in tiles) == n_t * n_vc * n_h
