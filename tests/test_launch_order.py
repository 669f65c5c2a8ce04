"""Which kernels the library launches, in which order and with what they may read before the launch in front of
them is done: the host code on a CUDA runtime that runs nothing (tests/helpers/fake_cudart.cu)."""
import ctypes as C

import numpy as np
import pytest

import helpers

V_Q, V_P, B, K = 1000, 4000, 40, 4


def _aligned(n):
    raw = np.zeros(n + 64, np.uint8)
    at = -raw.ctypes.data % 64
    return raw[at:at + n]


class Lib:
    """One context of the library on the fake runtime. Every array is zeros, or what a call was given."""

    def __init__(self, v_q=V_Q, v_p=V_P, max_batch=B, k=K, vocab_map=None):
        self.L, self.k, self.v_q, self.v_p, self.kept = helpers.fake_runtime_lib(), k, v_q, v_p, []
        self.L.fake_unpin_all()
        self.L.fake_no_driver_functions(0)
        h = C.c_void_p()
        self.call("od_create", C.byref(h), 0, v_q, v_p, max_batch, k)
        self.ctx = h
        if vocab_map is None:
            vocab_map = np.where(np.arange(v_q) % 10 < 7, np.arange(v_q) + 1, -1)
        self.call("od_set_vocab_map", h, self.array(vocab_map.astype(np.int32)))
        self.call("od_cache_build", h, None, None, None, C.c_int64(0))
        self.log()

    def close(self):
        self.call("od_destroy", self.ctx)

    def call(self, name, *args):
        assert getattr(self.L, name)(*args) == 0, name

    def array(self, a):
        b = _aligned(a.nbytes).view(a.dtype)[:a.size]
        b[:] = a.ravel()
        self.kept.append(b)
        return C.c_void_p(b.ctypes.data)

    def zeros(self, n, dtype=np.int32):
        return self.array(np.zeros(n, dtype))

    def log(self):
        """(kernel, grid, early) of every launch, (direction, bytes) of every copy, since the last call."""
        out = []
        for line in self.L.fake_log().decode().splitlines():
            w = line.split()
            out.append((w[0], tuple(map(int, w[1:4])), int(w[4])) if len(w) == 5 else (w[0], int(w[1])))
        return out

    def early(self, *kernels):
        """The launches' names and their `early`, copies left out."""
        return [(x[0], x[2]) for x in self.log() if len(x) == 3 and (not kernels or x[0] in kernels)]

    def inputs(self, n=B):
        """Pointers that the calls below share: outputs and inputs of a step for n sequences."""
        K, z = self.k, self.zeros
        self.n = n
        names = dict(draft_ids=n * K, draft_len=n, q_sel=n * K, temperature=n, seed=2 * n, tgt_ids=n * K, q_prime=n * K,
                     span_start=n * K, span_len=n * K, m=n, tail=n, row_max=n * (K + 1), row_sum=n * (K + 1), p_sel=n * K,
                     ratio=n * K, n_acc=n, n_draft=n, vflags=n, token=n, mass=n, sflags=n, counters=8)
        self.p = {name: z(count) for name, count in names.items()}
        self.p["q_rows"] = z(n * K * self.v_q)
        self.p["logits"] = z(n * (K + 1) * self.v_p, np.uint16)
        return self.p

    def strides(self):
        return C.c_int64(self.v_p), C.c_int64(self.v_p * (self.k + 1))

    def map(self):
        p = self.p
        self.call("od_map_proposals", self.ctx, self.n, self.k, p["draft_ids"], p["draft_len"], p["q_sel"], p["tgt_ids"], p["q_prime"],
                  p["span_start"], p["span_len"], p["m"], p["tail"], p["counters"], None)

    def verify(self):
        p = self.p
        self.call("od_verify", self.ctx, self.n, self.k, p["logits"], 1, *self.strides(), p["tgt_ids"], p["q_prime"], p["span_len"], p["m"],
                  p["temperature"], p["seed"], C.c_uint64(0), p["row_max"], p["row_sum"], p["p_sel"], p["ratio"], p["n_acc"],
                  p["n_draft"], p["vflags"], None)

    def sample(self):
        p = self.p
        self.call("od_sample_residual", self.ctx, self.n, self.k, p["logits"], 1, *self.strides(), p["row_max"], p["row_sum"], p["q_rows"],
                  p["draft_ids"], p["tgt_ids"], p["q_prime"], p["span_start"], p["span_len"], p["m"], p["tail"], p["n_acc"],
                  p["temperature"], p["seed"], C.c_uint64(0), p["token"], p["mass"], p["sflags"], None)

    def step(self):
        p = self.p
        self.call("od_step", self.ctx, self.n, self.k, p["draft_ids"], p["draft_len"], p["q_sel"], p["q_rows"], p["logits"], 1,
                  *self.strides(), p["temperature"], p["seed"], C.c_uint64(0), p["tgt_ids"], p["q_prime"], p["span_start"],
                  p["span_len"], p["m"], p["tail"], p["counters"], p["row_max"], p["row_sum"], p["p_sel"], p["ratio"], p["n_acc"],
                  p["n_draft"], p["vflags"], p["token"], p["mass"], p["sflags"], None)

    def step_host(self):
        p = self.p
        self.call("od_step_host", self.ctx, self.n, self.k, p["draft_ids"], p["draft_len"], p["q_sel"], p["q_rows"], p["logits"], 1,
                  p["temperature"], p["seed"], C.c_uint64(0), p["n_acc"], p["n_draft"], p["token"], p["tgt_ids"], p["m"],
                  p["vflags"], p["sflags"], None)

    def pin(self, name, bytes_=None):
        a = next(a for a in self.kept if a.ctypes.data == self.p[name].value)
        self.L.fake_pin(a.ctypes.data, a.nbytes if bytes_ is None else bytes_)


@pytest.fixture
def lib():
    made = []

    def make(**kw):
        made.append(Lib(**kw))
        return made[-1]
    yield make
    for x in made:
        x.close()


# ---- what the sampler may read ahead: the translation's outputs, where the launch in front let it start only after
# the translation was complete

@pytest.mark.parametrize("pinned", [True, False])
@pytest.mark.parametrize("grid", [0, 100])
def test_the_draw_from_host_buffers_reads_nothing_ahead_of_the_rows_that_are_fetched(lib, pinned, grid):
    c = lib()
    c.inputs()
    c.call("od_set_option", c.ctx, b"verify_grid", C.c_int64(grid))
    c.call("od_host_step_reserve", c.ctx, 1)
    if pinned:
        c.pin("logits"); c.pin("q_rows")
    c.step_host()
    step2 = [("od_verify_stream_kernel", -1), ("od_verify_decide_kernel", -1)] if grid else [("od_verify_rows_kernel", -1)]
    fetch = lambda name: [(name, -1)] if pinned else []
    assert c.early() == ([("od_map_kernel", 0)] + fetch("fetch_logits_kernel") + step2 + fetch("fetch_drafter_kernel") +
                         [("od_sample_kernel", 0 if pinned else 1)])


@pytest.mark.parametrize("kw,lens,fetched", [
    (dict(v_q=1000, v_p=4000, k=2), 1, True), (dict(v_q=7000, v_p=40000, k=1), 1, False), (dict(v_q=7000, v_p=40000, k=1), 2, False),
    (dict(v_q=7000, v_p=40000, k=1), 0, True), (dict(v_q=7000, v_p=40000, k=2), 2, True), (dict(v_q=7000, v_p=14000, k=1), 1, True),
    (dict(v_q=7000, v_p=13992, k=1), 1, True), (dict(v_q=30000, v_p=59992, k=1), 1, True), (dict(v_q=30000, v_p=60000, k=1), 1, False),
    (dict(v_q=40000, v_p=80000, k=1, vocab_map=np.arange(40000)), 1, True)])
def test_large_buffers_with_one_token_from_every_sequence_are_copied(lib, kw, lens, fetched):
    """And not: small ones, an empty proposal among them, two tokens, drafter rows longer than the target's, one vocabulary."""
    c = lib(max_batch=40, **kw)
    p = c.inputs(40)
    next(a for a in c.kept if a.ctypes.data == p["draft_len"].value)[:] = [1] * 20 + [lens] + [1] * 19
    c.call("od_host_step_reserve", c.ctx, 1)
    c.pin("logits"); c.pin("q_rows")
    c.log()
    c.step_host()
    log = c.log()
    assert [x[0] for x in log if x[0].startswith("fetch")] == (["fetch_logits_kernel", "fetch_drafter_kernel"] if fetched else [])
    rows = [x[1] for x in log if x[0] == "to_device" and x[1] >= 1 << 20]
    assert sorted(rows) == ([] if fetched else sorted([40 * 2 * kw["v_p"] * 2, 40 * kw["v_q"] * 4]))


# page-locked only in part (the range ends inside), off 16 bytes, and a driver that does not say how far the range goes
@pytest.mark.parametrize("how", ["short", "offset", "no_driver", "one_pageable"])
def test_buffers_that_the_device_cannot_read_for_certain_are_copied(lib, how):
    c = lib()
    p = c.inputs()
    c.call("od_host_step_reserve", c.ctx, 1)
    n = B * (K + 1) * V_P * 2
    if how == "offset":
        p["logits"] = C.c_void_p(c.zeros(n + 64, np.uint8).value + 8)
        c.L.fake_pin(p["logits"], n)
    else:
        c.pin("logits", n - 1 if how == "short" else None)
    if how != "one_pageable":
        c.pin("q_rows")
    c.L.fake_no_driver_functions(how == "no_driver")
    c.step_host()
    assert not any(x[0].startswith("fetch") for x in c.log())


@pytest.mark.parametrize("calls,early", [("sample", [0]), ("map sample", [0]), ("map verify sample", [1]), ("map verify sample sample", [1, 0]),
                                         ("map verify map sample", [0]), ("step sample", [0]), ("map verify step sample", [0])])
@pytest.mark.parametrize("n", [1, B])
def test_a_draw_reads_the_translation_ahead_only_behind_a_verification(lib, calls, early, n):
    c = lib()
    c.inputs(n)
    c.call("od_set_option", c.ctx, b"early_inputs", C.c_int64(0))
    for name in calls.split():
        getattr(c, name)()
    seen = c.early("od_sample_kernel", "od_step_kernel")
    assert [e for k, e in seen if k == "od_sample_kernel"] == early
    assert ("od_step_kernel" in [k for k, _ in seen]) == ("step" in calls)


# ---- how many blocks draw for a sequence

@pytest.mark.parametrize("v_p,blocks", [(102400, 4), (128000, 6), (153600, 6), (160000, 8)])
def test_a_part_with_more_mapped_ids_than_two_blocks_can_stage_is_cut_in_the_samplers_own_steps(lib, v_p, blocks):
    """Most of the ids of a part mapped: 25600 of them are 100 KB. Five blocks would do for 128000 ids; they are the
    one-launch step's."""
    c = lib(v_q=65000, v_p=v_p, max_batch=200, k=1, vocab_map=np.arange(65000, dtype=np.int32) + 1)
    c.inputs(200)
    c.map(); c.verify(); c.log()
    c.sample()
    assert [x for x in c.log() if x[0] == "od_sample_kernel"] == [("od_sample_kernel", (blocks, 200, 1), 1)]


# a device that has room for no cluster of this many blocks, as the part of a divided one may; every number of a shard's
# sequences, narrow and wide windows, and tiles per warp that the caller sets
@pytest.mark.parametrize("limit", [1, 3, 8, 16])
@pytest.mark.parametrize("v_p", [1000, 152064, 4000000])
def test_a_shards_mass_asks_for_no_cluster_that_the_device_has_no_room_for(lib, limit, v_p):
    helpers.fake_runtime_lib().fake_cluster_limit(limit)
    try:
        c = lib(v_q=1000, v_p=v_p, max_batch=512, k=1)
        c.L.fake_no_driver_functions(1)                     # (the device is asked again for every context)
        c.call("od_destroy", c.ctx)
        c.call("od_create", C.byref(c.ctx), 0, 1000, v_p, 512, 1)
        c.call("od_set_vocab_map", c.ctx, c.array(np.arange(1000, dtype=np.int32)[::-1].copy()))
        p = c.zeros(64)                                     # (nothing is read)
        for tiles in (0, 1, 1000):
            c.call("od_set_option", c.ctx, b"sample_tiles_per_warp", C.c_int64(tiles))
            for n in (1, 2, 37, 148, 149, 512):
                c.log()
                c.call("od_sample_shard_mass", c.ctx, n, 1, 0, v_p, p, 1, C.c_int64(v_p), C.c_int64(2 * v_p), *[p] * 11, p, p, None)
                (name, grid, _), = c.log()
                assert name == "od_sample_shard_kernel" and grid[0] == n and grid[1] <= limit
    finally:
        helpers.fake_runtime_lib().fake_cluster_limit(16)
