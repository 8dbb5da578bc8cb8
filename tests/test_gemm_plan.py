"""The launch rules of the tensor-core GEMMs, compiled for the host: tiles that cover every token once, rings that fit, and waits of the
accumulator ring that can only return for the phase they mean."""
import functools
import random

import pytest

import gemm_plan as gp

SIZES = [97, 128, 129, 150, 160, 192, 193, 224, 256, 257, 300, 384, 400, 515, 576, 700, 768, 1000, 1152, 1500, 2044, 4096]
WIDTHS = [256, 1500, 4096, 6144, 8192, 10240, 19000, 28672, 57344, 128256]


@functools.lru_cache(None)
def plans():
    """One shape for every distinct launch of a few K blocks or many: rings, widths and the halves of a pair's first tiles."""
    seen = {}
    for M in SIZES:
        for N in WIDTHS:
            for K in (128, 384, 640, 4096, 16384):
                for a8 in (False, True):
                    p = gp.pair_plan(M, N, K, a8)
                    tiles, _ = gp.pair_tiles(p)
                    seen.setdefault((p.half_units, p.n_land, p.n_a, p.n_b, p.n_acc, tuple((t.u0, t.u1) for t in tiles[:8])), (M, N, K, a8))
    return sorted(seen.values())


def test_tiles_cover_the_tokens_and_rings_fit():
    for M, N, K, a8 in plans():
        p = gp.pair_plan(M, N, K, a8)
        assert p.n_land >= p.n_a >= 4 and p.n_b >= p.n_a and p.n_land * p.stage + p.n_b * p.slot <= 192 * 1024
        assert p.n_acc * p.acc_cols + 32 * p.n_a <= 512 and p.n_acc >= (2 if p.widest > p.half_units else 1)
        done = 0
        for i in range(p.t_tiles):
            t = gp.tile_at(p, i)
            assert (t.n0, t.t0) == (0, done) and 1 <= t.u0 <= 4 and 0 <= t.u1 <= t.u0 and (t.u1 == 0 or t.u0 == p.half_units)
            done += 32 * (t.u0 + t.u1)
        assert done - 32 < M <= done


def test_an_accumulator_slot_belongs_to_one_half():
    """Issuer and epilogue of a half wait for every phase of their slots in turn; a parity cannot be mistaken then. A slot that
    both halves took in turn would be waited on by warps that have not seen its phase before."""
    for M, N, K, a8 in plans():
        _, slots = gp.pair_tiles(gp.pair_plan(M, N, K, a8))
        owner, uses = {}, {}
        for h in range(2):
            for s, ph in slots[h]:
                if s >= 0:
                    assert owner.setdefault(s, h) == h, f"{M} x {N} x {K}: slot {s} serves both halves"
                    assert ph == uses.get(s, 0) % 2
                    uses[s] = uses.get(s, 0) + 1


class Walk:
    """The waits and arrivals of one CTA pair as the kernel makes them, one step of a randomly chosen role at a time. Barriers count
    completed phases; a wait sees their parity only, and the walk checks that it returned for the phase that was meant."""

    def __init__(self, p, n_kb, rng, count):
        tiles, slots = gp.pair_tiles(p)
        self.p, self.n_kb, self.rng = p, n_kb, rng
        self.tiles, self.slots = tiles[:count], [s[:count] for s in slots]
        used, self.nth = {}, [[], []]  # which use of its slot a half is
        for i in range(len(self.tiles)):
            for h in range(2):
                s = self.slots[h][i][0]
                self.nth[h].append(used.get(s, 0))
                if s >= 0:
                    used[s] = used.get(s, 0) + 1
        self.full, self.empty = [0] * 4, [0] * 4
        total = len(self.tiles) * n_kb
        self.s8_full, self.s8_done = [False] * total, [0] * total
        self.queue = [[], []]  # arrivals of the issuers' commits: in order, some time after the commit

    def parity(self, phases, parity, meant):
        if phases % 2 == parity:
            return False
        assert phases == meant + 1, f"a wait for phase {meant} returned in phase {phases}"
        return True

    def issuer(self, h):
        for i in range(len(self.tiles)):
            slot, ph = self.slots[h][i]
            if slot >= 0:
                while self.nth[h][i] > 0 and not self.parity(self.empty[slot], ph ^ 1, self.nth[h][i] - 1):
                    yield False
            for kb in range(self.n_kb):
                b = i * self.n_kb + kb
                while not self.s8_full[b]:
                    yield False
                self.queue[h].append(("s8", b))
                yield True
            if slot >= 0:
                self.queue[h].append(("acc", slot))
            yield True

    def commits(self, h):
        while True:
            if self.queue[h]:
                what, i = self.queue[h].pop(0)
                if what == "s8":
                    self.s8_done[i] += 1
                else:
                    self.full[i] += 1
                yield True
            else:
                yield False

    def group(self, g):
        for b in range(g, len(self.s8_full), 4):
            while b >= self.p.n_a and self.s8_done[b - self.p.n_a] < 2:
                yield False
            self.s8_full[b] = True
            yield True

    def epilogue(self, h):
        for i, t in enumerate(self.tiles):
            slot, ph = self.slots[h][i]
            if slot < 0:
                continue
            while not self.parity(self.full[slot], ph, self.nth[h][i]):
                yield False
            for _ in range(t.u1 if h else t.u0):
                yield True
            self.empty[slot] += 1
            yield True

    def run(self):
        roles = {("issuer", h): self.issuer(h) for h in range(2)} | {("epilogue", h): self.epilogue(h) for h in range(2)}
        roles |= {("group", g): self.group(g) for g in range(4)}
        commits = {("commits", h): self.commits(h) for h in range(2)}
        weight = {k: self.rng.choice((1, 1, 4, 20)) for k in roles | commits}
        idle = 0
        while roles:
            names = list(roles) + list(commits)
            if self.rng.random() < 0.02:
                weight[self.rng.choice(names)] = self.rng.choice((0.1, 1, 4, 20))
            k = self.rng.choices(names, [weight[n] for n in names])[0]
            try:
                idle = 0 if next((roles | commits)[k]) else idle + 1
            except StopIteration:
                del roles[k]
                idle = 0
            assert idle < 20000, "no role gets on"


def test_waits_return_for_the_phase_they_mean_under_any_interleaving():
    for n, (M, N, K, a8) in enumerate(plans()):
        p = gp.pair_plan(M, N, K, a8)
        if p.c_tiles * p.t_tiles <= gp.SMS // 2:
            continue  # one tile a pair: no slot comes round again
        for n_kb in (1, 2, 3, 5, 8):
            for seed in range(3):
                Walk(p, n_kb, random.Random(n * 100 + n_kb * 10 + seed), 6).run()


@pytest.mark.parametrize("M,N,K,a8,want", [
    (8, 57344, 8192, False, "stream"), (16, 4096, 4096, False, "stream"), (9, 5120, 4096, False, "split"), (96, 57344, 8192, True, "split"),
    (128, 18944, 4096, False, "split"), (128, 18945, 4096, False, "pair_ts"), (256, 8192, 8192, False, "split"), (257, 8192, 8192, False, "pair_ts"),
    (4096, 57344, 8192, True, "pair"), (4096, 57344, 8192, False, "pair_ts"), (2044, 28672, 16384, True, "pair_ts"),
    # 8-bit tokens: up to 128 the split kernel while its channel tiles are resident at once; the kernel of whole 256-token tiles only
    # for many tokens that fill them
    (128, 37888, 4096, True, "split"), (97, 37889, 4096, True, "pair_ts"), (97, 57344, 8192, True, "pair_ts"), (128, 128256, 4096, True, "pair_ts"),
    (129, 57344, 8192, True, "pair_ts"), (515, 57344, 8192, True, "pair_ts"), (1023, 57344, 8192, True, "pair_ts"), (1024, 57344, 8192, True, "pair"), (1100, 57344, 8192, True, "pair_ts"),
    (1215, 28672, 4096, True, "pair_ts"), (1216, 28672, 4096, True, "pair"), (2044, 28672, 4096, True, "pair"), (2044, 28672, 1920, True, "pair_ts"),
    (2044, 4096, 4096, True, "pair_ts"),
])
def test_route(M, N, K, a8, want):
    assert gp.route(M, N, K, a8) == want


def test_ctas_that_fit_one_sm_find_their_tensor_memory():
    """The split kernel's clusters hold their columns until all their CTAs have met, and an allocation waits without a bound: two launches
    whose CTAs share SMs by shared memory, but not by tensor memory, could each hold what the other waits for."""
    forms = gp.split_shapes()
    for a in forms:
        for b in forms:
            for c in forms + [(0, 0, 0, 0)]:
                group = [f for f in (a, b, c) if f[0]]
                if sum(smem + 1024 for *_, smem in group) <= 228 * 1024:
                    assert sum(cols for _, _, cols, _ in group) <= 512, group


def test_ctas_kept_to_one_an_sm_find_their_tensor_memory_too():
    """The same where one of the CTAs is of a launch kept to one to an SM; two of those never share one."""
    one = (64, 0, 256, gp.alone_smem())
    assert 2 * (one[3] + 1024) > 228 * 1024
    for b in gp.split_shapes() + gp.whole_shapes():
        for c in gp.split_shapes() + [(0, 0, 0, 0)]:
            group = [f for f in (one, b, c) if f[0]]
            if sum(smem + 1024 for *_, smem in group) <= 228 * 1024:
                assert sum(cols for _, _, cols, _ in group) <= 512, group


def test_two_ctas_of_33_to_96_tokens_leave_no_room_for_a_rotation():
    """16 elements to a thread keep 2176 floats of shared memory at the least."""
    for nt, _, _, smem in gp.split_shapes():
        if 32 < nt < 128:
            assert 0 <= 228 * 1024 - 2 * (smem + 1024) < 2176 * 4


@pytest.mark.parametrize("M,ctas,splits,want", [
    (96, 96, 3, True), (64, 96, 3, False), (65, 75, 1, True), (65, 74, 2, False), (128, 129, 3, True), (128, 130, 2, False), (128, 128, 4, True),
    (100, 120, 5, False), (100, 128, 8, False), (96, 240, 5, False),
])
def test_launches_kept_to_one_cta_an_sm(M, ctas, splits, want):
    assert gp.alone(M, ctas, splits) == want


def test_narrow_forms_that_take_an_sm_alone_share_it_with_no_other():
    for a in gp.whole_shapes():
        for b in gp.whole_shapes() + gp.split_shapes():
            assert a[3] + b[3] + 2048 > 228 * 1024 or a[2] + b[2] <= 512, (a, b)


@pytest.mark.parametrize("M,N,K,a8,want", [
    (256, 4096, 4096, False, 128), (192, 6144, 4096, False, 64), (130, 4096, 4096, False, 192), (512, 4096, 4096, False, 256),
    (256, 8192, 28672, False, 256), (256, 4096, 14336, True, 128), (130, 6144, 4096, True, 64), (512, 4096, 14336, True, 256),
])
def test_width_above_128_tokens(M, N, K, a8, want):
    assert gp.width_whole(M, N, K, a8) == want


@pytest.mark.parametrize("tiles,K,M,a8,want", [
    (32, 4096, 64, False, 6), (32, 4096, 65, False, 3), (32, 14336, 128, False, 8), (32, 14336, 88, True, 8), (32, 14336, 89, True, 4),
    (48, 4096, 96, False, 5), (48, 4096, 97, False, 2), (48, 4096, 66, True, 2), (64, 8192, 96, True, 4), (80, 8192, 128, True, 3), (8, 8192, 128, True, 8),
    (1, 32, 100, True, 1), (224, 4096, 100, True, 1), (3, 640, 128, False, 1), (20, 1408, 100, True, 2),
])
def test_k_splits_of_two_ctas_to_an_sm(tiles, K, M, a8, want):
    assert gp.splits_pairs(tiles, K, M, a8) == want


def test_every_split_has_k_blocks_and_a_place():
    for tiles in list(range(1, 40)) + [48, 64, 80, 131, 148, 149, 224, 296, 448]:
        for K in (32, 96, 640, 1280, 1408, 4096, 8192, 14336, 28672):
            for M in (17, 64, 65, 88, 89, 96, 97, 128):
                for a8 in (False, True):
                    s = gp.splits_pairs(tiles, K, M, a8)
                    assert 1 <= s <= 8 and (s == 1 or (K >= 640 * s and tiles * s <= 2 * 148 * 7 // 8))


def test_clusters_of_one_cta_an_sm_all_find_a_place():
    """Whole clusters that a 148-SM GPU places at once with a CTA to an SM, as its driver reports them."""
    places = {1: 148, 2: 74, 3: 45, 4: 33, 5: 26, 6: 22, 7: 15, 8: 15}
    for tiles in range(1, 149):
        for K in (640, 1280, 4096, 8832, 14336, 28672):
            s = gp.splits_whole(tiles, K)
            assert s == 1 or tiles <= places[s], (tiles, K, s)
    assert [gp.splits_whole(t, 14336) for t in (15, 16, 18, 21, 22)] == [8, 6, 6, 6, 5]
