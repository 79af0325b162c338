"""The paper's GA at the population sizes where the lanes per individual change, with up to
16 models and with most individuals infeasible (the repairs), against a run in numpy: the
same genome, and its fitness by the same float32 sums."""
import numpy as np
import pytest

from paper_2609_02109_gb300 import workload as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mf():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2609_02109_gb300 import mf as m
    return m


def _run(prob, ctx, p, seed):
    """The GA in numpy on the device's own table (float32 sums in model order)."""
    ks = np.asarray(prob["n_options"], np.int64)
    n, pop = ks.size, p["pop"]
    off = np.concatenate([[0], np.cumsum(ks)])[:-1]
    _, _, u, ok = ctx.fc_table()
    vr = np.asarray(prob["demand"], np.float32)[:, 1]
    M = np.uint64

    def draw(gen, slot, purpose, j):
        slot, j = np.broadcast_arrays(np.asarray(slot, M), np.asarray(j, M))
        ctr = (M(gen) << M(32)) | (slot << M(12)) | M(purpose << 8) | j
        with np.errstate(over="ignore"):
            z = M(seed) + (ctr + M(1)) * M(0x9E3779B97F4A7C15)
            z = (z ^ (z >> M(30))) * M(0xBF58476D1CE4E5B9)
            z = (z ^ (z >> M(27))) * M(0x94D049BB133111EB)
        return z ^ (z >> M(31))

    below = lambda z, k: (((z >> M(32)) * np.asarray(k, M)) >> M(32)).astype(np.int64)  # noqa: E731

    def fitness(g):
        J = np.zeros(g.shape[:-1], np.float32)
        V = np.zeros(g.shape[:-1], np.float32)
        good = np.ones(g.shape[:-1], bool)
        for i in range(n):
            J = J + u[off[i] + g[..., i]]
            V = V + vr[off[i] + g[..., i]]
            good &= ok[off[i] + g[..., i]]
        return np.where(good & (V <= np.float32(prob["vram_cap"])), J, np.float32(-np.inf))

    def settle(g, gen, first):
        f = fitness(g)
        bad = np.flatnonzero(np.isneginf(f))
        bad = bad[bad >= first]
        if p["repair"] and bad.size:
            j = np.arange(256 // n)[:, None] * n + np.arange(n)[None, :]
            cand = below(draw(gen, bad[:, None, None], 7, j[None]), ks)
            cf = fitness(cand)
            at = np.argmax(~np.isneginf(cf), axis=1)
            got = np.flatnonzero(~np.isneginf(cf[np.arange(bad.size), at]))
            g[bad[got]], f[bad[got]] = cand[got, at[got]], cf[got, at[got]]
        return f

    slot, gene = np.arange(pop)[:, None], np.arange(n)[None, :]
    g = below(draw(0, slot, 0, gene), ks)
    f = settle(g, 0, 0)
    for gen in range(1, p["gens"]):
        win = []
        for purpose in (1, 2):
            s = np.sort(below(draw(gen, slot, purpose, np.arange(p["tournament"])[None, :]), pop), axis=1)
            win.append(s[np.arange(pop), np.argmax(f[s], axis=1)])
        cross = (draw(gen, slot, 6, 0) >> M(40)) < round(p["crossover_p"] * 2 ** 24)
        take = (draw(gen, slot, 3, gene) >> M(63)).astype(bool) & cross
        c = np.where(take, g[win[1]], g[win[0]])
        mut = (draw(gen, slot, 4, gene) >> M(40)) < np.floor(p["mutation_p"] * 2 ** 24 + 0.5)
        c = np.where(mut, below(draw(gen, slot, 5, gene), ks), c)
        if p["elitism"]:
            c[0] = g[int(np.argmax(f))]
        g, f = c, None
        f = settle(g, gen, 1 if p["elitism"] else 0)
    b = int(np.argmax(f))
    return f[b], g[b]


@pytest.mark.parametrize("pop", [2, 100, 128, 129, 256, 257, 512, 513, 600, 1024])
@pytest.mark.parametrize("options,cap", [([12, 9, 9, 9, 9], 55.0), ([12, 9, 9, 9, 9], 25.0), ([7, 10, 7], 30.0),
                                         ([3] * 16, 160.0), ([30], 8.0), ([10] * 12, 118.0)])
def test_every_population(mf, pop, options, cap):
    prob = W.make_problem(options, 8, 64, 64, 5, cap)
    fc = W.fc_scenario(prob, 9)
    fc["tau"] = np.full(len(options), -0.5, np.float32)
    for elitism, repair, tournament in ((1, 1, 3), (0, 1, 2), (1, 0, 40)):
        p = dict(W.PAPER_GA_PARAMS, pop=pop, gens=6, elitism=elitism, repair=repair, tournament=tournament)
        with mf.Context(prob) as ctx:
            ctx.fc_set(fc)
            fit, genome = ctx.fc_ga_run(p, 77)
            want, g = _run(prob, ctx, p, 77)
        assert np.float32(fit) == want and np.array_equal(genome, g)
