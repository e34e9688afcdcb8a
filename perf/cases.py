"""The work that programs using this library have it do, as timed cases.

Every case is one call pattern of the public interface (the Python binding,
and the C entry points of include/sw.h where the result stays in device
memory): a chain of sweeps followed by a read of its E/M trace and its state,
a host loop that sets the state, sweeps and reads E and M, a batch of
replicas advanced by a chunk, a label query, Potts sweeps and phi^4 cluster
updates.

  kind   chain   sw_sweep(n) on one lattice, then the trace and the spins
         step    sw_set_state_async from pinned host memory, one sweep, E and M
         batch   sw_batch_sweep(n) on many replicas, then every trace and state
         labels  sw_labels of the next sweep's bonds, into device memory
         potts   n sweeps of a q-state Potts lattice, then trace and states
         phi4    n multicluster updates of an O(4) field, then trace and field
"""
from __future__ import annotations

import ctypes
import math

import numpy as np
import torch

import paper_2302_14720_gb300 as sw

BETA_C = 0.44068679   # critical coupling of the Ising model as the benchmark quotes it
KAPPA_C = 0.304       # the hopping coupling of the phi^4 benchmark
MIX_SIDES = (64, 128, 256, 512, 1024)  # sides of the replica mix
MOST_SITES = 10 * 8192 * 8192          # site-updates of one pass, at most

# The C interface for calls that leave their result in device memory.
_abi = ctypes.CDLL(sw.LIBRARY_PATH)
for _name, (_res, _args) in sw.SIGNATURES.items():
    getattr(_abi, _name).restype = _res
    getattr(_abi, _name).argtypes = _args


def _ok(rc: int) -> None:
    if rc != sw.SW_OK:
        raise RuntimeError(f"status {rc}: {sw.sw_last_error()}")


def _potts_beta_c(q: int) -> float:
    return math.log(1.0 + math.sqrt(q))


def listed():
    return [
        # the shortest call there is: one sweep of a small lattice, read back
        # at once (an interactive or host-driven loop; launches and the read count)
        {"name": "ising_32_call", "kind": "chain", "L": 32, "beta": BETA_C, "sweeps": 1, "rule": 0, "stats": False,
         "cold": False},
        # the L = 64 configuration: a long chain of a small lattice, read per 100 sweeps
        {"name": "ising_64_chain", "kind": "chain", "L": 64, "beta": BETA_C, "sweeps": 100, "rule": 0, "stats": False,
         "cold": False},
        # an odd side (Philox pairs straddle rows, rows off 16-byte boundaries,
        # ragged tiles) with the fresh-spin rule
        {"name": "ising_1001_assign", "kind": "chain", "L": 1001, "beta": BETA_C, "sweeps": 20, "rule": 1,
         "stats": False, "cold": False},
        # the L = 1024 configuration: cold start, cluster statistics of every sweep
        {"name": "ising_1024_stats", "kind": "chain", "L": 1024, "beta": BETA_C, "sweeps": 20, "rule": 0, "stats": True,
         "cold": True},
        # the headline lattice as a chain at the critical coupling
        {"name": "ising_8192_chain", "kind": "chain", "L": 8192, "beta": BETA_C, "sweeps": 10, "rule": 0,
         "stats": False, "cold": False},
        # the headline lattice driven from the host: state in, one sweep, E and M out
        {"name": "ising_8192_step", "kind": "step", "L": 8192, "beta": 0.5},
        # the replica mix of a temperature scan, advanced by one chunk
        {"name": "batch_256_mix", "kind": "batch", "replicas": 256, "top": 1024, "sweeps": 50, "mix": 4},
        # cluster labels for an analysis program, left in device memory
        {"name": "labels_4096", "kind": "labels", "L": 4096, "beta": BETA_C},
        # the Potts runs of the benchmark: L2-resident and large
        {"name": "potts_q3_1024", "kind": "potts", "L": 1024, "q": 3, "beta": _potts_beta_c(3), "sweeps": 20},
        {"name": "potts_q3_8192", "kind": "potts", "L": 8192, "q": 3, "beta": _potts_beta_c(3), "sweeps": 5},
        # phi^4: the smallest lattice of the paper's table, and one whose field exceeds L2
        {"name": "phi4_16", "kind": "phi4", "L": 16, "kappa": KAPPA_C, "updates": 20},
        {"name": "phi4_64", "kind": "phi4", "L": 64, "kappa": KAPPA_C, "updates": 4},
    ]


def _log_int(rng, lo: int, hi: int) -> int:
    return max(lo, min(hi, round(math.exp(rng.uniform(math.log(lo), math.log(hi))))))


def _count(rng, sites: int, most: int) -> int:
    """Sweeps of a pass: log-uniform, bounded by the largest pass."""
    return _log_int(rng, 1, max(1, min(most, MOST_SITES // sites)))


def draw(rng):
    kind = rng.choice(["chain", "chain", "chain", "step", "batch", "labels", "potts", "potts", "phi4", "phi4"])
    beta = round(rng.choice([BETA_C, rng.uniform(0.30, 0.60)]), 8)
    if kind == "chain":
        L = _log_int(rng, 8, 8192)
        return {"kind": kind, "L": L, "beta": beta, "sweeps": _count(rng, L * L, 100), "rule": int(rng.random() < 0.3),
                "stats": rng.random() < 0.3, "cold": rng.random() < 0.3}
    if kind == "step":
        return {"kind": kind, "L": _log_int(rng, 64, 8192), "beta": beta}
    if kind == "batch":
        return {"kind": kind, "replicas": _log_int(rng, 2, 256), "top": rng.choice(MIX_SIDES),
                "sweeps": rng.randint(10, 50), "mix": rng.randrange(1 << 16)}
    if kind == "labels":
        return {"kind": kind, "L": _log_int(rng, 64, 8192), "beta": beta}
    if kind == "potts":
        L, q = _log_int(rng, 64, 8192), rng.randint(2, 8)
        return {"kind": kind, "L": L, "q": q, "beta": round(_potts_beta_c(q) * rng.uniform(0.9, 1.1), 8),
                "sweeps": _count(rng, 2 * L * L, 50)}
    L = _log_int(rng, 6, 64)
    return {"kind": kind, "L": L, "kappa": round(rng.uniform(0.2, 0.4), 6), "updates": _count(rng, 10 * L**4, 20)}


def _replicas(case):
    """Sides and couplings of a replica mix: sides drawn from MIX_SIDES up to
    `top`, couplings on a grid around the critical one."""
    n, r = case["replicas"], np.random.default_rng(case["mix"])
    sides = [int(x) for x in r.choice([s for s in MIX_SIDES if s <= case["top"]], n)]
    betas = [0.40 + 0.08 * i / max(1, n - 1) for i in range(n)]
    return sides, betas


def _phi4_field(L: int, seed: int) -> torch.Tensor:
    """A field as the theory's local updates leave it: directions correlated
    between neighbours around a common one, lengths fluctuating about 1."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    f = torch.randn((L, L, L, L, 4), generator=g, device="cuda", dtype=torch.float64)
    s = f.clone()
    for d in range(4):
        s += 0.5 * (f.roll(1, d) + f.roll(-1, d))
    s += torch.randn(4, generator=g, device="cuda", dtype=torch.float64)
    length = 1.0 + 0.1 * torch.randn((L, L, L, L, 1), generator=g, device="cuda", dtype=torch.float64)
    return (s / s.norm(dim=-1, keepdim=True) * length).contiguous()


class _Batch:
    """A batch handle with its replicas and a device buffer for their states."""

    def __init__(self, case, seed):
        self.sides, betas = _replicas(case)
        self.n = case["sweeps"]
        self.t = 0
        self.h = sw.sw_batch_create(self.sides, betas, [(seed << 16) + r for r in range(len(self.sides))])
        self.spins = torch.empty(sum(L * L for L in self.sides), dtype=torch.int8, device="cuda")

    def sweep(self):
        sw.sw_batch_sweep(self.h, self.n)
        self.t += self.n

    def __del__(self):
        if getattr(self, "h", None):
            sw.sw_batch_destroy(self.h)
            self.h = None


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        b = _Batch(case, seed)
        b.sweep()  # away from the hot start
        sw.sw_batch_observables(b.h, 0, 0, 1)
        return case, b, None, None
    L = case["L"]
    if kind == "phi4":
        f = sw.Phi4(L, case["kappa"], seed)
        phi = _phi4_field(L, seed)
        torch.cuda.synchronize()
        _ok(_abi.sw_phi4_set_field(f.h, phi.data_ptr(), 0, 1))  # synchronises
        return case, f, phi, None  # phi receives the updated field
    if kind == "potts":
        p = sw.Potts(L, case["q"], case["beta"], seed)
        p.sweep(10)  # away from the hot start
        p.observables(0, 10)
        return case, p, torch.empty((L, L), dtype=torch.int8, device="cuda"), None
    lat = sw.Lattice(L, case["beta"], seed, sw.SW_INIT_COLD if case.get("cold") else sw.SW_INIT_HOT)
    lat.sweep(10)  # away from the start state
    if kind == "step":
        host = torch.empty((L, L), dtype=torch.int8, pin_memory=True).numpy()
        host[:] = lat.spins()
        return case, lat, torch.empty((L, L), dtype=torch.int8, device="cuda"), host
    lat.observables(0, 10)
    if kind == "labels":
        return case, lat, torch.empty((L, L), dtype=torch.int32, device="cuda"), None
    lat.set_rule(case["rule"])
    lat.histogram(case["stats"])
    return case, lat, torch.empty((L, L), dtype=torch.int8, device="cuda"), None


def run(state):
    case, h, out, host = state
    kind = case["kind"]
    if kind == "chain":
        n, t = case["sweeps"], h.t
        h.sweep(n)
        sw.sw_spins(h.h, h.L, out.data_ptr())
        E, M = h.observables(t, n)  # waits for the handle's stream
        r = {"spins": out, "E": E, "M": M}
        if case["stats"]:
            r["clusters"] = h.histograms(t, n)
        return r
    if kind == "step":
        h.set_state_async(host, 10)
        h.sweep(1)
        sw.sw_spins(h.h, h.L, out.data_ptr())
        E, M = h.observables(10, 1)
        return {"spins": out, "E": E, "M": M}
    if kind == "batch":
        n, t = h.n, h.t
        h.sweep()
        at = 0
        for slot, L in enumerate(h.sides):
            _ok(_abi.sw_batch_spins(h.h, slot, h.spins.data_ptr() + at, 1))
            at += L * L
        EM = [sw.sw_batch_observables(h.h, slot, t, n) for slot in range(len(h.sides))]
        return {"E": np.stack([e for e, _ in EM]), "M": np.stack([m for _, m in EM]), "spins": h.spins}
    if kind == "labels":
        sw.sw_labels(h.h, h.L, out.data_ptr())
        h.observables(0, 0)  # waits for the handle's stream
        return out
    if kind == "potts":
        n, t = case["sweeps"], h.t
        h.sweep(n)
        _ok(_abi.sw_potts_states(h.h, out.data_ptr(), 1))
        E, M = h.observables(t, n)
        return {"states": out, "E": E, "M": M}
    n, t = case["updates"], h.t
    h.sweep(n)
    _ok(_abi.sw_phi4_field(h.h, out.data_ptr(), 1))
    E, M = h.observables(t, n)
    return {"field": out, "E": E, "M": M}


def work(case):
    """Bytes: every state read and written once per sweep, other inputs and
    outputs once. Operations: the Philox rounds of the draws (two multiplies
    and four exclusive-ors each) and, for phi^4, the binary64 arithmetic of
    the projection, the bond products, the reflection and E."""
    kind = case["kind"]
    block = 60.0  # operations of one Philox block
    if kind == "batch":
        sites = sum(L * L for L in _replicas(case)[0])
        n = case["sweeps"]
        return {"bytes": 2.0 * sites * n + 2.0 * sites, "flops": sites * n * block / 2}
    L = case["L"]
    N = float(L) * L
    if kind == "chain":
        n = case["sweeps"]
        return {"bytes": 2 * N * n + 2 * N, "flops": N * n * block / 2}
    if kind == "step":
        return {"bytes": 5 * N, "flops": N * block / 2}
    if kind == "labels":
        return {"bytes": N + 4 * N, "flops": N * block / 2}
    if kind == "potts":
        n = case["sweeps"]
        return {"bytes": 2 * N * n + 2 * N, "flops": N * n * block / 2}
    n, N = case["updates"], N * N
    return {"bytes": 64 * N * n + 64 * N, "flops": N * n * (block + 7 + 8 + 9 + 32)}


# ----------------------------------------------------------------- 64 bits
#
# Only the phi^4 field, E and M are computed numbers; every other output is
# whole numbers. The update restated in plain torch (conventions O3 to O5 of
# include/sw.h).

_M32 = 0xFFFFFFFF


def _philox(c0, c1: int, c2: int, seed: int):
    """Philox-4x32-10 words of counters (c0[i], c1, c2, 0); c0 an int64 tensor."""
    def mul(a, m):
        p, q = (a >> 16) * m, (a & 0xFFFF) * m
        return (p + (q >> 16)) >> 16, (q + ((p & 0xFFFF) << 16)) & _M32

    x, y, z, w = c0, torch.full_like(c0, c1), torch.full_like(c0, c2), torch.zeros_like(c0)
    k0, k1 = seed & _M32, (seed >> 32) & _M32
    for _ in range(10):
        ha, la = mul(x, 0xD2511F53)
        hb, lb = mul(z, 0xCD9E8D57)
        x, y, z, w = hb ^ y ^ k0, lb, ha ^ w ^ k1, la
        k0, k1 = (k0 + 0x9E3779B9) & _M32, (k1 + 0xBB67AE85) & _M32
    return x, y, z, w


def _direction(seed: int, t: int):
    for k in range(1000):
        v = [(float(w.item()) + 0.5) * 2.0**-31 - 1.0 for w in _philox(torch.tensor([k], device="cuda"), t, 5, seed)]
        s = sum(x * x for x in v)
        if 2.0**-20 < s <= 1.0:
            return torch.tensor([x / math.sqrt(s) for x in v], device="cuda", dtype=torch.float64)
    raise RuntimeError("no direction found")


def _phi4_update(phi, kappa: float, seed: int, t: int):
    """One multicluster update of phi [L, L, L, L, 4], axis 3 - mu for direction mu."""
    L = phi.shape[0]
    n = L**4
    r = _direction(seed, t)
    a = phi @ r
    site = torch.arange(n, device="cuda")
    grid = site.view(L, L, L, L)
    words = _philox(site, t, 4, seed)
    xs, ys = [], []
    for mu in range(4):
        q = (a * a.roll(-1, 3 - mu)).reshape(-1)
        bond = (q > 0) & (words[mu].double() < (1.0 - torch.exp(-4.0 * kappa * q)) * 2.0**32)
        xs.append(site[bond])
        ys.append(grid.roll(-1, 3 - mu).reshape(-1)[bond])
    x, y = torch.cat(xs), torch.cat(ys)
    lab = site.clone()
    while True:  # hang the larger root under the smaller, then point all at their roots
        u, v = lab[x], lab[y]
        hi, lo = torch.maximum(u, v), torch.minimum(u, v)
        if bool((hi == lo).all()):
            break
        lab.scatter_reduce_(0, hi, lo, "amin")
        while True:
            nxt = lab[lab]
            if bool((nxt == lab).all()):
                break
            lab = nxt
    flip = (_philox(lab, t, 6, seed)[0] >> 31).view(L, L, L, L).double()
    return phi - (2.0 * a * flip)[..., None] * r


def exact(case, seed):
    if case["kind"] != "phi4":
        return None
    phi = _phi4_field(case["L"], seed)
    E, M = [], []
    for t in range(case["updates"]):
        phi = _phi4_update(phi, case["kappa"], seed, t)
        E.append(sum((phi * phi.roll(-1, d)).sum() for d in range(4)))
        M.append(phi.reshape(-1, 4).sum(0))
    return {"field": phi, "E": torch.stack(E), "M": torch.stack(M)}
