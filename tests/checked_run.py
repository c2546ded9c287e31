"""Runs a few decode steps and single calls with whichever libpced the environment selects
(PCED_LIB=checked: the bounds-checked build) and prints, per case, the device
status word, the chosen tokens and a hash of the final hidden states (of the
outputs, for a call) as one JSON line.  Used by test_gpu_checked.py in a child process."""
import hashlib
import json
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

CASES = [("tiny", {}, 4, {}), ("llama8", {"L": 4}, 2, {}), ("tiny", {}, 3, {"aggregation": 1}),
         ("tiny", {}, 3, {"dynamic_beta": True}), ("llama8", {"L": 2}, 2, {"paged": 64}),
         ("tiny", {"B": 7, "N": 22, "V": 1128}, 2, {}), ("tiny", {"B": 20, "N": 19, "V": 300}, 2, {"aggregation": 1})]
# one layer of attention: (lengths, query heads, kv heads, head dim); the LM head: (rows, d, V)
ATTENTION = [([257, 32, 1], 8, 2, 64), ([5000, 1, 700], 32, 8, 128), ([300] * 70, 28, 4, 128)]
LM_HEAD = [(9, 128, 1000), (161, 128, 1128), (400, 64, 20000)]


def _sha(*tensors):
    import torch
    h = hashlib.sha256()
    for t in tensors:
        h.update(t.cpu().contiguous().view(torch.uint8).numpy().tobytes())
    return h.hexdigest()[:16]


def run_cases():
    import torch
    import paper_2601_08670_gb300 as pced
    import synth
    out = []
    for name, over, steps, kw in CASES:
        kw = dict(kw)
        paged = kw.pop("paged", 0)
        w = synth.get(name, **over)
        t = synth.device_inputs(w, "cuda", paged=paged)
        dm = pced.dims(w.B, w.N, w.L, w.Hq, w.Hkv, w.D, w.V)
        dec = pced.decoder_from_inputs(dm, t, gamma=w.gamma, max_steps=w.steps, bos=w.bos, keep_hidden=True, **kw)
        for _ in range(steps):
            dec.step()
        torch.cuda.synchronize()
        out.append({"case": f"{name}{over}{kw}{'paged' if paged else ''}", "status": dec.status(),
                    "tokens": dec.history[:, :steps].cpu().numpy().tolist(),
                    "hidden": _sha(dec.hidden)})
        del dec, t
        torch.cuda.empty_cache()
    g = torch.Generator(device="cuda").manual_seed(3)

    def normal(*shape):
        return torch.empty(shape, dtype=torch.bfloat16, device="cuda").normal_(generator=g)

    for lens, Hq, Hkv, D in ATTENTION:
        n = torch.tensor(lens, dtype=torch.int32)
        off = torch.cat([torch.zeros(1, dtype=torch.int64), (n.long() * Hkv * D).cumsum(0)])
        ws = pced.workspace(pced.decode_attention_workspace_size(len(lens), Hq, Hkv, D), "cuda")
        o = pced.decode_attention(normal(len(lens), Hq, D), normal(int(off[-1])), normal(int(off[-1])),
                                  off[:-1].cuda(), n.cuda(), n.cuda(), Hkv, sum(lens), ws=ws)
        out.append({"case": f"attention {len(lens)} {Hq}/{Hkv}/{D}", "status": pced.device_status(ws), "tokens": [],
                    "hidden": _sha(o)})
    for S, d, V in LM_HEAD:
        ws = pced.workspace(pced.lm_head_workspace_size(S, V), "cuda")
        lp, lse = pced.lm_head_logprobs(normal(S, d), normal(V, d), ws=ws)
        out.append({"case": f"lm_head {S} {d} {V}", "status": pced.device_status(ws), "tokens": [],
                    "hidden": _sha(lp, lse)})
    return out


if __name__ == "__main__":
    print(json.dumps(run_cases()))
