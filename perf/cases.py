"""The work a program that serves (and once converts) a TransMLA layer has this library do, as measurable cases.

Kinds of passes, each through the public binding with the buffers a server keeps between steps:
  step     one decode step on device buffers: append the new tokens' latents, absorbed split-KV attention, combine
  host     the same step driven from pinned host buffers, results back on the host
  fp8      one decode step over the FP8 latent cache: quantising append, attention, combine
  layer    one decode step of the whole attention layer: query projections (full-rank or low-rank), step, W_O
  prefill  a chunk of q_len prompt positions per sequence in the MHA form over the latent cache
  convert  the conversion of one layer on calibration activations: rotation, balancing, joint PCA, rewrite

Sizes come from the library's configurations (synth.py) and benchmark workloads; cached lengths are uniform in
[len_lo, len_hi] from a seed that belongs to the case.  Values are those of synth.py: activations and cache rows
N(0,1), weights N(0, 1/sqrt(fan_in)), bf16 (fp32 for the conversion).
"""
import dataclasses
import math

import torch

from paper_2502_07864_b200 import binding, synth

MODELS = {'llama2-7b': synth.LLAMA2_7B, 'qwen2.5-72b': synth.QWEN25_72B}
FP8_ROW = synth.FP8_ROW_BYTES
FOLD, ROUNDS = 4, 20            # FreqFold and subspace rounds of the conversion, as in the benchmark's workload


def _case(kind, batch, len_lo, len_hi, model='llama2-7b', q_len=1, q_rank=0, len_seed=4, name=None):
    c = {'kind': kind, 'model': model, 'batch': batch, 'q_len': q_len, 'len_lo': len_lo, 'len_hi': len_hi,
         'len_seed': len_seed, 'q_rank': q_rank}
    return dict(c, name=name) if name else c


def listed():
    return [
        # a single short chat: nothing but latency and launches
        _case('step', 1, 777, 777, name='step_b1_short'),
        # the headline workload: a medium serving batch at 8K context
        _case('step', 16, 8192, 8192, name='step_b16_8k'),
        # a mixed serving batch, short chats beside long documents
        _case('step', 32, 1024, 32768, name='step_b32_ragged'),
        # the largest serving batch of the target range
        _case('step', 128, 8192, 8192, name='step_b128_8k'),
        # a larger model with two new tokens per sequence (multi-token prediction), ragged lengths
        _case('step', 64, 2048, 8192, model='qwen2.5-72b', q_len=2, len_seed=5, name='step_64heads_b64_s2'),
        # the headline workload as an engine on the host sees it: inputs and results in pinned host memory
        _case('host', 16, 8192, 8192, name='host_b16_8k'),
        # the quantised cache, ragged lengths of a serving batch
        _case('fp8', 64, 4001, 8192, name='fp8_b64_ragged'),
        # the whole attention layer, full-rank queries, medium batch
        _case('layer', 16, 8192, 8192, name='layer_b16_8k'),
        # the whole attention layer with compressed queries, larger batch of mixed lengths
        _case('layer', 64, 1024, 8192, q_rank=1536, name='layer_lowrank_b64_ragged'),
        # a chunk of a long prompt over what is already cached
        _case('prefill', 4, 8192, 8192, q_len=512, name='prefill_b4_8k_s512'),
        # prompts of mixed lengths, the last 1900 positions of each
        _case('prefill', 12, 1900, 8192, q_len=1900, name='prefill_b12_ragged_s1900'),
        # offline: one layer of a checkpoint converted on 8192 calibration tokens
        _case('convert', 1, 8192, 8192, name='convert_n8192'),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges; kinds in about the proportion in which they are used."""
    most = max(_cost(c) for c in listed())
    while True:
        kind = rng.choice(['step'] * 5 + ['host'] + ['fp8'] * 2 + ['layer'] * 3 + ['prefill'] * 3 + ['convert'])
        seed = rng.randrange(1 << 20)
        if kind == 'convert':
            n = _log_uniform(rng, 2048, 8192)
            c = _case('convert', 1, n, n, len_seed=seed)
        elif kind == 'prefill':
            q_len = _log_uniform(rng, 64, 4096)
            hi = _log_uniform(rng, max(q_len, 256), 16384)
            c = _case('prefill', _log_uniform(rng, 1, 16), rng.randint(max(q_len, hi // 4), hi), hi, q_len=q_len, len_seed=seed)
        else:
            model = 'qwen2.5-72b' if kind in ('step', 'layer') and rng.random() < 0.3 else 'llama2-7b'
            q_len = rng.choice([1, 2]) if model == 'qwen2.5-72b' else rng.choice([1, 1, 1, 2])
            hi = _log_uniform(rng, 128, 131072)
            lo = hi if rng.random() < 0.25 else rng.randint(max(64, hi // 16), hi)
            q_rank = 1536 if kind == 'layer' and rng.random() < 0.5 else 0
            c = _case(kind, _log_uniform(rng, 1, 128), lo, hi, model=model, q_len=q_len, q_rank=q_rank, len_seed=seed)
            if sum(_lengths(c)) > 128 * 8192:     # the most cached tokens a layer holds here
                continue
        if _cost(c) <= most:
            return c


def _lengths(case):
    return synth.uniform_seqlens(case['batch'], case['len_lo'], case['len_hi'], case['len_seed'])


def _shape(case):
    return dataclasses.replace(MODELS[case['model']], S=case['q_len'])


def _visible(case):
    """(query position, cached token) pairs that attention has to look at, per head."""
    S = case['q_len']
    return sum(S * L - S * (S - 1) // 2 for L in _lengths(case))


def work(case):
    sh, B, S = _shape(case), case['batch'], case['q_len']
    n, tok = B * S, sum(_lengths(case))
    HdR, Hdn, Hdv = sh.H * sh.dR, sh.H * sh.dn, sh.H * sh.dv
    if case['kind'] == 'convert':
        n, g, d, D, r = case['len_lo'], sh.H, sh.dn, sh.D, sh.r
        m, mz = g * FOLD, (2 * g - 1) * d
        flops = 2.0 * n * D * (g * d + mz)                        # key, NoPE-key and value activations
        flops += 2.0 * 2 * n * (d // 2 // FOLD) * m * m           # covariances, real and imaginary parts
        flops += 2.0 * n * mz * mz                                # joint second moment
        flops += 2.0 * ROUNDS * (mz * mz * r + 2 * mz * r * r)    # subspace rounds with their orthonormalisations
        flops += 2.0 * r * mz * D                                 # rewrite
        return {'bytes': 4.0 * (n * D + 2 * g * d * D + mz * r + g * d * D + mz * mz + mz * r + r * D), 'flops': flops}
    if case['kind'] == 'prefill':
        flops = 2.0 * sh.r * (Hdn + Hdv) * tok + 2.0 * (sh.dn + sh.dR + sh.dv) * sh.H * _visible(case)
        return {'bytes': 2.0 * (tok * sh.row + n * (Hdn + HdR + Hdv) + sh.r * (Hdn + Hdv)) + 4.0 * n * sh.H, 'flops': flops}
    row = FP8_ROW if case['kind'] == 'fp8' else 2 * sh.row
    weights = sh.row * sh.D + sh.r * (Hdn + Hdv)
    flops = 2.0 * sh.H * (sh.row + sh.r) * _visible(case) + 2.0 * n * weights
    nbytes = float(tok * row) + 2.0 * (weights + n * sh.D)
    if case['kind'] == 'layer':
        Dq = case['q_rank'] or sh.D
        maps = (Hdn + HdR) * Dq + sh.D * Hdv + (case['q_rank'] * sh.D)
        return {'bytes': nbytes + 2.0 * (maps + n * sh.D), 'flops': flops + 2.0 * n * maps}
    return {'bytes': nbytes + 2.0 * n * (Hdn + HdR + Hdv) + 4.0 * n * sh.H, 'flops': flops}


def _cost(case):
    w = work(case)
    return max(w['bytes'], w['flops'] / 50)


def tolerance(case):
    # About four times what is seen against the same arithmetic in fp64.  bf16 operands, probabilities and results: rel
    # 2.5e-3, max 1.7e-2 for a step, 2.8e-2 for a prefill chunk; the layer adds two linear maps: 3.8e-3, 1.8e-2.  The
    # conversion (fp32), with its sums over tokens and hidden coordinates in another order: rel 4.6e-5, max 1.1e-3,
    # both from the subspace rounds, which amplify roundings.  FP8 codes may fall on the other side of a tie, and an
    # appended row's fp32 scale may differ in its last bits; the other rows of the cache stay as they are.
    return {'convert': {'rel': 2e-4, 'max': 4.5e-3}, 'prefill': {'rel': 1e-2, 'max': 0.11}, 'layer': {'rel': 1.5e-2, 'max': 0.075},
            'fp8': {'rel': 1e-2, 'max': 0.07, 'differ': 2e-3}}.get(case['kind'], {'rel': 1e-2, 'max': 0.07})


# ------------------------------------------------------------------------------------------------ inputs and passes
def prepare(case, seed):
    return {'convert': _prepare_convert, 'prefill': _prepare_prefill}.get(case['kind'], _prepare_decode)(case, seed)


def run(state):
    return state['pass'](state)


def _prepare_decode(case, seed):
    sh, lengths, kind = _shape(case), _lengths(case), case['kind']
    B, S = case['batch'], case['q_len']
    s = synth.make_decode_case(sh, lengths, seed, device='cuda')
    a = synth.make_append_case(sh, [L - S for L in lengths], seed + 1, device='cuda')
    s.update(x=a['x'], w_dkv_kr=a['w_dkv_kr'], positions=a['positions'])
    if kind == 'fp8':
        s['cache'] = synth.make_fp8_cache(sh, s['cache'].shape[0], seed + 2, device='cuda')
        s['scratch'] = torch.empty(B * S * sh.row, dtype=torch.float32, device='cuda')
    s['params'] = binding.make_params(sh, B, s['cache'].shape[0], s['page_table'].shape[1], (sh.dn + sh.dR) ** -0.5)
    s['workspace'], _ = binding.alloc_workspace(s['params'])
    s['status'] = torch.zeros(1, dtype=torch.int32, device='cuda')
    s['out'] = torch.empty(B, S, sh.H, sh.dv, dtype=torch.bfloat16, device='cuda')
    s['lse'] = torch.empty(B, S, sh.H, dtype=torch.float32, device='cuda')
    if kind == 'layer':
        w = synth.make_layer_weights(sh, seed + 3, q_lora_rank=case['q_rank'], device='cuda')
        s['weights'] = dict(w, w_dkv_kr=s['w_dkv_kr'], w_uk=s['w_uk'], w_uv=s['w_uv'])
        nbytes = binding.transmla_layer_scratch_bytes(s['params'], case['q_rank'])
        s['scratch'] = torch.empty(nbytes, dtype=torch.uint8, device='cuda')
        s['y'] = torch.empty(B, S, sh.D, dtype=torch.bfloat16, device='cuda')
    if kind == 'host':
        nbytes = binding.transmla_step_staging_bytes(s['params'])
        s['staging'] = torch.empty(nbytes, dtype=torch.uint8, device='cuda')
        for k in ('x', 'q_nope', 'q_pe', 'page_table', 'seqlens', 'out', 'lse'):
            s[k] = s[k].cpu().pin_memory()
    s['pass'] = {'step': _run_step, 'host': _run_host, 'fp8': _run_fp8, 'layer': _run_layer}[kind]
    return s


def _run_step(s):
    binding.transmla_decode_step(s['params'], s['x'], s['q_nope'], s['q_pe'], s['page_table'], s['seqlens'], s['w_dkv_kr'],
                                 s['w_uk'], s['w_uv'], s['cache'], s['workspace'], s['out'], s['lse'], s['status'])
    return {'out': s['out'], 'lse': s['lse'], 'cache': s['cache'], 'status': s['status']}


def _run_host(s):
    word = binding.transmla_decode_step_host(s['params'], s['x'], s['q_nope'], s['q_pe'], s['page_table'], s['seqlens'],
                                             s['w_dkv_kr'], s['w_uk'], s['w_uv'], s['cache'], s['staging'], s['workspace'],
                                             s['out'], s['lse'])
    return {'out': s['out'], 'lse': s['lse'], 'cache': s['cache'], 'status': word}


def _run_fp8(s):
    binding.transmla_latent_append_fp8(s['params'], s['x'], s['w_dkv_kr'], s['positions'], s['page_table'], s['cache'],
                                       s['scratch'], s['status'])
    binding.transmla_mla_decode_fp8(s['params'], s['q_nope'], s['q_pe'], s['w_uk'], s['cache'], s['page_table'],
                                    s['seqlens'], s['workspace'], s['status'])
    binding.transmla_mla_combine(s['params'], s['workspace'], s['w_uv'], s['out'], s['lse'], s['status'])
    return {'out': s['out'], 'lse': s['lse'], 'cache': s['cache'], 'status': s['status']}


def _run_layer(s):
    binding.transmla_layer_decode_step(s['params'], s['weights'], s['x'], s['page_table'], s['seqlens'], s['cache'],
                                       s['workspace'], s['scratch'], s['y'], s['status'])
    return {'y': s['y'], 'cache': s['cache'], 'status': s['status']}


def _prepare_prefill(case, seed):
    sh, B = _shape(case), case['batch']
    s = synth.make_decode_case(sh, _lengths(case), seed, device='cuda')
    s['params'] = binding.make_params(sh, B, s['cache'].shape[0], s['page_table'].shape[1], (sh.dn + sh.dR) ** -0.5)
    nbytes = binding.transmla_prefill_scratch_bytes(s['params'])
    s['scratch'] = torch.empty(nbytes // 2, dtype=torch.bfloat16, device='cuda')
    s['status'] = torch.zeros(1, dtype=torch.int32, device='cuda')
    s['out'] = torch.empty(B, sh.S, sh.H, sh.dv, dtype=torch.bfloat16, device='cuda')
    s['lse'] = torch.empty(B, sh.S, sh.H, dtype=torch.float32, device='cuda')
    s['pass'] = _run_prefill
    return s


def _run_prefill(s):
    binding.transmla_mla_prefill(s['params'], s['q_nope'], s['q_pe'], s['w_uk'], s['w_uv'], s['cache'], s['page_table'],
                                 s['seqlens'], s['scratch'], s['out'], s['lse'], s['status'])
    return {'out': s['out'], 'lse': s['lse'], 'status': s['status']}


def _prepare_convert(case, seed):
    sh, n = _shape(case), case['len_lo']
    g, d, D, r = sh.H, sh.dn, sh.D, sh.r
    groups, m, mz = d // 2 // FOLD, g * FOLD, (2 * g - 1) * d
    s = synth.make_conversion_case(n, D, g, d, seed, device='cuda')
    f32 = dict(dtype=torch.float32, device='cuda')
    gen = torch.Generator(device='cuda')
    gen.manual_seed(seed + 1)
    s['q0'] = torch.randn(mz, r, generator=gen, device='cuda')
    # Orthogonal rotations, as a program keeps them from the layer's calibration.  The pass searches them again, but
    # eigenvectors are unique only up to their signs: going on with one of two equally valid results would make every
    # later output of the pass depend on a rounding.
    s['kept_u'] = torch.linalg.qr(torch.randn(groups, m, m, generator=gen, device='cuda'))[0].contiguous()
    for name, size in {'k_act': (n, g * d), 'k_nope': (n, (g - 1) * d), 'v_act': (n, g * d), 'cov': (groups, m, m),
                       'vals': (groups, m), 'u': (groups, m, m), 'w_rot': (g * d, D), 'w_dkv': (mz, D), 'norms': (2 * n,),
                       'z': (n, mz), 'c': (mz, mz), 'q': (mz, r), 'new_dkv': (r, D)}.items():
        s[name] = torch.empty(size, **f32)
    s['alpha'] = torch.zeros(1, **f32)
    s['seg'] = torch.empty(binding.transmla_conv_rorope_scratch_bytes(n, g, d, FOLD) // 4, **f32)
    s['ws'] = torch.empty(binding.transmla_conv_subspace_scratch_bytes(mz, r), dtype=torch.uint8, device='cuda')
    s['status'] = torch.zeros(1, dtype=torch.int32, device='cuda')
    s['g'], s['d'], s['pass'] = g, d, _run_convert
    return s


def _run_convert(s):
    x, w_k, w_v, w_rot, g, d = s['x'], s['w_k'], s['w_v'], s['w_rot'], s['g'], s['d']
    binding.transmla_conv_gemm(x, w_k, s['k_act'], tb=True)
    binding.transmla_conv_rorope_covariance(s['k_act'], g, d, FOLD, s['seg'], s['cov'])
    binding.transmla_conv_sym_eig(s['cov'], s['vals'], s['u'], s['status'])
    rebuilt = torch.bmm(s['u'] * s['vals'][:, None, :], s['u'].mT)  # what the eigenvectors stand for, whatever their signs
    binding.transmla_conv_rorope_apply(w_k, s['kept_u'], g, d, FOLD, w_rot)
    binding.transmla_conv_gemm(x, w_rot[d:], s['k_nope'], tb=True)
    binding.transmla_conv_gemm(x, w_v, s['v_act'], tb=True)
    binding.transmla_conv_alpha(s['k_nope'], s['v_act'], s['norms'], s['alpha'])
    binding.transmla_conv_balance_concat(s['k_nope'], s['v_act'], s['alpha'], s['z'])
    binding.transmla_conv_gemm(s['z'], s['z'], s['c'], ta=True)
    s['q'].copy_(s['q0'])
    binding.transmla_conv_top_subspace(s['c'], s['q'], ROUNDS, s['ws'], s['status'])
    torch.div(w_rot[d:], s['alpha'], out=s['w_dkv'][:(g - 1) * d])
    s['w_dkv'][(g - 1) * d:].copy_(w_v)
    binding.transmla_conv_gemm(s['q'], s['w_dkv'], s['new_dkv'], ta=True)
    out = {k: s[k] for k in ('cov', 'vals', 'w_rot', 'alpha', 'c', 'q', 'new_dkv', 'status')}
    return dict(out, rebuilt=rebuilt)
