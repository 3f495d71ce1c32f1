// Special functions of the synthetic solve's face flux on 2D and 3D meshes, by table
// and short polynomial: on GB300 every FP64 instruction of a warp holds its sub-partition's
// FP64 pipe for 64 cycles, and the library's erf, exp and log spend 45, 17 and
// 25 of them.
//  * exp_tab, log_tab: Tang's table-driven method (P. T. P. Tang, ACM TOMS 15
//    (1989) 144 and 16 (1990) 378): exp(y) = 2^(k/64) exp(r) with |r| <= ln 2/128,
//    log(2^e m) = e ln 2 + log(1/c_j) + log1p(m c_j - 1) with |m c_j - 1| < 2^-8;
//    tables as pairs of doubles.  11 and 14 operations.  Arguments outside the
//    normal range go to the library's functions.
//  * mills: h(t) = (1/2) erfc(t/sqrt 2) exp(t^2/2) for 0 <= t <= 10 as its Taylor
//    series of degree 6 about the nearest multiple of 1/64; h satisfies
//    h' = t h - 1/sqrt(2 pi), so (n+1) c_{n+1} = t c_n + c_{n-1}.
// Errors in units in the last place, bound (largest seen over every table interval, by
// tests/test_gpu_special.py): exp 0.85 (0.80); log 0.55 plus 2^-58, absolute near log x = 0, where the
// table value cancels e ln 2 (0.50); h 4 (3.2; half of 1 - erf loses the tail's relative accuracy
// altogether); T^0.81 for 0.05 <= T <= 20 5 (3.5).  Outside their ranges exp and log
// are the library's, and h keeps its value at 10.
#pragma once
#include "gsis_device.cuh"

namespace gsis {

struct Pair { double hi, lo; };
struct LogEntry { double c, hi, lo; };

// 2^(j/64)
__device__ const Pair g_exp_tab[64] = {
    {0x1.0000000000000p+0, 0x0.0p+0}, {0x1.02c9a3e778061p+0, -0x1.19083535b085dp-56},
    {0x1.059b0d3158574p+0, 0x1.d73e2a475b465p-55}, {0x1.0874518759bc8p+0, 0x1.186be4bb284ffp-57},
    {0x1.0b5586cf9890fp+0, 0x1.8a62e4adc610bp-54}, {0x1.0e3ec32d3d1a2p+0, 0x1.03a1727c57b53p-59},
    {0x1.11301d0125b51p+0, -0x1.6c51039449b3ap-54}, {0x1.1429aaea92de0p+0, -0x1.32fbf9af1369ep-54},
    {0x1.172b83c7d517bp+0, -0x1.19041b9d78a76p-55}, {0x1.1a35beb6fcb75p+0, 0x1.e5b4c7b4968e4p-55},
    {0x1.1d4873168b9aap+0, 0x1.e016e00a2643cp-54}, {0x1.2063b88628cd6p+0, 0x1.dc775814a8495p-55},
    {0x1.2387a6e756238p+0, 0x1.9b07eb6c70573p-54}, {0x1.26b4565e27cddp+0, 0x1.2bd339940e9d9p-55},
    {0x1.29e9df51fdee1p+0, 0x1.612e8afad1255p-55}, {0x1.2d285a6e4030bp+0, 0x1.0024754db41d5p-54},
    {0x1.306fe0a31b715p+0, 0x1.6f46ad23182e4p-55}, {0x1.33c08b26416ffp+0, 0x1.32721843659a6p-54},
    {0x1.371a7373aa9cbp+0, -0x1.63aeabf42eae2p-54}, {0x1.3a7db34e59ff7p+0, -0x1.5e436d661f5e3p-56},
    {0x1.3dea64c123422p+0, 0x1.ada0911f09ebcp-55}, {0x1.4160a21f72e2ap+0, -0x1.ef3691c309278p-58},
    {0x1.44e086061892dp+0, 0x1.89b7a04ef80d0p-59}, {0x1.486a2b5c13cd0p+0, 0x1.3c1a3b69062f0p-56},
    {0x1.4bfdad5362a27p+0, 0x1.d4397afec42e2p-56}, {0x1.4f9b2769d2ca7p+0, -0x1.4b309d25957e3p-54},
    {0x1.5342b569d4f82p+0, -0x1.07abe1db13cadp-55}, {0x1.56f4736b527dap+0, 0x1.9bb2c011d93adp-54},
    {0x1.5ab07dd485429p+0, 0x1.6324c054647adp-54}, {0x1.5e76f15ad2148p+0, 0x1.ba6f93080e65ep-54},
    {0x1.6247eb03a5585p+0, -0x1.383c17e40b497p-54}, {0x1.6623882552225p+0, -0x1.bb60987591c34p-54},
    {0x1.6a09e667f3bcdp+0, -0x1.bdd3413b26456p-54}, {0x1.6dfb23c651a2fp+0, -0x1.bbe3a683c88abp-57},
    {0x1.71f75e8ec5f74p+0, -0x1.16e4786887a99p-55}, {0x1.75feb564267c9p+0, -0x1.0245957316dd3p-54},
    {0x1.7a11473eb0187p+0, -0x1.41577ee04992fp-55}, {0x1.7e2f336cf4e62p+0, 0x1.05d02ba15797ep-56},
    {0x1.82589994cce13p+0, -0x1.d4c1dd41532d8p-54}, {0x1.868d99b4492edp+0, -0x1.fc6f89bd4f6bap-54},
    {0x1.8ace5422aa0dbp+0, 0x1.6e9f156864b27p-54}, {0x1.8f1ae99157736p+0, 0x1.5cc13a2e3976cp-55},
    {0x1.93737b0cdc5e5p+0, -0x1.75fc781b57ebcp-57}, {0x1.97d829fde4e50p+0, -0x1.d185b7c1b85d1p-54},
    {0x1.9c49182a3f090p+0, 0x1.c7c46b071f2bep-56}, {0x1.a0c667b5de565p+0, -0x1.359495d1cd533p-54},
    {0x1.a5503b23e255dp+0, -0x1.d2f6edb8d41e1p-54}, {0x1.a9e6b5579fdbfp+0, 0x1.0fac90ef7fd31p-54},
    {0x1.ae89f995ad3adp+0, 0x1.7a1cd345dcc81p-54}, {0x1.b33a2b84f15fbp+0, -0x1.2805e3084d708p-57},
    {0x1.b7f76f2fb5e47p+0, -0x1.5584f7e54ac3bp-56}, {0x1.bcc1e904bc1d2p+0, 0x1.23dd07a2d9e84p-55},
    {0x1.c199bdd85529cp+0, 0x1.11065895048ddp-55}, {0x1.c67f12e57d14bp+0, 0x1.2884dff483cadp-54},
    {0x1.cb720dcef9069p+0, 0x1.503cbd1e949dbp-56}, {0x1.d072d4a07897cp+0, -0x1.cbc3743797a9cp-54},
    {0x1.d5818dcfba487p+0, 0x1.2ed02d75b3707p-55}, {0x1.da9e603db3285p+0, 0x1.c2300696db532p-54},
    {0x1.dfc97337b9b5fp+0, -0x1.1a5cd4f184b5cp-54}, {0x1.e502ee78b3ff6p+0, 0x1.39e8980a9cc8fp-55},
    {0x1.ea4afa2a490dap+0, -0x1.e9c23179c2893p-54}, {0x1.efa1bee615a27p+0, 0x1.dc7f486a4b6b0p-54},
    {0x1.f50765b6e4540p+0, 0x1.9d3e12dd8a18bp-54}, {0x1.fa7c1819e90d8p+0, 0x1.74853f3a5931ep-55},};

// c_j (24 bits) near 1/m for the j-th of 128 intervals of m in [1, 2), and -log(c_j)
__device__ const LogEntry g_log_tab[128] = {
    {0x1.fe01fe0000000p-1, 0x1.ff00ac2b10bc0p-9, 0x1.6821ad5a97dfep-63},
    {0x1.fa11ca0000000p-1, 0x1.7dc49e7810addp-7, 0x1.8494a240c11b8p-61},
    {0x1.f6310a0000000p-1, 0x1.3cea5df46a5c8p-6, -0x1.765a22a70ef09p-61},
    {0x1.f25f640000000p-1, 0x1.b9fc0afaf91a1p-6, 0x1.ea334206f1a7fp-65},
    {0x1.ee9c800000000p-1, 0x1.1b0d90923d990p-5, -0x1.e9ae9df101997p-60},
    {0x1.eae8080000000p-1, 0x1.58a5b57c8e4dcp-5, 0x1.c6a8e74f1fcffp-61},
    {0x1.e741aa0000000p-1, 0x1.95c836cc8e3f4p-5, 0x1.e683b0fa78541p-61},
    {0x1.e3a9180000000p-1, 0x1.d276b22db0b5dp-5, -0x1.7870f0ef4ab4bp-59},
    {0x1.e01e020000000p-1, 0x1.075982498e472p-4, -0x1.fb25acff68f9dp-59},
    {0x1.dca01e0000000p-1, 0x1.253f6120a1419p-4, -0x1.8a1259e302f7ap-58},
    {0x1.d92f220000000p-1, 0x1.42edcd9a646f2p-4, -0x1.5f1582feaf49bp-58},
    {0x1.d5cac80000000p-1, 0x1.60658ad3750c4p-4, -0x1.188458ebcc614p-58},
    {0x1.d272ca0000000p-1, 0x1.7da76907b12cfp-4, -0x1.73b7eff915a12p-60},
    {0x1.cf26e60000000p-1, 0x1.9ab42252033afp-4, -0x1.c99e337dce8bep-63},
    {0x1.cbe6da0000000p-1, 0x1.b78c7d2b0edb1p-4, -0x1.fcf0f47751aabp-58},
    {0x1.c8b2660000000p-1, 0x1.d4313a96cb361p-4, 0x1.4b0dd7773d0fep-58},
    {0x1.c5894e0000000p-1, 0x1.f0a30391162cap-4, -0x1.80d0c48b83f68p-62},
    {0x1.c26b540000000p-1, 0x1.06714f3ca5972p-3, -0x1.4e7379db88c08p-59},
    {0x1.bf583e0000000p-1, 0x1.14785c6e742bep-3, -0x1.4477d42daf5b9p-57},
    {0x1.bc4fd60000000p-1, 0x1.2266f328a5acep-3, 0x1.e47c0717be8bbp-61},
    {0x1.b951e20000000p-1, 0x1.303d74c647fddp-3, 0x1.6b5199274c898p-57},
    {0x1.b65e2e0000000p-1, 0x1.3dfc2c26cc62bp-3, -0x1.93a8d9e3256b5p-62},
    {0x1.b374840000000p-1, 0x1.4ba37269a55f0p-3, -0x1.f367d96839876p-57},
    {0x1.b094b40000000p-1, 0x1.5933896982097p-3, 0x1.7116d231c3f5dp-57},
    {0x1.adbe880000000p-1, 0x1.66acd4072ad51p-3, -0x1.d201c9c47fc0fp-59},
    {0x1.aaf1d20000000p-1, 0x1.740f93fc037bap-3, 0x1.dfce1e9130fd3p-57},
    {0x1.a82e660000000p-1, 0x1.815c059c357ffp-3, -0x1.89e4bbf1dee80p-58},
    {0x1.a574100000000p-1, 0x1.8e92902886d46p-3, -0x1.169d814e56763p-57},
    {0x1.a2c2a80000000p-1, 0x1.9bb36547dfb89p-3, -0x1.8a1c998d17394p-61},
    {0x1.a01a020000000p-1, 0x1.a8becdf082f1cp-3, 0x1.493c82b98db76p-58},
    {0x1.9d79f20000000p-1, 0x1.b5b51740fb5abp-3, 0x1.f327f7825570fp-57},
    {0x1.9ae24e0000000p-1, 0x1.c2968890c18cbp-3, -0x1.6f6c364d84555p-64},
    {0x1.9852f00000000p-1, 0x1.cf6359209c5eep-3, 0x1.639a216c061e3p-57},
    {0x1.95cbb00000000p-1, 0x1.dc1bcdcabec8bp-3, 0x1.c34c632d8b75fp-57},
    {0x1.934c680000000p-1, 0x1.e8c0250aa5a60p-3, -0x1.2e03a39ca7345p-59},
    {0x1.90d4f20000000p-1, 0x1.f550a0ecb7b4bp-3, -0x1.5057e10ede540p-64},
    {0x1.8e65280000000p-1, 0x1.00e6c38ad501ep-2, 0x1.88d52b24cad58p-58},
    {0x1.8bfce80000000p-1, 0x1.071b860cd590dp-2, 0x1.f1707f98133d5p-58},
    {0x1.899c100000000p-1, 0x1.0d46b3d9ab750p-2, 0x1.a1f63b293b43ap-56},
    {0x1.87427c0000000p-1, 0x1.13686fa13a8b1p-2, -0x1.0a675a9140c2cp-58},
    {0x1.84f00c0000000p-1, 0x1.1980d34542370p-2, -0x1.10c2e4dad040fp-56},
    {0x1.82a4a00000000p-1, 0x1.1f8ffa248a2f3p-2, -0x1.49fdf99b6f5b1p-56},
    {0x1.8060180000000p-1, 0x1.2596011df763ap-2, -0x1.deed8ae041291p-59},
    {0x1.7e22560000000p-1, 0x1.2b93013789d31p-2, -0x1.64eb73873ef99p-56},
    {0x1.7beb3a0000000p-1, 0x1.31871a4144190p-2, -0x1.7135ba3e86ad9p-57},
    {0x1.79baa60000000p-1, 0x1.37726827fd863p-2, -0x1.6c589289f1453p-57},
    {0x1.7790820000000p-1, 0x1.3d54f7e81f71cp-2, -0x1.bea6701908e51p-56},
    {0x1.756cac0000000p-1, 0x1.432ef2f84e814p-2, -0x1.bc98b83e79d6fp-59},
    {0x1.734f0c0000000p-1, 0x1.490068ec009d2p-2, 0x1.c201e6ee8196ap-56},
    {0x1.7137860000000p-1, 0x1.4ec9758200275p-2, -0x1.7450d828f6d1ap-57},
    {0x1.6f26020000000p-1, 0x1.548a2aa6dd268p-2, -0x1.a89d025e1c2ffp-57},
    {0x1.6d1a620000000p-1, 0x1.5a42ac334cfe4p-2, 0x1.b38694373d63fp-57},
    {0x1.6b14900000000p-1, 0x1.5ff308ea793dbp-2, -0x1.7c60de1bc6f0bp-57},
    {0x1.6914740000000p-1, 0x1.659b56383e1f4p-2, 0x1.896c2aad6c368p-56},
    {0x1.6719f40000000p-1, 0x1.6b3bb05b59444p-2, -0x1.e215d15ac1e2bp-58},
    {0x1.6524f80000000p-1, 0x1.70d42f1789238p-2, -0x1.a1663f757c6a9p-56},
    {0x1.63356c0000000p-1, 0x1.7664dfcb9dbd2p-2, 0x1.7695119c1e7e7p-56},
    {0x1.614b360000000p-1, 0x1.7bede21f7afc4p-2, 0x1.8fc38c45e0623p-60},
    {0x1.5f66440000000p-1, 0x1.816f3fb20d49fp-2, 0x1.1b8513aa2074bp-61},
    {0x1.5d867c0000000p-1, 0x1.86e91a5b30ba1p-2, 0x1.27cd8d7a51445p-58},
    {0x1.5babcc0000000p-1, 0x1.8c5b7dad8b48dp-2, 0x1.a2a9646004a3ap-57},
    {0x1.59d6200000000p-1, 0x1.91c67bf45a84dp-2, -0x1.60e0c9ddf57d7p-56},
    {0x1.5805600000000p-1, 0x1.972a345135159p-2, -0x1.da3f62d5f39d1p-56},
    {0x1.56397c0000000p-1, 0x1.9c86af25c0865p-2, -0x1.0f7eece03541cp-56},
    {0x1.54725e0000000p-1, 0x1.a1dc07915b999p-2, -0x1.9f6d76b34af3ep-56},
    {0x1.52aff60000000p-1, 0x1.a72a47a2bd9f0p-2, 0x1.4b1da5133076dp-56},
    {0x1.50f22e0000000p-1, 0x1.ac718c598b0e4p-2, 0x1.0958f5c2d4870p-57},
    {0x1.4f38f60000000p-1, 0x1.b1b1e177dfc5cp-2, 0x1.18f2c80ece010p-61},
    {0x1.4d843c0000000p-1, 0x1.b6eb599bcf35ep-2, -0x1.28dbccd6b94e7p-56},
    {0x1.4bd3ee0000000p-1, 0x1.bc1e083cdad0bp-2, -0x1.51978faf6c115p-56},
    {0x1.4a27fa0000000p-1, 0x1.c14a01ad5f034p-2, 0x1.2bc35ea46185fp-56},
    {0x1.4880520000000p-1, 0x1.c66f4ea3f6ff8p-2, 0x1.afb5c6fc55665p-57},
    {0x1.46dce40000000p-1, 0x1.cb8e04fcd7ad4p-2, 0x1.97bbb35ab30acp-56},
    {0x1.453d9e0000000p-1, 0x1.d0a63b7321e65p-2, -0x1.06198f3eca4dcp-56},
    {0x1.43a2740000000p-1, 0x1.d5b7f6a62c696p-2, 0x1.5c4136354ece4p-57},
    {0x1.420b520000000p-1, 0x1.dac35526c5957p-2, 0x1.5cb9a874cbe06p-56},
    {0x1.40782e0000000p-1, 0x1.dfc856946d5c7p-2, 0x1.098458bb5a8a9p-58},
    {0x1.3ee8f40000000p-1, 0x1.e4c71b0e87705p-2, -0x1.0ac36ddbd7d63p-56},
    {0x1.3d5d9a0000000p-1, 0x1.e9bfa37586206p-2, 0x1.a8eb7125c1e74p-58},
    {0x1.3bd60e0000000p-1, 0x1.eeb20b000ddf8p-2, 0x1.3a6e2ca16857ap-58},
    {0x1.3a52440000000p-1, 0x1.f39e5a4011e60p-2, 0x1.f601bf78a4879p-56},
    {0x1.38d22e0000000p-1, 0x1.f884a0dbe9ecfp-2, 0x1.de0ace16e94b1p-56},
    {0x1.3755be0000000p-1, 0x1.fd64ef2361583p-2, -0x1.14b0eeb21757ep-57},
    {0x1.35dce60000000p-1, 0x1.011fab085ff8ap-1, 0x1.9a0dd407f2889p-57},
    {0x1.34679a0000000p-1, 0x1.0389f052e6342p-1, 0x1.7eeaef519a40ap-55},
    {0x1.32f5ce0000000p-1, 0x1.05f14d38645a4p-1, -0x1.16a8ff1addca1p-56},
    {0x1.3187760000000p-1, 0x1.0855c7c6b4511p-1, -0x1.bf67db4990a34p-55},
    {0x1.301c820000000p-1, 0x1.0ab76d0ee14d7p-1, -0x1.d9d907a58734fp-57},
    {0x1.2eb4ea0000000p-1, 0x1.0d163d019d6b8p-1, 0x1.c28cad150b9e2p-58},
    {0x1.2d50a00000000p-1, 0x1.0f7241e9b497dp-1, 0x1.7a8443bc85c47p-55},
    {0x1.2bef980000000p-1, 0x1.11cb83007cd02p-1, -0x1.79c77227f8815p-55},
    {0x1.2a91ca0000000p-1, 0x1.142200ec43d4dp-1, -0x1.d6c3a65750bddp-56},
    {0x1.2937260000000p-1, 0x1.1675ca44ba60fp-1, -0x1.1699c25fe3736p-56},
    {0x1.27dfa40000000p-1, 0x1.18c6e0335cf09p-1, -0x1.a835da5a8b30fp-55},
    {0x1.268b380000000p-1, 0x1.1b154affda29fp-1, 0x1.a3b852a91d005p-55},
    {0x1.2539d80000000p-1, 0x1.1d610fbe77003p-1, 0x1.0a75635a0eb92p-56},
    {0x1.23eb7a0000000p-1, 0x1.1faa33be70950p-1, -0x1.1b2126109b585p-56},
    {0x1.22a0120000000p-1, 0x1.21f0c0105beecp-1, 0x1.bb5879f93070dp-56},
    {0x1.2157980000000p-1, 0x1.2434b6fc83934p-1, -0x1.cebb8cf0cc266p-57},
    {0x1.2012020000000p-1, 0x1.26761e85430e9p-1, 0x1.e0eb403483a7dp-55},
    {0x1.1ecf440000000p-1, 0x1.28b5007b60783p-1, 0x1.2d09f9a8f3ff8p-55},
    {0x1.1d8f560000000p-1, 0x1.2af15fd0640b0p-1, -0x1.30fe6bef6b99cp-55},
    {0x1.1c52300000000p-1, 0x1.2d2b3fa2edc9ep-1, 0x1.bee9d2f3f8e00p-55},
    {0x1.1b17c60000000p-1, 0x1.2f62aa7b09549p-1, 0x1.a074377b2718cp-55},
    {0x1.19e0120000000p-1, 0x1.3197a0487fe6cp-1, 0x1.8e69111b2baafp-58},
    {0x1.18ab080000000p-1, 0x1.33ca2c0b28995p-1, 0x1.c46ba6cb5b3bbp-55},
    {0x1.1778a20000000p-1, 0x1.35fa4e1336ea2p-1, 0x1.ff7ea0a1864d2p-55},
    {0x1.1648d60000000p-1, 0x1.38280e2b8798bp-1, -0x1.4f1beed5e7a96p-55},
    {0x1.151b9a0000000p-1, 0x1.3a53745debdfap-1, 0x1.98b0892a265e9p-55},
    {0x1.13f0e80000000p-1, 0x1.3c7c81877320fp-1, 0x1.497f4adbefac8p-56},
    {0x1.12c8b80000000p-1, 0x1.3ea33a5eb2f61p-1, -0x1.19321c971164fp-56},
    {0x1.11a3020000000p-1, 0x1.40c7a3ca0dcebp-1, 0x1.5ab914c5ce7a5p-55},
    {0x1.107fbc0000000p-1, 0x1.42e9c6a1f80bfp-1, 0x1.93bee3c19430ep-55},
    {0x1.0f5ee00000000p-1, 0x1.4509a4733bb0cp-1, -0x1.fc0763e9f67d9p-57},
    {0x1.0e40660000000p-1, 0x1.472742b53aab3p-1, 0x1.76f66dd056cf0p-55},
    {0x1.0d24460000000p-1, 0x1.4942a7102fc0dp-1, -0x1.92ced08d28701p-57},
    {0x1.0c0a780000000p-1, 0x1.4b5bd75d6e276p-1, -0x1.1e810cf7f2f01p-61},
    {0x1.0af2f80000000p-1, 0x1.4d72d1fb9fd0bp-1, 0x1.00d4bbd9aac28p-55},
    {0x1.09ddba0000000p-1, 0x1.4f87a4c3026ebp-1, 0x1.cdd5deae6a06dp-57},
    {0x1.08cabc0000000p-1, 0x1.519a4a87a3450p-1, -0x1.a3ce000336d2ep-55},
    {0x1.07b9f20000000p-1, 0x1.53aad18999b82p-1, 0x1.dceeb0dd3db5fp-56},
    {0x1.06ab5a0000000p-1, 0x1.55b934dd40bcep-1, -0x1.9b3435192d0dfp-59},
    {0x1.059eea0000000p-1, 0x1.57c57f416f191p-1, -0x1.dd13a3bc4eee7p-55},
    {0x1.04949c0000000p-1, 0x1.59cfb3dbae887p-1, -0x1.c3ca1e3269b21p-56},
    {0x1.038c6c0000000p-1, 0x1.5bd7d20271c77p-1, 0x1.f8e36398517e8p-55},
    {0x1.0286500000000p-1, 0x1.5ddde50149924p-1, 0x1.d9f46eca133a8p-56},
    {0x1.0182440000000p-1, 0x1.5fe1ec791891ep-1, 0x1.5e7495a8207d9p-55},
    {0x1.0080400000000p-1, 0x1.61e3f01a46467p-1, -0x1.436e4fb134b1cp-56},};

constexpr int MILLS_N = 640;        // t up to 10 in steps of 1/64
struct MillsTab { double c[MILLS_N + 1][8]; };

// Values from the continued fraction 1/(t + 1/(t + 2/(t + ...))) / sqrt(2 pi) at
// t = 10, carried down by the series itself (stable in that direction: an
// error shrinks like exp((t^2 - 100)/2)).
constexpr MillsTab make_mills() {
    MillsTab T{};
    const double k0 = 0.39894228040143267794;   // 1/sqrt(2 pi)
    double f = 0.0;
    for (int n = 120; n >= 1; --n) f = n / (10.0 + f);
    double h = k0 / (10.0 + f);
    for (int i = MILLS_N; i >= 0; --i) {
        const double t = i / 64.0;
        double c[16] = {};
        c[0] = h;
        c[1] = t * c[0] - k0;
        for (int n = 1; n < 15; ++n) c[n + 1] = (t * c[n] + c[n - 1]) / (n + 1);
        for (int n = 0; n < 7; ++n) T.c[i][n] = c[n];
        double v = c[15];
        for (int n = 14; n >= 0; --n) v = v * (-1.0 / 64.0) + c[n];
        h = v;
    }
    return T;
}
__device__ const MillsTab g_mills = make_mills();

// exp(y)
__device__ __forceinline__ double exp_tab(double y) {
    if (((unsigned)__double2hiint(y) & 0x7fffffffu) >= 0x4085e000u) return exp(y);   // |y| >= 700, inf, nan
    const double magic = 6755399441055744.0;   // 1.5 2^52: the sum's low word is the rounded integer
    const double z = fma(y, 0x1.71547652b82fep+6, magic), kd = z - magic;
    const int k = __double2loint(z);
    const double r = fma(kd, -0x1.a39ef35793c76p-39, fma(kd, -0x1.62e42feep-7, y));
    double p = fma(r, 1.0 / 120.0, 1.0 / 24.0);
    p = fma(r, p, 1.0 / 6.0);
    p = fma(r, p, 0.5);
    p = fma(r * r, p, r);
    const Pair t = g_exp_tab[k & 63];
    const double v = t.hi + fma(t.hi, p, t.lo);
    return __hiloint2double(__double2hiint(v) + (k >> 6) * (1 << 20), __double2loint(v));
}

// log(x); near x = 1 the error is absolute (2^-58), not relative: enough for x^omega
__device__ __forceinline__ double log_tab(double x) {
    const unsigned hi = (unsigned)__double2hiint(x);
    if (hi - 0x00100000u >= 0x7fe00000u) return log(x);   // not a positive normal number
    const int e = (int)(hi >> 20) - 1023;
    const LogEntry t = g_log_tab[(hi >> 13) & 127];
    const double m = __hiloint2double((int)((hi & 0xfffffu) | 0x3ff00000u), __double2loint(x));
    const double r = fma(m, t.c, -1.0), ed = (double)e;
    double p = fma(r, -1.0 / 6.0, 0.2);
    p = fma(r, p, -0.25);
    p = fma(r, p, 1.0 / 3.0);
    p = fma(r, p, -0.5);
    const double q = fma(r * r, p, r);
    const double h = fma(ed, 0x1.62e42feep-1, t.hi);             // its rounding error comes back through lo
    const double lo = fma(ed, 0x1.a39ef35793c76p-33, t.lo) + (t.hi - fma(-ed, 0x1.62e42feep-1, h));
    return h + (q + lo);
}

// h(t) for t >= 0 (constant above t = 10, where exp(-t^2/2) < 2e-22)
__device__ __forceinline__ double mills(double t) {
    const double magic = 6755399441055744.0;
    if (__double_as_longlong(t) > 0x4024000000000000LL) t = 10.0;   // (t >= 0: ordered like its bits)
    const double z = fma(t, 64.0, magic), d = fma(z - magic, -1.0 / 64.0, t);
    const double2* c = reinterpret_cast<const double2*>(g_mills.c[__double2loint(z)]);
    const double2 a = __ldg(c), b = __ldg(c + 1), e = __ldg(c + 2);
    const double f = __ldg(reinterpret_cast<const double*>(c + 3));
    double p = fma(d, f, e.y);
    p = fma(d, p, e.x);
    p = fma(d, p, b.y);
    p = fma(d, p, b.x);
    p = fma(d, p, a.y);
    return fma(d, p, a.x);
}

}  // namespace gsis
