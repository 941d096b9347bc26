// FP64 exponential of a non-positive argument for the kernels that evaluate one Gaussian per
// basis function and Euler-Maruyama step.  FP64 instructions issue at 1/64 of the FP32 rate on
// this part, so the FP64 instruction count is the cost: table-driven reduction (P. T. P. Tang,
// ACM TOMS 15, 1989) with 256 entries keeps the polynomial at degree 4.
#pragma once

namespace pdd {

static constexpr int kExpTab = 256;

// 2^(j/256) correctly rounded, and what the rounding left, relative to it
static __device__ const double2 kExp2Tab[kExpTab] = {
    {0x1.0000000000000p+0, 0x0.0p+0}, {0x1.00b1afa5abcbfp+0, -0x1.4e82fc61851acp-55},
    {0x1.0163da9fb3335p+0, 0x1.b3b4f1a88bf6ep-54}, {0x1.02168143b0281p+0, -0x1.2985dd8521d32p-55},
    {0x1.02c9a3e778061p+0, -0x1.160139cd8dc5dp-56}, {0x1.037d42e11bbccp+0, 0x1.51e617061bfbdp-57},
    {0x1.04315e86e7f85p+0, -0x1.05e7a108766d1p-54}, {0x1.04e5f72f654b1p+0, 0x1.45fad437fa426p-55},
    {0x1.059b0d3158574p+0, 0x1.cd2523567f613p-55}, {0x1.0650a0e3c1f89p+0, -0x1.54529642b232fp-54},
    {0x1.0706b29ddf6dep+0, -0x1.bce8023f98efap-55}, {0x1.07bd42b72a836p+0, 0x1.293708ef5c32ep-55},
    {0x1.0874518759bc8p+0, 0x1.0f74e61e6c861p-57}, {0x1.092bdf66607e0p+0, -0x1.5b9280905b2a4p-54},
    {0x1.09e3ecac6f383p+0, 0x1.0a3e45b33d399p-54}, {0x1.0a9c79b1f3919p+0, 0x1.4f31f32c4b7e7p-55},
    {0x1.0b5586cf9890fp+0, 0x1.79aa65d837b6dp-54}, {0x1.0c0f145e46c85p+0, 0x1.407fb30d06420p-54},
    {0x1.0cc922b7247f7p+0, 0x1.eb51a92fdeffcp-55}, {0x1.0d83b23395decp+0, -0x1.a5d04b3b9911bp-54},
    {0x1.0e3ec32d3d1a2p+0, 0x1.ebe3d702f9cd1p-60}, {0x1.0efa55fdfa9c5p+0, -0x1.37a01f0739546p-54},
    {0x1.0fb66affed31bp+0, -0x1.a033489906e0bp-57}, {0x1.1073028d7233ep+0, 0x1.b8268b04ef0a5p-55},
    {0x1.11301d0125b51p+0, -0x1.556522a2fbd0ep-54}, {0x1.11edbab5e2ab6p+0, -0x1.ac46e44a2ebccp-54},
    {0x1.12abdc06c31ccp+0, -0x1.080ef8c4eea55p-58}, {0x1.136a814f204abp+0, -0x1.5704e90c9f860p-57},
    {0x1.1429aaea92de0p+0, -0x1.1c923b9d5f416p-54}, {0x1.14e95934f312ep+0, -0x1.97cea57e46280p-55},
    {0x1.15a98c8a58e51p+0, 0x1.0d3e3e95c55afp-55}, {0x1.166a45471c3c2p+0, 0x1.6f01429e2b9d2p-58},
    {0x1.172b83c7d517bp+0, -0x1.01b15eaa59348p-55}, {0x1.17ed48695bbc0p+0, 0x1.e653b2459034bp-57},
    {0x1.18af9388c8deap+0, -0x1.f1ff055de323dp-55}, {0x1.1972658375d2fp+0, 0x1.2cc7ea345b7dcp-54},
    {0x1.1a35beb6fcb75p+0, 0x1.b898c3f1353bfp-55}, {0x1.1af99f8138a1cp+0, 0x1.57bfb2876ea9ep-54},
    {0x1.1bbe084045cd4p+0, -0x1.6d99c7611eb26p-54}, {0x1.1c82f95281c6bp+0, 0x1.cdc1873af2155p-55},
    {0x1.1d4873168b9aap+0, 0x1.aecf73e3a2f60p-54}, {0x1.1e0e75eb44027p+0, -0x1.493684653a131p-54},
    {0x1.1ed5022fcd91dp+0, -0x1.fe782cb86389dp-55}, {0x1.1f9c18438ce4dp+0, -0x1.8e2899077520ap-54},
    {0x1.2063b88628cd6p+0, 0x1.a6f4144a6c38dp-55}, {0x1.212be3578a819p+0, 0x1.120fcd4f59273p-54},
    {0x1.21f49917ddc96p+0, 0x1.07a05b0e4047dp-55}, {0x1.22bdda27912d1p+0, 0x1.9b788c188c9b8p-55},
    {0x1.2387a6e756238p+0, 0x1.68efde3a8a894p-54}, {0x1.2451ffb82140ap+0, 0x1.77afbca90ef84p-55},
    {0x1.251ce4fb2a63fp+0, 0x1.75e18f274487dp-55}, {0x1.25e85711ece75p+0, 0x1.1512f082876eep-54},
    {0x1.26b4565e27cddp+0, 0x1.0472b981fe7f2p-55}, {0x1.2780e341ddf29p+0, 0x1.a02f0c7d75ec6p-54},
    {0x1.284dfe1f56381p+0, -0x1.6b87b3f71085ep-54}, {0x1.291ba7591bb70p+0, -0x1.03297e78260bfp-55},
    {0x1.29e9df51fdee1p+0, 0x1.2f7e16d09ab31p-55}, {0x1.2ab8a66d10f13p+0, -0x1.5b77e5ccd9fbfp-54},
    {0x1.2b87fd0dad990p+0, -0x1.d219b1a6fbffap-60}, {0x1.2c57e39771b2fp+0, -0x1.1e75c40b4251ep-54},
    {0x1.2d285a6e4030bp+0, 0x1.b3782720c0ab4p-55}, {0x1.2df961f641589p+0, 0x1.8a911f1f7785ap-54},
    {0x1.2ecafa93e2f56p+0, 0x1.e149289cecb8fp-57}, {0x1.2f9d24abd886bp+0, -0x1.1e7c998db7dbbp-57},
    {0x1.306fe0a31b715p+0, 0x1.34d754db0abb6p-55}, {0x1.31432edeeb2fdp+0, 0x1.5425c11faadf4p-55},
    {0x1.32170fc4cd831p+0, 0x1.64201e2ac744cp-55}, {0x1.32eb83ba8ea32p+0, -0x1.79517a03e2847p-54},
    {0x1.33c08b26416ffp+0, 0x1.fdd395dd3f84ap-55}, {0x1.3496266e3fa2dp+0, -0x1.00e2a46da4beep-55},
    {0x1.356c55f929ff1p+0, -0x1.6a3803b8e5b04p-55}, {0x1.36431a2de883bp+0, -0x1.7430803972b34p-55},
    {0x1.371a7373aa9cbp+0, -0x1.24aedcc4b5068p-54}, {0x1.37f26231e754ap+0, -0x1.54de30ae02d94p-54},
    {0x1.38cae6d05d866p+0, -0x1.907f81b512d8ep-54}, {0x1.39a401b7140efp+0, -0x1.4f2487e1c03ecp-54},
    {0x1.3a7db34e59ff7p+0, -0x1.1d1e83e9436d2p-56}, {0x1.3b57fbfec6cf4p+0, 0x1.14a5432fcb2f4p-54},
    {0x1.3c32dc313a8e5p+0, -0x1.91919b3ce1b15p-54}, {0x1.3d0e544ede173p+0, 0x1.9c3bba5562a2fp-56},
    {0x1.3dea64c123422p+0, 0x1.59f48a72a4c6dp-55}, {0x1.3ec70df1c5175p+0, -0x1.5a71612e21658p-55},
    {0x1.3fa4504ac801cp+0, -0x1.312607a28698ap-54}, {0x1.40822c367a024p+0, 0x1.6421f6f1d24d6p-55},
    {0x1.4160a21f72e2ap+0, -0x1.8a78f4817895bp-58}, {0x1.423fb2709468ap+0, -0x1.348a6815fce65p-54},
    {0x1.431f5d950a897p+0, -0x1.c2c9b67499a1bp-56}, {0x1.43ffa3f84b9d4p+0, 0x1.35c43984d9871p-55},
    {0x1.44e086061892dp+0, 0x1.363ed60c2ac11p-59}, {0x1.45c2042a7d232p+0, -0x1.32afc8d9473a0p-57},
    {0x1.46a41ed1d0057p+0, 0x1.666093b0664efp-54}, {0x1.4786d668b3237p+0, -0x1.5fc5e44de020ep-54},
    {0x1.486a2b5c13cd0p+0, 0x1.ecce1daa10379p-57}, {0x1.494e1e192aed2p+0, -0x1.ea0148327c42fp-56},
    {0x1.4a32af0d7d3dep+0, 0x1.3ff8e3f0f1230p-54}, {0x1.4b17dea6db7d7p+0, -0x1.a843ad1a88022p-56},
    {0x1.4bfdad5362a27p+0, 0x1.690cebb7aafb0p-56}, {0x1.4ce41b817c114p+0, 0x1.92ca3bf144e63p-55},
    {0x1.4dcb299fddd0dp+0, 0x1.31dbdeb54e077p-54}, {0x1.4eb2d81d8abffp+0, -0x1.02c99b04aa8b0p-54},
    {0x1.4f9b2769d2ca7p+0, -0x1.f94340071a38ep-55}, {0x1.508417f4531eep+0, 0x1.3e34f67e67118p-56},
    {0x1.516daa2cf6642p+0, -0x1.7deccdc93a349p-55}, {0x1.5257de83f4eefp+0, -0x1.5a3b1197ba0f0p-56},
    {0x1.5342b569d4f82p+0, -0x1.8dec6bd0f385fp-56}, {0x1.542e2f4f6ad27p+0, 0x1.1bd2888075068p-55},
    {0x1.551a4ca5d920fp+0, -0x1.61246ec7b5cf6p-55}, {0x1.56070dde910d2p+0, -0x1.96be8ae89ef8fp-55},
    {0x1.56f4736b527dap+0, 0x1.3350518fdd78ep-54}, {0x1.57e27dbe2c4cfp+0, -0x1.8e6ac90348602p-55},
    {0x1.58d12d497c7fdp+0, 0x1.b98b72f8a9b05p-56}, {0x1.59c0827ff07ccp+0, -0x1.1af7f1365c3acp-54},
    {0x1.5ab07dd485429p+0, 0x1.063e1e21c5409p-54}, {0x1.5ba11fba87a03p+0, -0x1.43a3540d1898ap-54},
    {0x1.5c9268a5946b7p+0, 0x1.4c7855019c6eap-60}, {0x1.5d84590998b93p+0, -0x1.51f58ddaa8090p-54},
    {0x1.5e76f15ad2148p+0, 0x1.432e62b64c035p-54}, {0x1.5f6a320dceb71p+0, -0x1.2e1648e50a17cp-55},
    {0x1.605e1b976dc09p+0, -0x1.ce44a6199769fp-55}, {0x1.6152ae6cdf6f4p+0, 0x1.5f30eda98a575p-54},
    {0x1.6247eb03a5585p+0, -0x1.c33c53bef4da8p-55}, {0x1.633dd1d1929fdp+0, 0x1.17ecda8a72159p-54},
    {0x1.6434634ccc320p+0, -0x1.45378892be9aep-55}, {0x1.652b9febc8fb7p+0, -0x1.345f3cee1ae6ep-54},
    {0x1.6623882552225p+0, -0x1.3cedd78565858p-54}, {0x1.671c1c70833f6p+0, -0x1.5c33fdf910406p-55},
    {0x1.68155d44ca973p+0, 0x1.710aa807e1964p-58}, {0x1.690f4b19e9538p+0, 0x1.1079ab5789604p-55},
    {0x1.6a09e667f3bcdp+0, -0x1.3b3efbf5e2228p-54}, {0x1.6b052fa75173ep+0, 0x1.27df161cd7778p-56},
    {0x1.6c012750bdabfp+0, -0x1.a12ad8734b982p-57}, {0x1.6cfdcddd47645p+0, 0x1.3f9924a05b767p-54},
    {0x1.6dfb23c651a2fp+0, -0x1.367efb86da9eep-57}, {0x1.6ef9298593ae5p+0, -0x1.7557939a8b5efp-55},
    {0x1.6ff7df9519484p+0, -0x1.0dc3d54e08851p-55}, {0x1.70f7466f42e87p+0, 0x1.1ed2f56fa9d1ap-58},
    {0x1.71f75e8ec5f74p+0, -0x1.81f647e5a3ecfp-56}, {0x1.72f8286ead08ap+0, -0x1.8e67a9006c909p-55},
    {0x1.73f9a48a58174p+0, -0x1.6ee4ac08b7db0p-55}, {0x1.74fbd35d7cbfdp+0, 0x1.6597566977ac8p-55},
    {0x1.75feb564267c9p+0, -0x1.619321e55e68ap-55}, {0x1.77024b1ab6e09p+0, 0x1.2c0b7028a5c3ap-54},
    {0x1.780694fde5d3fp+0, 0x1.09ccb5e09d4d3p-54}, {0x1.790b938ac1cf6p+0, 0x1.a30faf49cc78cp-55},
    {0x1.7a11473eb0187p+0, -0x1.b32dcb94da51dp-56}, {0x1.7b17b0976cfdbp+0, -0x1.2dad3519d7b5bp-54},
    {0x1.7c1ed0130c132p+0, 0x1.4ecfd5467c06bp-54}, {0x1.7d26a62ff86f0p+0, 0x1.7d51410fd15c2p-55},
    {0x1.7e2f336cf4e62p+0, 0x1.5ebe1abd66c55p-57}, {0x1.7f3878491c491p+0, -0x1.60a3629969871p-56},
    {0x1.80427543e1a12p+0, -0x1.8a1c52fb3cf42p-55}, {0x1.814d2add106d9p+0, 0x1.b18c6e3fdef5dp-55},
    {0x1.82589994cce13p+0, -0x1.369b6f13b3734p-54}, {0x1.8364c1eb941f7p+0, 0x1.0ec1ddcb1390ap-54},
    {0x1.8471a4623c7adp+0, -0x1.05e843a19ff1ep-55}, {0x1.857f4179f5b21p+0, -0x1.22cea4f3afa1ep-58},
    {0x1.868d99b4492edp+0, -0x1.4d450d872576ep-54}, {0x1.879cad931a436p+0, 0x1.c88549b958471p-56},
    {0x1.88ac7d98a6699p+0, 0x1.0ad675b0e8a00p-54}, {0x1.89bd0a478580fp+0, 0x1.31143962f7877p-54},
    {0x1.8ace5422aa0dbp+0, 0x1.db72fc1f0eab4p-55}, {0x1.8be05bad61778p+0, 0x1.3e9e96f112479p-54},
    {0x1.8cf3216b5448cp+0, -0x1.5b6609cc5e7ffp-57}, {0x1.8e06a5e0866d9p+0, -0x1.dac42a4a38df0p-55},
    {0x1.8f1ae99157736p+0, 0x1.bf68359f35f44p-56}, {0x1.902fed0282c8ap+0, 0x1.b99dd98b1ed84p-55},
    {0x1.9145b0b91ffc6p+0, -0x1.3091fa71e3d83p-54}, {0x1.925c353aa2fe2p+0, -0x1.885ad50cbb750p-56},
    {0x1.93737b0cdc5e5p+0, -0x1.da9b88b6c1e29p-58}, {0x1.948b82b5f98e5p+0, -0x1.2d5e85f3e0301p-55},
    {0x1.95a44cbc8520fp+0, -0x1.c23f97c90b959p-57}, {0x1.96bdd9a7670b3p+0, -0x1.1669428996971p-58},
    {0x1.97d829fde4e50p+0, -0x1.2434322f4f9aap-54}, {0x1.98f33e47a22a2p+0, 0x1.1f2b2c1c4c014p-56},
    {0x1.9a0f170ca07bap+0, -0x1.5ca6cd7668e4bp-55}, {0x1.9b2bb4d53fe0dp+0, -0x1.294f304f166b6p-54},
    {0x1.9c49182a3f090p+0, 0x1.1affc2b91ce27p-56}, {0x1.9d674194bb8d5p+0, -0x1.a1e58414c07d3p-55},
    {0x1.9e86319e32323p+0, 0x1.dd235e10a73bbp-57}, {0x1.9fa5e8d07f29ep+0, -0x1.9740b58a20091p-56},
    {0x1.a0c667b5de565p+0, -0x1.7c50422622263p-55}, {0x1.a1e7aed8eb8bbp+0, 0x1.165830a2b96c2p-54},
    {0x1.a309bec4a2d33p+0, 0x1.b1c86e3e231d5p-55}, {0x1.a42c980460ad8p+0, -0x1.03d5cbe27874bp-54},
    {0x1.a5503b23e255dp+0, -0x1.1bbd1d3bcbb15p-54}, {0x1.a674a8af46052p+0, 0x1.986178980fce0p-58},
    {0x1.a799e1330b358p+0, 0x1.0cc319cee31d2p-54}, {0x1.a8bfe53c12e59p+0, -0x1.9472975b1f2a5p-55},
    {0x1.a9e6b5579fdbfp+0, 0x1.469846e735ab3p-55}, {0x1.ab0e521356ebap+0, 0x1.d8157a34b7e7fp-56},
    {0x1.ac36bbfd3f37ap+0, -0x1.2dfcd978e9db4p-55}, {0x1.ad5ff3a3c2774p+0, 0x1.c8a4e231ebb7dp-55},
    {0x1.ae89f995ad3adp+0, 0x1.c1a7792cb3387p-55}, {0x1.afb4ce622f2ffp+0, -0x1.88c8d11a142e5p-55},
    {0x1.b0e07298db666p+0, -0x1.07b8f4ad1d9fap-54}, {0x1.b20ce6c9a8952p+0, 0x1.89c2ea41433c7p-55},
    {0x1.b33a2b84f15fbp+0, -0x1.5c3d956dcaebap-58}, {0x1.b468415b749b1p+0, -0x1.274aedac8ff80p-56},
    {0x1.b59728de5593ap+0, -0x1.0a40e3da6f640p-54}, {0x1.b6c6e29f1c52ap+0, 0x1.5c620ce76df06p-55},
    {0x1.b7f76f2fb5e47p+0, -0x1.8d6f438ad9334p-57}, {0x1.b928cf22749e4p+0, -0x1.fda52e1b51e41p-55},
    {0x1.ba5b030a1064ap+0, -0x1.1eee26b588a35p-54}, {0x1.bb8e0b79a6f1fp+0, -0x1.2141a7b3e2cd8p-60},
    {0x1.bcc1e904bc1d2p+0, 0x1.4ffd70a5fddcdp-56}, {0x1.bdf69c3f3a207p+0, -0x1.02899507554e5p-60},
    {0x1.bf2c25bd71e09p+0, -0x1.1bdfbfa9298acp-54}, {0x1.c06286141b33dp+0, -0x1.0dda2d4c0010cp-55},
    {0x1.c199bdd85529cp+0, 0x1.36eae30af0cb3p-56}, {0x1.c2d1cd9fa652cp+0, -0x1.a007daadf8d68p-55},
    {0x1.c40ab5fffd07ap+0, 0x1.ee3325c9ffd94p-55}, {0x1.c544778fafb22p+0, 0x1.36909391181d3p-55},
    {0x1.c67f12e57d14bp+0, 0x1.4e08fd10959acp-55}, {0x1.c7ba88988c933p+0, -0x1.11cd7dbdf9547p-55},
    {0x1.c8f6d9406e7b5p+0, 0x1.3cdaf384e1a67p-57}, {0x1.ca3405751c4dbp+0, -0x1.ac28b7bef6621p-56},
    {0x1.cb720dcef9069p+0, 0x1.76b2c6c921968p-57}, {0x1.ccb0f2e6d1675p+0, -0x1.030587207b9e1p-56},
    {0x1.cdf0b555dc3fap+0, -0x1.08a1883ccb5d2p-55}, {0x1.cf3155b5bab74p+0, -0x1.cc734592af7fcp-55},
    {0x1.d072d4a07897cp+0, -0x1.fad5d3ffffa6fp-55}, {0x1.d1b532b08c968p+0, 0x1.7752a44f587e8p-55},
    {0x1.d2f87080d89f2p+0, -0x1.00dae3875a949p-54}, {0x1.d43c8eacaa1d6p+0, 0x1.5b66fefeef52ep-55},
    {0x1.d5818dcfba487p+0, 0x1.4a385a63d07a7p-56}, {0x1.d6c76e862e6d3p+0, 0x1.159d9d908a96ep-58},
    {0x1.d80e316c98398p+0, -0x1.2919e2040220fp-55}, {0x1.d955d71ff6075p+0, 0x1.c254d16117a68p-55},
    {0x1.da9e603db3285p+0, 0x1.e5a50d5c192acp-55}, {0x1.dbe7cd63a8315p+0, -0x1.d8c329fbd0e03p-55},
    {0x1.dd321f301b460p+0, 0x1.43a59ac016b4bp-55}, {0x1.de7d5641c0658p+0, -0x1.ea6e6fbd5f2a6p-55},
    {0x1.dfc97337b9b5fp+0, -0x1.2d52107b43e1fp-55}, {0x1.e11676b197d17p+0, -0x1.3e8e3eab2cbb4p-57},
    {0x1.e264614f5a129p+0, -0x1.92ab93b470dc9p-55}, {0x1.e3b333b16ee12p+0, -0x1.b7966cd0d2cd9p-55},
    {0x1.e502ee78b3ff6p+0, 0x1.4b604603a88d3p-56}, {0x1.e653924676d76p+0, -0x1.76caa4c2ff1cfp-56},
    {0x1.e7a51fbc74c83p+0, 0x1.3c5ec519d7271p-55}, {0x1.e8f7977cdb740p+0, -0x1.1d5fc525d9940p-55},
    {0x1.ea4afa2a490dap+0, -0x1.ff7128fd391f0p-55}, {0x1.eb9f4867cca6ep+0, 0x1.55cd8aaea3d21p-55},
    {0x1.ecf482d8e67f1p+0, -0x1.dae98e223747dp-55}, {0x1.ee4aaa2188510p+0, 0x1.269947c2bed4ap-55},
    {0x1.efa1bee615a27p+0, 0x1.ec3bc41aa2008p-55}, {0x1.f0f9c1cb6412ap+0, -0x1.3b6137e9afe9ep-55},
    {0x1.f252b376bba97p+0, 0x1.42b94c3a9eb32p-55}, {0x1.f3ac948dd7274p+0, -0x1.9fa74878ba7c7p-57},
    {0x1.f50765b6e4540p+0, 0x1.a64a931d185eep-55}, {0x1.f6632798844f8p+0, 0x1.01f3a75ee0efep-54},
    {0x1.f7bfdad9cbe14p+0, -0x1.e37bae43be3edp-55}, {0x1.f91d802243c89p+0, -0x1.16a9ce6ed84fap-58},
    {0x1.fa7c1819e90d8p+0, 0x1.7893b4d91cd9dp-56}, {0x1.fbdba3692d514p+0, -0x1.99c7db2effc76p-57},
    {0x1.fd3c22b8f71f1p+0, 0x1.305c14160cc89p-58}, {0x1.fe9d96b2a23d9p+0, 0x1.4b458677f9840p-57},
};

// e^a for a <= 0 (0 below -708), tab = the 256 entries (shared memory).  a = k ln2/256 + r with
// |r| <= h = ln2/512: k ln2_hi is exact (ln2_hi/256 has 34 bits); e^r - 1 = r (1 + r/2 + r^2/6 + r^3/24)
// with the term r^5/120 folded into the odd coefficients (r^5 ~ (20 h^2 r^3 - 5 h^4 r)/16, off by
// h^5/16); the power of two goes into the table entry's exponent field.  10 FP64 instructions;
// within 0.53 ulp (4e6 arguments in [-700, 0] against 80-bit arithmetic).
__device__ __forceinline__ double exp_neg(double a, const double2 *tab) {
    const double magic = 6755399441055744.0;                   // 1.5 2^52: the sum's low word is the integer
    const double t = fma(a, 0x1.71547652b82fep+8, magic);
    const int k = __double2loint(t);
    const double kf = t - magic;
    double r = fma(kf, -0x1.62e42fef80000p-9, a);
    r = fma(kf, -0x1.1cf79abc9e3b4p-44, r);
    const double2 T = tab[k & (kExpTab - 1)];
    const double Ts = __hiloint2double(__double2hiint(T.x) + ((k >> 8) << 20), __double2loint(T.x));
    double p = fma(r, 0x1.5555555555555p-5, 0x1.555557e54fd55p-3);
    p = fma(p, r, 0.5);
    p = fma(p, r, 0x1.fffffffffffb1p-1);
    const double e = fma(Ts, fma(p, r, T.y), Ts);
    // a below -708 (by its high word: more negative is larger as an unsigned integer) gives 0
    return (unsigned)__double2hiint(a) > 0xC0862000u ? 0.0 : e;
}

}  // namespace pdd
